"""Row offsets of the level kernels on planes of 2^31 nodes and more, from the
kernels' own source built for the host (CPU only): a 2-D field is one plane, and
neither its rows nor those of its stream may wrap."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2503_06322_gb300", "csrc")

PRELUDE = r'''
#include <cstdio>
#include <cstdlib>
#define __host__
#define __device__
'''
MAIN = r'''
int main(int argc, char **argv)
{
    const PlaneRows w = plane_rows(atoi(argv[1]), atoi(argv[2]), atoi(argv[3]));
    printf("%lld %lld %lld %lld\n", w.x[0], w.x[1], w.k[0], w.k[1]);
    return 0;
}
'''


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    grid = open(os.path.join(CSRC, "internal.cuh")).read()
    a, b = grid.index("__host__ __device__ inline int cpos_of"), grid.index("// Explicitly rounded arithmetic")
    t = tmp_path_factory.mktemp("rows_host")
    (t / "p.cpp").write_text(PRELUDE + grid[a:b] + MAIN)
    subprocess.run([cxx, "-O2", "-std=c++17", "-Wall", "-fsanitize=undefined", "-fno-sanitize-recover", "-o", str(t / "p"),
                    str(t / "p.cpp")], check=True)
    return str(t / "p")


@pytest.mark.parametrize("m1,m2", [(5, 9), (46342, 46342), (65537, 65537), (70000, 70000), (2, 1 << 30), (1 << 30, 5)])
def test_row_offsets(exe, m1, m2):
    mc2 = m2 // 2 + 1
    for Ra in sorted({0, (m1 // 2) & ~1, (m1 - 2) & ~1}):
        got = [int(v) for v in subprocess.run([exe, *map(str, (m2, mc2, Ra))], check=True, capture_output=True,
                                              text=True).stdout.split()]
        kept = [Ra // 2, Ra // 2 + 1]           # kept rows before Ra and Ra + 1
        assert got == [Ra * m2, (Ra + 1) * m2, Ra * m2 - kept[0] * mc2, (Ra + 1) * m2 - kept[1] * mc2]
