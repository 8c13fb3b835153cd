"""Planes of any size and shape in the level kernels, from their own source built
for the host (CPU only): a 2-D field is one plane, so neither its rows nor those
of its stream may wrap from 2^31 nodes on, and its tiles have to fit the grid of a
launch however tall it is."""
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
    if (argc == 5) {     // every coarse row and column in exactly one tile, all of them in gridDim.x
        const int mc1 = atoi(argv[1]), mc2 = atoi(argv[2]), LC = atoi(argv[3]), R = tile_rows(LC);
        const long long n = plane_tiles(mc1, mc2, LC);
        long long next = 0;
        for (long long b = 0; b < n; b++) {
            const PlaneTile t = plane_tile((unsigned)b, mc2, LC);
            if (t.j1 >= mc1 || t.j2 >= mc2 || t.j1 % R || t.j2 % LC) return 1;
            if ((long long)(t.j1 / R) * tile_cols(mc2, LC) + t.j2 / LC != next++) return 2;
        }
        return n * R * LC < (long long)mc1 * mc2 || n > 2147483647ll;
    }
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
    src = open(os.path.join(CSRC, "adjoint.cu")).read()
    c = src.index("constexpr int kMpWarps")
    d = src.rindex("template <typename T", c, src.index("__global__ void", c))
    t = tmp_path_factory.mktemp("rows_host")
    (t / "p.cpp").write_text(PRELUDE + grid[a:b] + src[c:d] + MAIN)
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


@pytest.mark.parametrize("mc1,mc2", [(1, 2), (8, 32), (9, 33), (550001, 3), (1 << 29, 2), (3, 1 << 29), (35001, 35001)])
@pytest.mark.parametrize("cols", [32, 8])
def test_tiles(exe, mc1, mc2, cols):
    """550001 coarse rows: a field of 1.1 million rows, past 65535 tiles of eight"""
    assert subprocess.run([exe, str(mc1), str(mc2), str(cols), "tiles"]).returncode == 0
