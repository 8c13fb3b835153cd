"""The decoder's view of a chunk's words (BitQueue of csrc/huffman.cu), built for
the host (CPU only): the right bits from every start, wherever the stream starts
in memory and ends, with no word loaded from outside the stream."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_2503_06322_gb300", "csrc", "huffman.cu")

PRELUDE = r'''
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <vector>
#define __device__
#define __forceinline__ inline
constexpr int kDecThreads = 1024;
static const uint32_t *lo_, *hi_;          // the stream's words
static uint32_t load(const uint32_t *p)
{
    if (p < lo_ || p >= hi_) { printf("a load outside the stream\n"); exit(1); }
    return *p;
}
struct Words8 { uint32_t v[8]; };
static Words8 ldg32(const uint32_t *p) { Words8 r; for (int k = 0; k < 8; k++) r.v[k] = load(p + k); return r; }
static uint32_t ldw(const uint32_t *w, unsigned long long i, unsigned long long n) { return i < n ? load(w + i) : 0u; }
static uint32_t ring_[32 * kDecThreads];
static uint32_t lds32(uint32_t a) { return ring_[a / 4]; }
static void sts32(uint32_t a, uint32_t v) { ring_[a / 4] = v; }
static uint32_t __funnelshift_l(uint32_t lo, uint32_t hi, uint32_t s)
{
    return (uint32_t)((((uint64_t)hi << 32 | lo) << (s & 31)) >> 32);
}
constexpr unsigned kRingWords = 32;
'''
MAIN = r'''
int main()
{
    alignas(32) static uint32_t mem[256];
    for (int i = 0; i < 256; i++) mem[i] = (uint32_t)rand() * 2654435761u + (uint32_t)i;
    for (unsigned at = 32; at < 40; at++)
        for (unsigned n : {1u, 3u, 4u, 5u, 8u, 12u, 13u, 100u}) {
            const uint32_t *w = mem + at;
            lo_ = w; hi_ = w + n;
            auto bit = [&](unsigned long long i) { return i < 32ull * n ? w[i / 32] >> (31 - i % 32) & 1u : 0u; };
            for (unsigned pos = 0; pos < 32 * n; pos += 1 + (pos % 7)) {
                BitQueue q;
                q.ring = 4 * 17;
                uint32_t h, l;
                int nb;
                q.start(w, n, pos, h, l, nb);
                unsigned at0 = q.pos(nb);
                for (unsigned skip = 0; skip < 700; skip += 53) {
                    const uint64_t win = (uint64_t)h << 32 | l;
                    for (int i = 0; i < nb; i++)
                        if ((win >> (63 - i) & 1u) != bit(pos + skip + i)) { printf("wrong bit\n"); return 1; }
                    q.top_up();
                    q.seek(at0 + skip + 53, h, l, nb);
                }
            }
        }
    return 0;
}
'''


def test_decoder_queue(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src = open(SRC).read()
    a, b = src.index("struct BitQueue {"), src.index("// 64 bits of the stream from bit pos")
    (tmp_path / "q.cpp").write_text(PRELUDE + src[a:b] + MAIN)
    exe = str(tmp_path / "q")
    subprocess.run([cxx, "-O1", "-std=c++17", "-o", exe, str(tmp_path / "q.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
