// zfp.cu -- fixed-rate ZFP compression (Alg. 3, Sec. IV-C) on the GPU.
//
// The paper's outline: the field is cut into blocks of 4^d values, each
// block aligned to its largest exponent and made fixed point, decorrelated by
// a near-orthogonal transform, and its bit planes serialized most significant
// first and cut at a fixed number of bits.  Every block's output has the same
// size, so blocks need no coordination: one thread codes one block, with the
// block held in registers (all loops over the 4^d values unrolled) and its
// bits written straight to its own words; decoded rows leave a warp as whole
// lines.
//
// The details the paper leaves open are read as follows (the container, a
// 64-byte header and the block words, is documented with hpdr_zfp_compress
// in include/hpdr.h):
//   blocks      row-major over ceil(n_k / 4) blocks per dimension, values in
//               a block row-major (last index fastest); positions past the
//               array edge repeat the last in-range value of their dimension,
//               and are dropped on decoding.
//   exponent    emax = the binary exponent e of the block's largest magnitude
//               (x = f 2^e, 1/2 <= |f| < 1); a block of zeros codes a 0 flag.
//   fixed point q = trunc(x 2^(P - 5 - emax)), P = 32 (f32) or 64 (f64).
//   transform   along the last dimension, then the others in reverse order,
//               every line (a0..a3) becomes (S, D, d0, d1):
//                 s0 = floor((a0 + a1)/2), d0 = a0 - a1, s1 = floor((a2 + a3)/2),
//                 d1 = a2 - a3, S = floor((s0 + s1)/2), D = s0 - s1,
//               an exactly invertible integer S-transform (two Haar levels);
//               magnitudes stay below 2^(P-2) after three dimensions.
//   order       by the sum over dimensions of the class of the index within
//               the line (S 0, D 1, d0 and d1 2), ties in block order.
//   negabinary  u = (q + 0xAA..A) xor 0xAA..A in P-bit arithmetic.
//   coding      rate * 4^d bits per block (a multiple of 32): a flag bit,
//               EB = 9 (f32) or 12 (f64) exponent bits (emax + 2^(EB-1),
//               least significant first), then planes P-1..0: the bits of the
//               n coefficients already significant as they are, then group
//               tests (one bit: any of n.. set; after a 1 the coefficients'
//               bits from n up to and including the next 1); the block stops
//               where its budget ends, the rest of its bits zero.  Bits fill
//               32-bit words least significant first.
#include <cstdint>
#include <cstring>
#include <cmath>
#include "internal.cuh"

namespace hpdr {
namespace {

constexpr int kZfpThreads = 128;
constexpr int kZfpHdr = 64;

struct ZfpGeom {
    long long n[3];             // dims (row-major, last fastest), unused = 1
    long long nb[3];            // blocks per dim
    unsigned long long nblocks;
    uint32_t maxbits;           // bits per block
};

struct ZfpHdrBytes {
    uint8_t b[kZfpHdr];
};

// sequency order of a block of 4^D coefficients, built at compile time
template <int D>
struct SeqOrder {
    unsigned char p[64];
    constexpr SeqOrder() : p{}
    {
        int key[64] = {};
        const int cls[4] = {0, 1, 2, 2};
        const int B = 1 << (2 * D);
        for (int i = 0; i < B; i++) {
            int s = 0, r = i;
            for (int k = 0; k < D; k++) { s += cls[r % 4]; r /= 4; }
            key[i] = s;
        }
        int m = 0;
        for (int s = 0; s <= 2 * D; s++)
            for (int i = 0; i < B; i++)
                if (key[i] == s) p[m++] = (unsigned char)i;
    }
};

template <typename T> struct ZfpTypes;
template <> struct ZfpTypes<float> {
    typedef int32_t SI;
    typedef uint32_t UI;
    static constexpr int P = 32, EB = 9;
    static constexpr uint32_t M = 0xAAAAAAAAu;
};
template <> struct ZfpTypes<double> {
    typedef long long SI;
    typedef unsigned long long UI;
    static constexpr int P = 64, EB = 12;
    static constexpr unsigned long long M = 0xAAAAAAAAAAAAAAAAull;
};

// one line of the forward / inverse transform (arithmetic shifts = floor)
template <typename SI>
__device__ __forceinline__ void fwd_line(SI &a0, SI &a1, SI &a2, SI &a3)
{
    const SI s0 = (a0 + a1) >> 1, d0 = a0 - a1;
    const SI s1 = (a2 + a3) >> 1, d1 = a2 - a3;
    a0 = (s0 + s1) >> 1;
    a1 = s0 - s1;
    a2 = d0;
    a3 = d1;
}
// (s, d) -> (x, y): x + y = 2s + (d & 1), x - y = d; d + (d & 1) is even
template <typename SI>
__device__ __forceinline__ void inv_pair(SI s, SI d, SI &x, SI &y)
{
    x = s + ((d + (d & 1)) >> 1);
    y = x - d;
}
template <typename SI>
__device__ __forceinline__ void inv_line(SI &a0, SI &a1, SI &a2, SI &a3)
{
    SI s0, s1, x0, x1, x2, x3;
    inv_pair(a0, a1, s0, s1);
    inv_pair(s0, a2, x0, x1);
    inv_pair(s1, a3, x2, x3);
    a0 = x0; a1 = x1; a2 = x2; a3 = x3;
}

template <int D, typename SI>
__device__ __forceinline__ void fwd_block(SI *q)
{
    constexpr int B = 1 << (2 * D);
#pragma unroll
    for (int k = D - 1; k >= 0; k--) {
        const int st = 1 << (2 * (D - 1 - k));
#pragma unroll
        for (int i = 0; i < B; i++)
            if (((i / st) & 3) == 0) fwd_line(q[i], q[i + st], q[i + 2 * st], q[i + 3 * st]);
    }
}
template <int D, typename SI>
__device__ __forceinline__ void inv_block(SI *q)
{
    constexpr int B = 1 << (2 * D);
#pragma unroll
    for (int k = 0; k < D; k++) {
        const int st = 1 << (2 * (D - 1 - k));
#pragma unroll
        for (int i = 0; i < B; i++)
            if (((i / st) & 3) == 0) inv_line(q[i], q[i + st], q[i + 2 * st], q[i + 3 * st]);
    }
}

// position of block b: element offset of its first value, strides, and how many
// of its four positions along every dimension lie inside the array
struct BlockPos {
    long long base;
    long long st[3];
    int in[3];
};
template <int D>
__device__ __forceinline__ BlockPos block_pos(const ZfpGeom &g, unsigned long long b)
{
    BlockPos p;
    p.base = 0;
    long long stride = 1;
    unsigned long long r = b;
#pragma unroll
    for (int k = D - 1; k >= 0; k--) {
        const unsigned long long nb = (unsigned long long)g.nb[k];
        unsigned long long q;
        if (r >> 32 || nb >> 32) q = r / nb;
        else q = (uint32_t)r / (uint32_t)nb;   // the usual size: a 32-bit division
        const long long i = 4 * (long long)(r - q * nb);
        r = q;
        p.in[k] = g.n[k] - i < 4 ? (int)(g.n[k] - i) : 4;
        p.st[k] = stride;
        p.base += i * stride;
        stride *= g.n[k];
    }
    return p;
}
// element offset of position i of the block relative to its base, edge positions clamped
template <int D>
__device__ __forceinline__ long long value_offset(const BlockPos &p, int i)
{
    long long o = 0;
#pragma unroll
    for (int k = 0; k < D; k++) {
        const int j = (i >> (2 * (D - 1 - k))) & 3;
        o += (j < p.in[k] ? j : p.in[k] - 1) * p.st[k];
    }
    return o;
}
template <int D>
__device__ __forceinline__ bool value_inside(const BlockPos &p, int i)
{
    bool ok = true;
#pragma unroll
    for (int k = 0; k < D; k++) ok = ok && ((i >> (2 * (D - 1 - k))) & 3) < p.in[k];
    return ok;
}

// four words, or values, moved at once
struct alignas(16) Quad {
    uint32_t x, y, z, w;
};
template <typename T> struct alignas(16) Four {
    T v[4];
};

// the low n bits (1 <= n <= 32)
__device__ __forceinline__ uint32_t low_bits(int n) { return 0xFFFFFFFFu >> (32 - n); }

// bits of one block, least significant first.  The budget is a whole number of
// words, so what lies past it is dropped word by word: nothing is clipped on the
// way.  Blocks of whole 16-byte units are stored as such.
struct BitWriter {
    uint32_t *w;
    unsigned idx = 0, nwords;         // next word, words of the block
    bool quad;
    unsigned long long acc = 0;       // pending bits (fewer than 32)
    int nacc = 0;
    uint32_t q0 = 0, q1 = 0, q2 = 0;  // the last three words
    __device__ BitWriter(uint32_t *words, unsigned n) : w(words), nwords(n), quad(n % 4 == 0) {}
    __device__ __forceinline__ bool full() const { return idx >= nwords; }
    __device__ __forceinline__ void word(uint32_t x)
    {
        if (idx < nwords) {
            if (!quad) w[idx] = x;
            else if ((idx & 3u) == 3u) *reinterpret_cast<Quad *>(w + (idx - 3)) = Quad{q0, q1, q2, x};
        }
        q0 = q1; q1 = q2; q2 = x;
        idx++;
    }
    // append cnt bits (1 <= cnt <= 32; v has none above them)
    __device__ __forceinline__ void put(uint32_t v, int cnt)
    {
        acc |= (unsigned long long)v << nacc;
        nacc += cnt;
        if (nacc >= 32) {
            word((uint32_t)acc);
            acc >>= 32;
            nacc -= 32;
        }
    }
    __device__ __forceinline__ void zeros(int cnt)
    {
        for (; cnt > 0; cnt -= 32) put(0u, cnt > 32 ? 32 : cnt);
    }
    // write the pending bits and zero the block's remaining words
    __device__ __forceinline__ void finish()
    {
        if (nacc > 0) word((uint32_t)acc);
        while (idx < nwords) word(0u);
    }
};

// the block's bits, zeros after its end; at least 32 of them are always in buf.
// Blocks of whole aligned 16-byte units are read as such, one unit ahead.
struct BitReader {
    const uint32_t *w;
    unsigned idx = 0, nwords;
    bool quad;
    unsigned long long buf = 0;
    int nbuf = 0;
    Quad cur{}, nxt{};
    __device__ BitReader(const uint32_t *words, unsigned n)
        : w(words), nwords(n), quad(n % 4 == 0 && (reinterpret_cast<uintptr_t>(words) & 15) == 0)
    {
        if (quad) nxt = *reinterpret_cast<const Quad *>(w);
        refill();
    }
    __device__ __forceinline__ void refill()
    {
        if (nbuf >= 32) return;
        uint32_t x = 0;
        if (idx < nwords) {
            if (!quad) {
                x = w[idx];
            } else {
                if ((idx & 3u) == 0u) {
                    cur = nxt;
                    if (idx + 4 < nwords) nxt = *reinterpret_cast<const Quad *>(w + idx + 4);
                }
                x = cur.x;
                cur.x = cur.y; cur.y = cur.z; cur.z = cur.w;
            }
        }
        idx++;
        buf |= (unsigned long long)x << nbuf;
        nbuf += 32;
    }
    __device__ __forceinline__ uint32_t peek() const { return (uint32_t)buf; }
    __device__ __forceinline__ void skip(int cnt)   // cnt <= 32
    {
        buf >>= cnt;
        nbuf -= cnt;
        refill();
    }
    __device__ __forceinline__ bool done() const { return (long long)idx * 32 - nbuf >= (long long)nwords * 32; }
};

// Transpose of a 32 x 32 bit matrix: bit r of word c becomes bit c of word r.
// Blocks of 64 values turn their words into planes (and back) this way: 256
// operations for 32 planes of 32 values, where picking a plane's bits out of the
// words takes three operations a bit.
__device__ __forceinline__ void transpose32(uint32_t (&a)[32])
{
#pragma unroll
    for (int i = 0; i < 16; i++) {
        const uint32_t x = a[i], y = a[i + 16];
#ifdef __CUDA_ARCH__
        a[i] = __byte_perm(x, y, 0x5410);
        a[i + 16] = __byte_perm(x, y, 0x7632);
#else
        a[i] = (x & 0xFFFFu) | (y << 16);
        a[i + 16] = (x >> 16) | (y & 0xFFFF0000u);
#endif
    }
#pragma unroll
    for (int h = 0; h < 2; h++)
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const uint32_t x = a[16 * h + i], y = a[16 * h + i + 8];
#ifdef __CUDA_ARCH__
            a[16 * h + i] = __byte_perm(x, y, 0x6240);
            a[16 * h + i + 8] = __byte_perm(x, y, 0x7351);
#else
            a[16 * h + i] = (x & 0x00FF00FFu) | ((y & 0x00FF00FFu) << 8);
            a[16 * h + i + 8] = ((x >> 8) & 0x00FF00FFu) | (y & 0xFF00FF00u);
#endif
        }
    constexpr uint32_t m[3] = {0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int t = 0; t < 3; t++) {
        const int s = 4 >> t;
#pragma unroll
        for (int i = 0; i < 32; i++)
            if (!(i & s)) {
                const uint32_t x = a[i], y = a[i + s];
                a[i] = (x & m[t]) | ((y << s) & ~m[t]);
                a[i + s] = ((x >> s) & m[t]) | (y & ~m[t]);
            }
    }
}

// 2^e for -126 <= e <= 127
__device__ __forceinline__ float pow2f(int e)
{
    const uint32_t x = (uint32_t)(e + 127) << 23;
    float f;
    memcpy(&f, &x, 4);
    return f;
}

// the two conversions in binary64, out of line: for the rare blocks below
__attribute__((noinline)) __device__ int32_t to_fixed64(float v, int s) { return (int32_t)__double2ll_rz(ldexp((double)v, s)); }
__attribute__((noinline)) __device__ float from_fixed64(int32_t q, int e) { return (float)ldexp((double)q, e); }

// q = trunc(v 2^(P - 5 - emax)), emax the exponent of the largest magnitude mx.
// A power of two scales a binary32 value exactly (in two steps, since the power
// itself can leave the range; a result that underflows truncates to 0 all the
// same), so binary64, a sixty-fourth of whose rate this part has, is left to
// infinities, whose exponent is whatever frexp makes it.
template <int B>
__device__ __forceinline__ void to_fixed(const float (&v)[B], float mx, int emax, int32_t (&q)[B])
{
    const int s = 27 - emax;
    if (mx <= 3.402823466e38f) {
        const float f1 = pow2f(s / 2), f2 = pow2f(s - s / 2);
#pragma unroll
        for (int i = 0; i < B; i++) {
            const float x = v[i] * f1 * f2;
#ifdef __CUDA_ARCH__
            q[i] = (int32_t)x;   // 0 for a NaN
#else
            q[i] = x == x ? (int32_t)x : 0;
#endif
        }
    } else {
#pragma unroll
        for (int i = 0; i < B; i++) q[i] = to_fixed64(v[i], s);
    }
}
template <int B>
__device__ __forceinline__ void to_fixed(const double (&v)[B], double, int emax, long long (&q)[B])
{
#pragma unroll
    for (int i = 0; i < B; i++) q[i] = __double2ll_rz(ldexp(v[i], 59 - emax));
}
// v = q 2^(emax - (P - 5)), rounded once: in binary32 only where no value of q can
// make the product subnormal or infinite
template <int B>
__device__ __forceinline__ void from_fixed(const int32_t (&q)[B], int emax, float (&v)[B])
{
    const int e = emax - 27;
    if (e >= -126 && e <= 96) {
        const float f = pow2f(e);
#pragma unroll
        for (int i = 0; i < B; i++) v[i] = (float)q[i] * f;
    } else {
#pragma unroll
        for (int i = 0; i < B; i++) v[i] = from_fixed64(q[i], e);
    }
}
template <int B>
__device__ __forceinline__ void from_fixed(const long long (&q)[B], int emax, double (&v)[B])
{
#pragma unroll
    for (int i = 0; i < B; i++) v[i] = ldexp((double)q[i], emax - 59);
}

// Both directions are bound by instruction issue: one thread walks its block's
// bits, and the lanes of a warp meet different numbers of group tests.  A token (a
// test bit, the zeros and the coefficient's 1) is written or read at once, words
// move in units of 16 bytes, planes are transposed from and to words through local
// memory, and binary32 blocks scale in binary32.  300x431x517 binary32 at rate 8:
// encoding 920 -> 240 us, decoding 1014 -> 322 us.
template <typename T, int D>
__global__ void __launch_bounds__(kZfpThreads) zfp_encode_kernel(const T *__restrict__ u, uint32_t *__restrict__ out,
                                                                 ZfpGeom g)
{
    typedef ZfpTypes<T> Z;
    typedef typename Z::SI SI;
    typedef typename Z::UI UI;
    constexpr int B = 1 << (2 * D), P = Z::P, EB = Z::EB;
    constexpr SeqOrder<D> ord{};
    const unsigned long long b = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    if (b >= g.nblocks) return;
    const BlockPos bp = block_pos<D>(g, b);
    const T *ub = u + bp.base;
    T v[B];
    T mx = (T)0;
#pragma unroll
    for (int i = 0; i < B; i++) {
        v[i] = ub[value_offset<D>(bp, i)];
        const T a = v[i] < (T)0 ? -v[i] : v[i];
        mx = a > mx ? a : mx;
    }
    const unsigned nwords = g.maxbits / 32;
    BitWriter bw(out + b * nwords, nwords);
    if (!(mx > (T)0)) {
        bw.finish();   // a 0 flag
        return;
    }
    int emax;
    frexp((double)mx, &emax);
    bw.put(1u, 1);
    bw.put((uint32_t)(emax + (1 << (EB - 1))) & low_bits(EB), EB);
    SI q[B];
    to_fixed<B>(v, mx, emax, q);
    fwd_block<D>(q);
    UI w[B];
    UI any = 0;
#pragma unroll
    for (int r = 0; r < B; r++) {
        w[r] = ((UI)q[ord.p[r]] + (UI)Z::M) ^ (UI)Z::M;
        any |= w[r];
    }
    // the planes above the highest one set: a 0 test each
    int k = P - 1;
    while (k >= 0 && !((any >> k) & 1)) k--;
    bw.zeros(P - 1 - k);
    int n = 0;
    uint32_t pl[B == 64 ? 32 : 1][2];   // 32 planes of a block of 64
#pragma unroll
    for (int c = P / 32 - 1; c >= 0; c--) {
    if (P > 32 && (k < 32 * c || bw.full())) continue;   // binary64 at a low rate ends in its upper planes
    if constexpr (B == 64) {
#pragma unroll
        for (int h = 0; h < 2; h++) {
            uint32_t a[32];
#pragma unroll
            for (int r = 0; r < 32; r++) a[r] = (uint32_t)(w[32 * h + r] >> (32 * c));
            transpose32(a);
#pragma unroll
            for (int i = 0; i < 32; i++) pl[i][h] = a[i];
        }
    }
    for (; k >= 32 * c && !bw.full(); k--) {
        unsigned long long mask = 0;
        if constexpr (B == 64) {
            const int i = P > 32 ? k & 31 : k;
            mask = (unsigned long long)pl[i][1] << 32 | pl[i][0];
        } else {
#pragma unroll
            for (int r = 0; r < B; r++) mask |= (unsigned long long)((w[r] >> k) & 1) << r;
        }
        // the coefficients already significant, as they are
        if (n > 32) {
            bw.put((uint32_t)mask, 32);
            bw.put((uint32_t)(mask >> 32) & low_bits(n - 32), n - 32);
        } else if (n > 0) {
            bw.put((uint32_t)mask & low_bits(n), n);
        }
        if (n == B) continue;
        unsigned long long rest = mask >> n;   // n < B <= 64
        while (n < B) {
            if (!rest) { bw.put(0u, 1); break; }
            const int j = __ffsll((long long)rest) - 1;
            // test bit 1, then j zeros and the coefficient's 1
            if (j <= 30) {
                bw.put(1u | (2u << j), j + 2);
            } else {
                bw.put(1u, 32);
                int c = j - 30;
                if (c > 32) { bw.put(0u, 32); c -= 32; }
                bw.put(1u << (c - 1), c);
            }
            n += j + 1;
            rest = rest >> j >> 1;
        }
    }
    }
    bw.finish();
}

template <typename T, int D>
__global__ void __launch_bounds__(kZfpThreads) zfp_decode_kernel(const uint32_t *__restrict__ in, T *__restrict__ u,
                                                                 ZfpGeom g)
{
    typedef ZfpTypes<T> Z;
    typedef typename Z::SI SI;
    typedef typename Z::UI UI;
    constexpr int B = 1 << (2 * D), P = Z::P, EB = Z::EB;
    constexpr SeqOrder<D> ord{};
    const unsigned long long b = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    const bool live = b < g.nblocks;
    const unsigned nwords = g.maxbits / 32;
    T val[B];
#pragma unroll
    for (int i = 0; i < B; i++) val[i] = (T)0;
    BlockPos bp{};
    if (live) {
        bp = block_pos<D>(g, b);
        BitReader br(in + b * nwords, nwords);
        const bool flag = br.peek() & 1u;
        br.skip(1);
        if (flag) {
            const int emax = (int)(br.peek() & low_bits(EB)) - (1 << (EB - 1));
            br.skip(EB);
            UI w[B];
            uint32_t pl[B == 64 ? P : 1][2];
#pragma unroll
            for (int r = 0; r < B; r++) w[r] = 0;
            if constexpr (B == 64) {
#pragma unroll
                for (int k = 0; k < P; k++) pl[k][0] = pl[k][1] = 0u;
            }
            int n = 0, k = P - 1;
            for (; k >= 0 && !br.done(); k--) {
                unsigned long long mask = 0;
                // verbatim bits of coefficients 0..n-1
                if (n > 32) {
                    mask = br.peek();
                    br.skip(32);
                    mask |= (unsigned long long)(br.peek() & low_bits(n - 32)) << 32;
                    br.skip(n - 32);
                } else if (n > 0) {
                    mask = br.peek() & low_bits(n);
                    br.skip(n);
                }
                while (n < B) {
                    const uint32_t x = br.peek();
                    if (!(x & 1u)) { br.skip(1); break; }
                    const int j = __ffs((int)(x >> 1)) - 1;   // -1: no 1 among the next 31 bits
                    if (j >= 0 && j < B - n) {
                        br.skip(j + 2);
                        n += j + 1;
                        mask |= 1ull << (n - 1);
                        continue;
                    }
                    // a longer run of zeros; a malformed stream may run out at B
                    br.skip(1);
                    while (n < B) {
                        const int avail = B - n < 32 ? B - n : 32;
                        const uint32_t y = br.peek() & low_bits(avail);
                        if (!y) {
                            br.skip(avail);
                            n += avail;
                            continue;
                        }
                        const int i = __ffs((int)y) - 1;
                        br.skip(i + 1);
                        n += i + 1;
                        mask |= 1ull << (n - 1);
                        break;
                    }
                }
                if constexpr (B == 64) {
                    pl[k][0] = (uint32_t)mask;
                    pl[k][1] = (uint32_t)(mask >> 32);
                } else if (mask) {
#pragma unroll
                    for (int r = 0; r < B; r++) w[r] |= (UI)((mask >> r) & 1ull) << k;
                }
            }
            if constexpr (B == 64) {
#pragma unroll
                for (int h = 0; h < 2; h++)
#pragma unroll
                    for (int c = 0; c < P / 32; c++) {
                        if (P > 32 && c == 0 && k >= 31) continue;   // none of the lower planes was reached
                        uint32_t a[32];
#pragma unroll
                        for (int i = 0; i < 32; i++) a[i] = pl[32 * c + i][h];
                        transpose32(a);
#pragma unroll
                        for (int r = 0; r < 32; r++) w[32 * h + r] |= (UI)a[r] << (32 * c);
                    }
            }
            SI q[B];
#pragma unroll
            for (int r = 0; r < B; r++) q[ord.p[r]] = (SI)((w[r] ^ (UI)Z::M) - (UI)Z::M);
            inv_block<D>(q);
            from_fixed<B>(q, emax, val);
        }
    }
#ifdef __CUDA_ARCH__
    // binary64 rows of fewer dimensions are whole sectors as they are
    if constexpr (sizeof(T) == 8 && D < 3) {
        if (live) {
#pragma unroll
            for (int i = 0; i < B; i++)
                if (value_inside<D>(bp, i)) u[bp.base + value_offset<D>(bp, i)] = val[i];
        }
        return;
    }
    // A warp's blocks lie side by side along the last dimension: their rows of
    // four values meet in shared memory and leave as whole lines.  Value t = 32 it +
    // lane of a row of the warp belongs to lane t / 4 and sits at position t & 3.
    constexpr int R = B / 4, G = R < 4 ? R : 4;   // rows of a block, rows at a time
    __shared__ __align__(16) T sh[kZfpThreads / 32][G][128];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int in0 = D == 3 ? bp.in[0] : 1, in1 = D >= 2 ? bp.in[D - 2] : 1;   // rows inside: outer, inner dimension
    const int mine = live ? bp.in[D - 1] | in1 << 3 | in0 << 6 : 0;
    long long dst[4];
    int lim[4];   // rows inside of the value's block (inner | outer << 3), 0 if the value is outside
#pragma unroll
    for (int it = 0; it < 4; it++) {
        const int L = 8 * it + (lane >> 2), j = lane & 3;
        dst[it] = __shfl_sync(0xffffffffu, bp.base, L) + j;
        const int o = __shfl_sync(0xffffffffu, mine, L);
        lim[it] = j < (o & 7) ? o >> 3 : 0;
    }
    const long long s1 = D >= 2 ? bp.st[D >= 2 ? D - 2 : 0] : 0, s0 = D == 3 ? bp.st[0] : 0;
    const long long st1 = __shfl_sync(0xffffffffu, s1, 0), st0 = __shfl_sync(0xffffffffu, s0, 0);
#pragma unroll
    for (int r0 = 0; r0 < R; r0 += G) {
#pragma unroll
        for (int r = 0; r < G; r++) {
            const T *x = val + 4 * (r0 + r);
            *reinterpret_cast<Four<T> *>(&sh[wp][r][4 * lane]) = Four<T>{{x[0], x[1], x[2], x[3]}};
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < G; r++) {
            const int i0 = (r0 + r) >> 2, i1 = (r0 + r) & 3;
            T *row = u + (i0 * st0 + i1 * st1);
#pragma unroll
            for (int it = 0; it < 4; it++)
                if (i1 < (lim[it] & 7) && i0 < (lim[it] >> 3)) row[dst[it]] = sh[wp][r][32 * it + lane];
        }
        __syncwarp();
    }
#else
    if (live)
        for (int i = 0; i < B; i++)
            if (value_inside<D>(bp, i)) u[bp.base + value_offset<D>(bp, i)] = val[i];
#endif
}

__global__ void zfp_header_kernel(uint8_t *out, ZfpHdrBytes h)
{
    for (int i = threadIdx.x; i < kZfpHdr; i += blockDim.x) out[i] = h.b[i];
}

uint32_t zfp_crc32(const uint8_t *p, int n)
{
    uint32_t c = 0xFFFFFFFFu;
    for (int i = 0; i < n; i++) {
        c ^= p[i];
        for (int k = 0; k < 8; k++) c = (c >> 1) ^ (0xEDB88320u & (0u - (c & 1u)));
    }
    return ~c;
}

void zput32(uint8_t *p, uint32_t v) { for (int i = 0; i < 4; i++) p[i] = (uint8_t)(v >> (8 * i)); }
void zput64(uint8_t *p, uint64_t v) { for (int i = 0; i < 8; i++) p[i] = (uint8_t)(v >> (8 * i)); }
uint32_t zget32(const uint8_t *p) { uint32_t v = 0; for (int i = 0; i < 4; i++) v |= (uint32_t)p[i] << (8 * i); return v; }
uint64_t zget64(const uint8_t *p) { uint64_t v = 0; for (int i = 0; i < 8; i++) v |= (uint64_t)p[i] << (8 * i); return v; }

// geometry of a field at a rate; false on bad arguments
bool zfp_geom(int ndim, const size_t *dims, int dtype, uint32_t rate, ZfpGeom *g)
{
    if (ndim < 1 || ndim > 3 || !dims || (dtype != 0 && dtype != 1) || rate < 1 || rate > 256) return false;
    const uint32_t maxbits = rate << (2 * ndim);
    const int EB = dtype == 0 ? 9 : 12;
    if (maxbits % 32 || maxbits < (uint32_t)(EB + 2)) return false;
    memset(g, 0, sizeof(*g));
    g->nblocks = 1;
    for (int k = 0; k < 3; k++) {
        g->n[k] = k < ndim ? (long long)dims[k] : 1;
        if (g->n[k] < 1 || g->n[k] > (1ll << 40)) return false;
        g->nb[k] = (g->n[k] + 3) / 4;
        if (k < ndim) g->nblocks *= (unsigned long long)g->nb[k];
    }
    g->maxbits = maxbits;
    return true;
}

template <typename T>
cudaError_t launch_zfp(bool enc, int ndim, const void *src, void *dst, const ZfpGeom &g, cudaStream_t s)
{
    const unsigned grid = (unsigned)((g.nblocks + kZfpThreads - 1) / kZfpThreads);
    if (enc) {
        if (ndim == 1) zfp_encode_kernel<T, 1><<<grid, kZfpThreads, 0, s>>>((const T *)src, (uint32_t *)dst, g);
        else if (ndim == 2) zfp_encode_kernel<T, 2><<<grid, kZfpThreads, 0, s>>>((const T *)src, (uint32_t *)dst, g);
        else zfp_encode_kernel<T, 3><<<grid, kZfpThreads, 0, s>>>((const T *)src, (uint32_t *)dst, g);
    } else {
        if (ndim == 1) zfp_decode_kernel<T, 1><<<grid, kZfpThreads, 0, s>>>((const uint32_t *)src, (T *)dst, g);
        else if (ndim == 2) zfp_decode_kernel<T, 2><<<grid, kZfpThreads, 0, s>>>((const uint32_t *)src, (T *)dst, g);
        else zfp_decode_kernel<T, 3><<<grid, kZfpThreads, 0, s>>>((const uint32_t *)src, (T *)dst, g);
    }
    count_launch();
    return cudaGetLastError();
}

struct ZDevGuard {
    int prev = -1;
    bool changed = false;
    explicit ZDevGuard(int d)
    {
        cudaGetDevice(&prev);
        if (prev != d) changed = cudaSetDevice(d) == cudaSuccess;
    }
    ~ZDevGuard() { if (changed) cudaSetDevice(prev); }
};

}  // namespace
}  // namespace hpdr

using namespace hpdr;

extern "C" {

size_t hpdr_zfp_bound(int ndim, const size_t *dims, hpdr_dtype dtype, uint32_t rate)
{
    ZfpGeom g;
    if (!zfp_geom(ndim, dims, (int)dtype, rate, &g)) return 0;
    return (size_t)(kZfpHdr + g.nblocks * (g.maxbits / 8));
}

hpdr_status hpdr_zfp_compress(hpdr_ctx *ctx, const void *d_in, hpdr_dtype dtype, int ndim, const size_t *dims,
                              uint32_t rate, void *d_out, size_t out_capacity, size_t *out_bytes, void *stream)
{
    ZfpGeom g;
    if (!ctx || !d_in || !d_out || !out_bytes || !zfp_geom(ndim, dims, (int)dtype, rate, &g)) return HPDR_ERR_ARG;
    if (((uintptr_t)d_out & 15) || ((uintptr_t)d_in & ((dtype == HPDR_F64) ? 7 : 3))) return HPDR_ERR_ARG;
    const size_t total = (size_t)(kZfpHdr + g.nblocks * (g.maxbits / 8));
    if (out_capacity < total) return HPDR_ERR_CAPACITY;
    ZDevGuard dg(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    ZfpHdrBytes h;
    memset(&h, 0, sizeof(h));
    memcpy(h.b, "HPDZ", 4);
    zput32(h.b + 4, 1);
    zput32(h.b + 8, (uint32_t)dtype);
    zput32(h.b + 12, (uint32_t)ndim);
    for (int k = 0; k < 3; k++) zput64(h.b + 16 + 8 * k, k < ndim ? (uint64_t)dims[k] : 1);
    zput32(h.b + 40, rate);
    zput32(h.b + 44, g.maxbits);
    zput64(h.b + 48, g.nblocks);
    zput32(h.b + 60, zfp_crc32(h.b, 60));
    uint8_t *out = (uint8_t *)d_out;
    zfp_header_kernel<<<1, 64, 0, s>>>(out, h);
    count_launch();
    if (cudaGetLastError() != cudaSuccess) return HPDR_ERR_CUDA;
    cudaError_t e = dtype == HPDR_F32 ? launch_zfp<float>(true, ndim, d_in, out + kZfpHdr, g, s)
                                      : launch_zfp<double>(true, ndim, d_in, out + kZfpHdr, g, s);
    if (e != cudaSuccess) return HPDR_ERR_CUDA;
    *out_bytes = total;
    return HPDR_OK;
}

hpdr_status hpdr_zfp_inspect(const void *in, size_t in_bytes, hpdr_dtype *dtype, int *ndim, size_t *dims,
                             uint32_t *rate)
{
    if (!in || !dtype || !ndim || !dims || !rate) return HPDR_ERR_ARG;
    if (in_bytes < (size_t)kZfpHdr) return HPDR_ERR_FORMAT;
    uint8_t h[kZfpHdr];
    cudaPointerAttributes at;
    bool dev = cudaPointerGetAttributes(&at, in) == cudaSuccess &&
               (at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged);
    cudaGetLastError();
    if (dev) {
        if (cudaMemcpy(h, in, kZfpHdr, cudaMemcpyDeviceToHost) != cudaSuccess) return HPDR_ERR_CUDA;
    } else {
        memcpy(h, in, kZfpHdr);
    }
    if (memcmp(h, "HPDZ", 4) || zget32(h + 4) != 1 || zfp_crc32(h, 60) != zget32(h + 60)) return HPDR_ERR_FORMAT;
    const int dt = (int)zget32(h + 8), nd = (int)zget32(h + 12);
    size_t d[3];
    for (int k = 0; k < 3; k++) d[k] = (size_t)zget64(h + 16 + 8 * k);
    const uint32_t r = zget32(h + 40);
    ZfpGeom g;
    if (!zfp_geom(nd, d, dt, r, &g) || g.maxbits != zget32(h + 44) || g.nblocks != zget64(h + 48))
        return HPDR_ERR_FORMAT;
    if (kZfpHdr + g.nblocks * (g.maxbits / 8) > in_bytes) return HPDR_ERR_FORMAT;
    *dtype = (hpdr_dtype)dt;
    *ndim = nd;
    for (int k = 0; k < 3; k++) dims[k] = k < nd ? d[k] : 1;
    *rate = r;
    return HPDR_OK;
}

hpdr_status hpdr_zfp_decompress(hpdr_ctx *ctx, const void *d_in, size_t in_bytes, void *d_out, size_t out_capacity,
                                void *stream)
{
    if (!ctx || !d_in || !d_out) return HPDR_ERR_ARG;
    if ((uintptr_t)d_in & 15) return HPDR_ERR_ARG;
    ZDevGuard dg(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    if (cudaStreamSynchronize(s) != cudaSuccess) return HPDR_ERR_CUDA;
    hpdr_dtype dt;
    int nd;
    size_t dims[3];
    uint32_t rate;
    hpdr_status st = hpdr_zfp_inspect(d_in, in_bytes, &dt, &nd, dims, &rate);
    if (st != HPDR_OK) return st;
    ZfpGeom g;
    zfp_geom(nd, dims, (int)dt, rate, &g);
    size_t N = 1;
    for (int k = 0; k < nd; k++) N *= dims[k];
    const size_t esz = dt == HPDR_F64 ? 8 : 4;
    if (out_capacity < N * esz) return HPDR_ERR_CAPACITY;
    if ((uintptr_t)d_out & (esz - 1)) return HPDR_ERR_ARG;
    const uint8_t *in = (const uint8_t *)d_in + kZfpHdr;
    cudaError_t e = dt == HPDR_F32 ? launch_zfp<float>(false, nd, in, d_out, g, s)
                                   : launch_zfp<double>(false, nd, in, d_out, g, s);
    return e == cudaSuccess ? HPDR_OK : HPDR_ERR_CUDA;
}

}  // extern "C"
