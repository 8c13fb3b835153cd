// levels_dev.cuh -- device helpers shared by the level kernels (levels.cu,
// decomp.cu): the quantization decision, stream indices of the level-major
// coefficient order, escapes and dequantization.  Not part of the ABI.
#pragma once
#include "levels.cuh"

namespace hpdr {
namespace {

// The quantization decision (Sec. IV-A, Alg. 1: linear quantization of the
// coefficients with the level's bin q): k = sign(x) floor(|x| rho + 1/2),
// rho = 1/q rounded to binary64 and every operation rounded to binary64,
// whatever the data type, so that codes agree with a binary64 decision on
// the same coefficients everywhere but at half-bin ties.  Codes whose
// magnitude reaches 2^62 are clamped there (the escape store then flags them).
//
// Binary64 issue is slow on this part, so only the product and one addition use
// it below 2^30: adding 2^51 + 1/2 rounded down leaves floor(2 (p + 1/2)) in the
// low word (its last place is worth 1/2).  That is the floor of the exact
// p + 1/2; the rounded sum of the definition reaches the next integer only from
// p = n + 1/2 - ulp(p), whose low 20 bits are all ones (p < 2^30): such p, and
// larger ones, take the definition as it stands.  So does a NaN of either sign (an
// overflowed coefficient times a rho of zero): its code is refused.
__device__ __noinline__ long long quant_code_slow(double p)
{
    const double t = __dadd_rn(p, 0.5);
    if (t < 1073741824.0) return (long long)(int)floor(t);
    if (t < 4611686018427387904.0) return (long long)floor(t);
    return kEscMax;
}
template <typename T>
__device__ __forceinline__ long long quant_code(T x, double rho)
{
    const double p = __dmul_rn(fabs((double)x), rho);
    long long k;
    if ((unsigned)__double2hiint(p) < 0x41D00000u && (__double2loint(p) & 0xFFFFF) != 0xFFFFF)
        k = (unsigned)__double2loint(__dadd_rd(p, 2251799813685248.5)) >> 1;
    else
        k = quant_code_slow(p);
    return x < (T)0 ? -k : k;
}

// The same decision for a binary32 coefficient, in binary32 arithmetic on a
// double-word product (binary64 throughput is low on this part).  With
// rho = rho_hi + rho_lo (rho_hi = fl32(rho), rho_lo = fl32(rho - rho_hi)):
//   p = fl32(ax rho_hi); e = ax rho_hi - p exactly (one FMA); e2 = fl32(e + ax rho_lo),
// so ax rho = p + e2 to within about 2^-47 ax rho.  With n = rint(p) and
// d = p - n (exact), floor(ax rho + 1/2) = n + [d + e2 >= 1/2] - [d + e2 < -1/2],
// and both comparisons are exact (1/2 - d and -1/2 - d are representable
// whenever the result can change).  Valid while p < kSmallQuant = 2^22 (then
// ulp(p) <= 1/4, |d + e2| < 3/4, and n is an exact integer); the result
// differs from the binary64 decision only when ax rho lies within about
// 2^-46 ax rho of a half-integer.
constexpr float kSmallQuant = 4194304.0f;
__device__ __forceinline__ int quant_small_f32(float ax, float rho_hi, float rho_lo)
{
    const float p = __fmul_rn(ax, rho_hi);
    const float e = __fmaf_rn(ax, rho_hi, -p);
    const float e2 = __fmaf_rn(ax, rho_lo, e);
    const float n = rintf(p);
    const float d = __fsub_rn(p, n);
    return __float2int_rn(n) + (e2 >= __fsub_rn(0.5f, d) ? 1 : 0) - (e2 < __fsub_rn(-0.5f, d) ? 1 : 0);
}

__device__ __forceinline__ double rho64_of(const Scalars *sc, int l) { return sc->rho_d[l]; }


template <typename T> __device__ __forceinline__ T q_of(const Scalars *sc, int l);
template <> __device__ __forceinline__ float q_of<float>(const Scalars *sc, int l) { return sc->q_f[l]; }
template <> __device__ __forceinline__ double q_of<double>(const Scalars *sc, int l) { return sc->q[l]; }

// Stream index of the new nodes of row (p0, p1) of level l:
//   every node new (p0 or p1 new):        base + p2
//   p0 and p1 kept (only odd p2 new):     base + (p2 - 1) / 2
template <typename T>
__device__ __forceinline__ long long row_base(const LevelGeom<T> &g, long long plane_base, bool k0,
                                              int p1)
{
    const long long m2 = g.dim[2].m, mc2 = g.dim[2].mc;
    return plane_base + (long long)p1 * m2 - (k0 ? (long long)kept_before(p1) * mc2 : 0LL);
}
template <typename T>
__device__ __forceinline__ long long plane_base_of(const LevelGeom<T> &g, int p0)
{
    const long long m1 = g.dim[1].m, m2 = g.dim[2].m;
    const long long mc1 = g.dim[1].mc, mc2 = g.dim[2].mc;
    return g.Nprev + (long long)p0 * m1 * m2 - (long long)kept_before(p0) * mc1 * mc2;
}

// an escaped code (symbol 0) keeps its k at its stream position; the encoder
// writes it into the bitstream after the escape's codeword, as zigzag(k) in
// the container's payload width.  Returns the bit length of zigzag(k).
__device__ __forceinline__ unsigned escape_store(const QuantOut &qo, long long si, long long k)
{
    if (k >= kEscMax || k <= -kEscMax) atomicExch(&qo.sc->status, (unsigned int)DS_ARG);
    qo.esc[si] = k;
    const unsigned long long z = k >= 0 ? 2ULL * (unsigned long long)k : 2ULL * (unsigned long long)(-(k + 1)) + 1ULL;
    return 64u - (unsigned)__clzll((long long)z);
}

// An escape of a binary32 coefficient (|k| >= D/2): its exact code (the
// double-word decision below 2^22, binary64 above) stored at its stream
// position; returns the payload bit length.  Out of line: escapes are rare.
__device__ __noinline__ unsigned escape_f32(const QuantOut &qo, long long si, float w, float rho_f, float rho_lo,
                                            double rho)
{
    const float ax = fabsf(w);
    long long k;
    if (__fmul_rn(ax, rho_f) < kSmallQuant) {
        const int ki = quant_small_f32(ax, rho_f, rho_lo);
        k = w < 0.0f ? -(long long)ki : (long long)ki;
    } else {
        k = quant_code(w, rho);
    }
    return escape_store(qo, si, k);
}

// The fast half of that decision: y = x rho_hi + 3 2^22 rounded to nearest holds
// the integer n nearest to x rho_hi in its low bits, and r = x rho - n (two fused
// multiply-adds, exact to 2^-24) tells whether n is the code: |r| safely below
// 1/2 leaves one integer within 1/2 of x rho.  Everything else -- a half-bin
// point nearby, a product near 2^22 and beyond, a NaN -- answers false.
__device__ __forceinline__ bool quant_near_f32(float x, float rho_hi, float rho_lo, int &n)
{
    const float magic = 12582912.0f;
    const float y = __fmaf_rn(x, rho_hi, magic);
    const float nf = __fsub_rn(y, magic);
    const float r = __fmaf_rn(x, rho_lo, __fmaf_rn(x, rho_hi, -nf));
    n = __float_as_int(y) - 0x4B400000;
    return fabsf(r) < 0.49998f && fabsf(nf) < 4194000.0f;
}
// The other half, out of line: the symbol in the low half (0: an escape, stored
// at its stream position), the payload's bit length in the high half.
__device__ __noinline__ unsigned quant_far_f32(const QuantOut &qo, long long si, float w, float rho_hi, float rho_lo,
                                               double rho)
{
    const int halfD = (int)(qo.D / 2);
    const float ax = fabsf(w);
    int ki = halfD;   // a code of 2^22 or more: an escape
    if (__fmul_rn(ax, rho_hi) < kSmallQuant) ki = quant_small_f32(ax, rho_hi, rho_lo);
    if (ki < halfD) return (unsigned)(halfD + (w < 0.0f ? -ki : ki));
    return escape_f32(qo, si, w, rho_hi, rho_lo, rho) << 16;
}

// quantize one coefficient into the symbol stream, the global histogram and the escapes
template <typename T>
__device__ __forceinline__ void quant_emit(const QuantOut &qo, long long si, T w, double rho)
{
    long long k = quant_code(w, rho);
    long long s = k + (long long)(qo.D / 2);
    unsigned int sym;
    if (s >= 1 && s <= (long long)qo.D - 1) {
        sym = (unsigned int)s;
    } else {
        sym = 0;
        atomicMax(&qo.sc->esc_w, escape_store(qo, si, k));
    }
    qo.sym[si] = (uint16_t)sym;
    atomicAdd(&qo.hist[sym], 1ULL);
}

// The binary64 decision of a binary32 coefficient without binary64 arithmetic
// almost everywhere: the double-word product of quant_small_f32 leaves
// ax rho - n within 2^-24 of r = d + e2 (p < 2^22), so away from the decision
// points +-1/2 by 2^-16 the code is the one that quant_code gives; closer, and
// for codes of 2^22 and more, quant_code decides (one coefficient in 2^15).
__device__ __noinline__ long long quant_code_call(float x, double rho) { return quant_code(x, rho); }
__device__ __forceinline__ long long quant_exact(float x, double rho, float rho_hi, float rho_lo)
{
    const float ax = fabsf(x);
    const float p = __fmul_rn(ax, rho_hi);
    const float e2 = __fmaf_rn(ax, rho_lo, __fmaf_rn(ax, rho_hi, -p));
    const float n = rintf(p);
    const float r = __fadd_rn(__fsub_rn(p, n), e2);
    if (p < kSmallQuant && fabsf(fabsf(r) - 0.5f) > 1.52587890625e-5f) {
        const int k = __float2int_rn(n) + (r >= 0.5f ? 1 : 0) - (r < -0.5f ? 1 : 0);
        return x < 0.0f ? -k : k;
    }
    return quant_code_call(x, rho);
}
__device__ __forceinline__ long long quant_exact(double x, double rho, float, float) { return quant_code(x, rho); }

// one coefficient into the symbol stream, the global histogram and the escapes
template <typename T>
__device__ __forceinline__ void quant_emit_exact(const QuantOut &qo, long long si, T w, double rho, float rho_hi,
                                                 float rho_lo)
{
    const long long k = quant_exact(w, rho, rho_hi, rho_lo);
    const long long s = k + (long long)(qo.D / 2);
    unsigned int sym = 0;
    if (s >= 1 && s <= (long long)qo.D - 1) sym = (unsigned int)s;
    else atomicMax(&qo.sc->esc_w, escape_store(qo, si, k));
    qo.sym[si] = (uint16_t)sym;
    atomicAdd(&qo.hist[sym], 1ULL);
}

template <typename T>
__device__ __forceinline__ T dequant_sym(const SymIn &si_, unsigned s, long long idx, T q)
{
    if (s != 0) return mul_rn((T)((int)s - (int)(si_.D / 2)), q);
    return mul_rn((T)si_.esc[idx], q);
}

// Binary64 issue is slow on this part, so the expansion takes the value of a
// symbol from a table, 64 KB per level, which its blocks copy into shared memory
// (bytes: size of it, 0 without): round trip of 500x500x100 3386 -> 3337 us against
// the product at every node.  The restriction stays with
// the product: it waits for shared memory more than for the pipe.
template <typename T>
__host__ __device__ inline size_t deq_bytes(const SymIn &si)
{
    return sizeof(T) == 8 && si.deq ? sizeof(double) * si.D : 0;
}
// starts the copy of a level's table (all threads; cp.async, committed by the caller)
__device__ __forceinline__ void deq_stage(double *dst, const SymIn &si, int level)
{
    const double *src = si.deq + (size_t)level * si.D;
    for (unsigned i = 2 * threadIdx.x; i < si.D; i += 2 * blockDim.x)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst + i)), "l"(src + i) : "memory");
}
// The value of an escaped code k, (T)k.  Converting 64-bit integers (and anything
// to binary64) takes the FP64 pipe, and where it is one side of a selection it is
// done for every symbol; so codes convert through 32 bits -- exactly for binary64
// below 2^24, its bits widened in integers -- and the rest out of line (the
// expansion kept the FP64 pipe 79% busy in binary32: decompression of 513^3 1448 ->
// 1402 us, round trip of 500x500x100 binary64 3154 -> 2943).
__device__ __forceinline__ double widen_bits(float x)   // x: an integer
{
    const unsigned f = __float_as_uint(x);
    const unsigned hi = (f & 0x80000000u) | (((f & 0x7FFFFFFFu) >> 3) + 0x38000000u);
    return __hiloint2double(f ? (int)hi : 0, (int)(f << 29));
}
template <typename T>
__device__ __noinline__ T escape_value_wide(long long k) { return (T)k; }
template <typename T>
__device__ __forceinline__ T escape_value(long long k)
{
    const int lo = (int)k;
    if constexpr (sizeof(T) == 4) {
        if (lo == k) return (T)lo;
    } else {
        if (lo == k && abs(lo) < (1 << 24)) return widen_bits((float)lo);
    }
    return escape_value_wide<T>(k);
}
// Whether every escape of a container holds in 32 bits (its payload width, set with
// its bins): then the binary32 level kernels read and convert the low words only
// (decompression of 300x431x517 at 1e-4 1290 -> 1273 us, of 513^3 1419 -> 1409).
__device__ __forceinline__ bool narrow_escapes(const Scalars *sc) { return sc->esc_w <= 32u; }
// s - D/2 for a symbol s
template <typename T>
__device__ __forceinline__ T code_value(unsigned s, int halfD)
{
    if constexpr (sizeof(T) == 4) {
        // 2^23 + s is the word 0x4B000000 | s, and both it and the difference are exact
        return __fsub_rn(__uint_as_float(0x4B000000u | s), 8388608.0f + (float)halfD);
    } else {
        // a conversion to binary64 takes the FP64 pipe more than the product does;
        // binary32 holds the code exactly, and its bits widen in integers
        // (500x500x100 round trip, with the norm's halves: 3590 -> 3315 us)
        return widen_bits((float)((int)s - halfD));
    }
}
// value of symbol s != 0; after a rejected header the symbols are another
// stream's, and any of them has to stay inside the table
template <typename T>
__device__ __forceinline__ T dequant_code(const double *deq, unsigned s, int halfD, T q)
{
    if (sizeof(T) == 8 && deq) return (T)deq[min(s, 2u * (unsigned)halfD - 1u)];
    return mul_rn(code_value<T>(s, halfD), q);
}

template <typename T>
__device__ __forceinline__ T dequant(const SymIn &si_, long long idx, int level)
{
    return dequant_sym<T>(si_, si_.sym[idx], idx, q_of<T>(si_.sc, level));
}

template <typename T>
__device__ __forceinline__ int first_coarse_at_or_after(const DimTables<T> &d, int p)
{
    // smallest coarse j with cpos(j) >= p
    int j = p <= 0 ? 0 : (p + 1) >> 1;
    return j < d.mc ? j : d.mc - 1;
}


}  // namespace

// Planes whose offsets take 64 bits (a 2-D field is one plane).  With 64 bits for
// every field 513^3 compression took 1448 us instead of 1410, decompression 1463
// instead of 1397, a training step at 257^3 647 instead of 641.
template <typename T>
bool big_planes(const LevelGeom<T> &g) { return (long long)g.dim[1].m * g.dim[2].m >= 1ll << 31; }

// Coarse planes per CTA (segment) for a grid of `tiles` x segments CTAs.
int choose_segment(int mc0, long long tiles, int per_sm);

// Resident CTAs per SM of a kernel at a block size and dynamic shared memory.
template <typename K>
int resident_ctas(K kernel, int threads, size_t smem)
{
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem) != cudaSuccess) {
        cudaGetLastError();
        n = 1;
    }
    return n > 1 ? n : 1;
}

}  // namespace hpdr
