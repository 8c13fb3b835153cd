// levels.cu -- per-level pieces of the multilevel decomposition (Sec. IV-A,
// Alg. 1) and of its inverse that are not the plane-streaming level kernels
// (those are in decomp.cu), for sm_103a:
//   * the Thomas solves of the coarse mass matrix along each dimension;
//   * level 0 (quantized or stored as it is) and its inverse;
//   * the norms of the field and the level bins;
//   * coarse_kernel: every level whose arrays fit one CTA's shared memory,
//     and level 0, in a single launch;
//   * the dispatch of restriction requests to the plane pipelines.
#include <cfloat>
#include <type_traits>
#include "levels_dev.cuh"

namespace hpdr {
namespace {

constexpr int kNormBlocks = 152 * 8;

// --------------------------------------------------------------------------
// Thomas solves of the coarse mass matrix along one dimension (Alg. 1
// tridiag; the paper's Iterative abstraction: one sequential sweep per line,
// many lines in parallel).

template <typename T>
__global__ void __launch_bounds__(256)
solve_strided_kernel(T *b, const T *src, int n, long long stride, long long nlines, const T *__restrict__ sub,
                     const T *__restrict__ cp, const T *__restrict__ inv_den, T *vc, int sign)
{
    next_begin();
    long long line = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (line >= nlines) return;
    long long o = line / stride, i = line - o * stride;
    T *p = b + o * (long long)n * stride + i;
    const T *f = src + o * (long long)n * stride + i;   // the right-hand side: b, or an array that is kept
    T y = (T)0;
#pragma unroll 4
    for (int t = 0; t < n; t++) {
        y = mul_rn(fma_rn(-sub[t], y, f[(long long)t * stride]), inv_den[t]);
        p[(long long)t * stride] = y;
    }
    T x = (T)0;
    T *q = vc ? vc + o * (long long)n * stride + i : nullptr;
#pragma unroll 4
    for (int t = n - 1; t >= 0; t--) {
        x = fma_rn(-cp[t], x, p[(long long)t * stride]);
        if (sign == 0) p[(long long)t * stride] = x;
        else if (sign > 0) q[(long long)t * stride] = add_rn(q[(long long)t * stride], x);
        else q[(long long)t * stride] = sub_rn(q[(long long)t * stride], x);
    }
}

// One thread per line, 32 adjacent lines per warp (every step one coalesced
// row), the line swept in place in global memory: the loads of the next sixteen
// steps are in flight while the current sixteen are computed; the Thomas
// factors sit in shared memory.  Blocks of two warps: the sweeps are bound by
// the recurrence, in binary64 by the FP64 pipe of the SMs that hold a line, so
// lines have to spread over all SMs (256 threads before: 65 -> 56 us for the
// finest level of 500x500x100 in binary64).
constexpr int kSolvePre = 16;
constexpr int kSolveThreads = 64;

template <typename T>
__global__ void __launch_bounds__(kSolveThreads)
solve_stream_kernel(T *b, const T *src, int n, long long st, long long ostride, long long ninner, long long nlines,
                    const T *__restrict__ sub, const T *__restrict__ cp, const T *__restrict__ inv_den)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *csub = reinterpret_cast<T *>(smem_raw), *ccp = csub + n, *cinv = ccp + n;
    // the plan's tables do not change: staged before the wait
    for (int t = threadIdx.x; t < n; t += blockDim.x) { csub[t] = sub[t]; ccp[t] = cp[t]; cinv[t] = inv_den[t]; }
    next_begin();
    __syncthreads();
    const long long line = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (line >= nlines) return;
    long long o, i;
    if (ninner == 1) { o = line; i = 0; }
    else if (nlines <= 0xFFFFFFFFll) { o = (unsigned)line / (unsigned)ninner; i = line - o * ninner; }
    else { o = line / ninner; i = line - o * ninner; }     // 64-bit division only for huge grids
    T *p = b + o * ostride + i;
    const T *f = src + o * ostride + i;   // the right-hand side: b, or an array that is kept
    constexpr int P = kSolvePre;
    const int nfull = n / P;   // blocks of P steps
    // forward sweep: y_t = (d_t - sub_t y_{t-1}) / den_t
    T y = (T)0;
    T cur[P], nxt[P];
    if (nfull > 0) {
#pragma unroll
        for (int u = 0; u < P; u++) cur[u] = f[(long long)u * st];
    }
    for (int k = 0; k < nfull; k++) {
        const int t0 = k * P;
        if (k + 1 < nfull) {
#pragma unroll
            for (int u = 0; u < P; u++) nxt[u] = f[(long long)(t0 + P + u) * st];
        }
#pragma unroll
        for (int u = 0; u < P; u++) {
            y = mul_rn(fma_rn(-csub[t0 + u], y, cur[u]), cinv[t0 + u]);
            p[(long long)(t0 + u) * st] = y;
        }
#pragma unroll
        for (int u = 0; u < P; u++) cur[u] = nxt[u];
    }
    for (int t = nfull * P; t < n; t++) {
        y = mul_rn(fma_rn(-csub[t], y, f[(long long)t * st]), cinv[t]);
        p[(long long)t * st] = y;
    }
    // backward sweep: x_t = y_t - cp_t x_{t+1}, from the end
    T x = (T)0;
    const int ntail = n - nfull * P;
    for (int t = n - 1; t >= n - ntail; t--) {
        x = fma_rn(-ccp[t], x, p[(long long)t * st]);
        p[(long long)t * st] = x;
    }
    if (nfull > 0) {
#pragma unroll
        for (int u = 0; u < P; u++) cur[u] = p[(long long)((nfull - 1) * P + u) * st];
    }
    for (int k = nfull - 1; k >= 0; k--) {
        const int t0 = k * P;
        if (k > 0) {
#pragma unroll
            for (int u = 0; u < P; u++) nxt[u] = p[(long long)(t0 - P + u) * st];
        }
#pragma unroll
        for (int u = P - 1; u >= 0; u--) {
            x = fma_rn(-ccp[t0 + u], x, cur[u]);
            p[(long long)(t0 + u) * st] = x;
        }
#pragma unroll
        for (int u = 0; u < P; u++) cur[u] = nxt[u];
    }
}

template <typename T>
__device__ __forceinline__ void cp_async_elem(T *dst_smem, const T *src)
{
    if (sizeof(T) == 4)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst_smem)), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst_smem)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

// U steps of a Thomas sweep from step t0 on, every load issued before the
// recurrence (in a plain loop each load waits for the store before it): forward
// y_t = (p_t - sub_t y) inv_t in place, backward x_t = p_t - cp_t x down from t0
// with fin(t, x) taking the solution.  One warp's chain is bound by its issue
// rate, so the steps carry no bound checks.
template <int U, typename T>
__device__ __forceinline__ T sweep_fwd(T *p, int st, const T *sub, const T *inv, int t0, T y)
{
    T v[U], f[U], g[U];
#pragma unroll
    for (int u = 0; u < U; u++) { v[u] = p[(t0 + u) * st]; f[u] = sub[t0 + u]; g[u] = inv[t0 + u]; }
#pragma unroll
    for (int u = 0; u < U; u++) { y = mul_rn(fma_rn(-f[u], y, v[u]), g[u]); p[(t0 + u) * st] = y; }
    return y;
}
template <int U, typename T, typename Fin>
__device__ __forceinline__ T sweep_bwd(const T *p, int st, const T *cp, int t0, T x, Fin fin)
{
    T v[U], f[U];
#pragma unroll
    for (int u = 0; u < U; u++) { v[u] = p[(t0 - u) * st]; f[u] = cp[t0 - u]; }
#pragma unroll
    for (int u = 0; u < U; u++) { x = fma_rn(-f[u], x, v[u]); v[u] = x; }
    fin(t0, v);
    return x;
}
// both sweeps of a line of n nodes; fin(t, x): x[u] is the solution at t - u
template <typename T, typename Fin>
__device__ __forceinline__ void sweep_line(T *p, int st, int n, const T *sub, const T *cp, const T *inv, Fin fin)
{
    constexpr int U = sizeof(T) == 4 ? 8 : 4;
    T y = (T)0;
    int t = 0;
    for (; t + U <= n; t += U) y = sweep_fwd<U>(p, st, sub, inv, t, y);
    if (U > 4 && t + 4 <= n) { y = sweep_fwd<4>(p, st, sub, inv, t, y); t += 4; }
    for (; t < n; t++) y = sweep_fwd<1>(p, st, sub, inv, t, y);
    T x = (T)0;
    t = n - 1;
    for (; t + 1 >= U; t -= U) x = sweep_bwd<U>(p, st, cp, t, x, [&](int q, const T(&v)[U]) { fin(q, v); });
    if (U > 4 && t + 1 >= 4) { x = sweep_bwd<4>(p, st, cp, t, x, [&](int q, const T(&v)[4]) { fin(q, v); }); t -= 4; }
    for (; t >= 0; t--) x = sweep_bwd<1>(p, st, cp, t, x, [&](int q, const T(&v)[1]) { fin(q, v); });
}

// i / d by a multiply-high: exact for i d < 2^32, so for i and d below 2^16 (the
// arrays of the coarse block hold at most kCoarseSmem / 2 / sizeof(float) = 25600
// nodes); mul = 0 for d = 1
__device__ __forceinline__ unsigned small_div_mul(int d) { return 0xFFFFFFFFu / (unsigned)d + 1u; }
__device__ __forceinline__ int small_div(int i, unsigned mul)
{
    return mul == 0u ? i : (int)__umulhi((unsigned)i, mul);
}

// a contiguous run of cnt elements between global and shared memory in 16-byte
// pieces, single elements at its ends; dst and src agree modulo 16 bytes
__device__ __forceinline__ void cp_async16(void *dst_smem, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst_smem)), "l"(src) : "memory");
}
template <typename T> struct alignas(16) Four16 {
    T v[16 / sizeof(T)];
};
template <typename T>
__device__ __forceinline__ int run_head(const T *g, int cnt)
{
    const int h = (int)((16 - ((uintptr_t)g & 15)) & 15) / (int)sizeof(T);
    return h < cnt ? h : cnt;
}
// where element i of a run of lines of n sits in a tile of pitch n, or (pad) in one
// of pitch n + V, V a 16-byte piece; mul: small_div factor of the n / V pieces of a line
template <typename T>
__device__ __forceinline__ int tile_at(int i, bool pad, unsigned mul)
{
    constexpr int V = 16 / sizeof(T);
    return pad ? i + small_div(i / V, mul) * V : i;
}
template <typename T>
__device__ __forceinline__ void run_load(T *dst, const T *src, int cnt, bool pad, unsigned mul)
{
    constexpr int V = 16 / sizeof(T);
    const int h = run_head(src, cnt), nv = (cnt - h) / V;
    for (int i = threadIdx.x; i < nv; i += blockDim.x)
        cp_async16(dst + tile_at<T>(h + i * V, pad, mul), src + h + i * V);
    if ((int)threadIdx.x < h) cp_async_elem(dst + threadIdx.x, src + threadIdx.x);
    for (int i = h + nv * V + threadIdx.x; i < cnt; i += blockDim.x) cp_async_elem(dst + i, src + i);
}
// the tile src into the run dst: as it is (sign 0), or added to it or subtracted
template <typename T>
__device__ __forceinline__ void run_store(T *dst, const T *src, int cnt, bool pad, unsigned mul, int sign)
{
    constexpr int V = 16 / sizeof(T), U = 4;
    const auto take = [&](T old, T x) { return sign == 0 ? x : sign > 0 ? add_rn(old, x) : sub_rn(old, x); };
    // whole pieces where the tile sits like the run modulo 16 bytes
    const bool vec = (smem_u32(src) & 15) == ((uintptr_t)dst & 15);
    const int h = vec ? run_head(dst, cnt) : cnt, nv = (cnt - h) / V;
    for (int i0 = threadIdx.x; i0 < nv; i0 += U * blockDim.x) {
        Four16<T> o[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int i = i0 + u * (int)blockDim.x;
            if (sign != 0 && i < nv) o[u] = *reinterpret_cast<const Four16<T> *>(dst + h + i * V);
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int i = i0 + u * (int)blockDim.x;
            if (i >= nv) break;
            Four16<T> x = *reinterpret_cast<const Four16<T> *>(src + tile_at<T>(h + i * V, pad, mul));
#pragma unroll
            for (int k = 0; k < V; k++) x.v[k] = take(o[u].v[k], x.v[k]);
            *reinterpret_cast<Four16<T> *>(dst + h + i * V) = x;
        }
    }
    for (int i = threadIdx.x; i < h; i += blockDim.x) dst[i] = take(sign ? dst[i] : (T)0, src[tile_at<T>(i, pad, mul)]);
    for (int i = h + nv * V + threadIdx.x; i < cnt; i += blockDim.x) dst[i] = take(sign ? dst[i] : (T)0, src[tile_at<T>(i, pad, mul)]);
}

// Contiguous lines: a tile of up to 32 lines, one lane of a warp each.  A tile is one
// contiguous run of memory: it arrives by 16-byte asynchronous copies, and leaves by
// 16-byte stores that add it to v_c.  What counts is how many lines an SM holds at
// once, so v_c does not sit beside the tile (binary64 lines of 1001, eight in one CTA
// with their v_c: 896 us at 15x1500x2000, eighteen in two CTAs without: 444;
// lines of 257 at 513^3, 204 MB: 53 and 42).
// A line keeps the pitch n that it has in memory, so the lanes of a warp meet in
// gcd(n, 32) words of a bank; where n is a multiple of kContigPad the lines are a
// 16-byte piece further apart (binary64 lines of 8 at 2000x2000x15, in memory's pitch
// with the lanes a step apart: 250 us, like this: 65).
constexpr int kContigRows = 32;
constexpr int kContigPad = 8;
constexpr int kContigThreads = 128;
constexpr size_t kContigMaxKb = 220;
template <typename T>
__global__ void __launch_bounds__(kContigThreads)
solve_contig_kernel(T *b, const T *src, int n, long long nlines, int rows, bool pad, const T *__restrict__ sub, const T *__restrict__ cp,
                    const T *__restrict__ inv_den, T *vc, int sign)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int V = 16 / sizeof(T);
    T *csub = reinterpret_cast<T *>(smem_raw), *ccp = csub + n, *cinv = ccp + n;
    T *tile = csub + (3 * n + V - 1) / V * V;
    const int pitch = pad ? n + V : n;
    const unsigned mul = pad ? small_div_mul(n / V) : 0u;
    const long long row0 = blockIdx.x * (long long)rows, first = row0 * n;
    const int nr = (int)min((long long)rows, nlines - row0), cnt = nr * n;
    for (int t = threadIdx.x; t < n; t += blockDim.x) { csub[t] = sub[t]; ccp[t] = cp[t]; cinv[t] = inv_den[t]; }
    next_begin();
    // the right-hand side (b, or an array that is kept) where it sits modulo 16
    // bytes; the solution takes its place
    T *B = tile + ((uintptr_t)(src + first) & 15) / sizeof(T);
    run_load(B, src + first, cnt, pad, mul);
    cp_async_wait_all();
    __syncthreads();
    if ((int)threadIdx.x < nr) {
        T *p = B + threadIdx.x * pitch;
        sweep_line<T>(p, 1, n, csub, ccp, cinv, [&](int t, const auto &v) {
#pragma unroll
            for (int u = 0; u < (int)(sizeof(v) / sizeof(T)); u++) p[t - u] = v[u];
        });
    }
    __syncthreads();
    run_store(sign == 0 ? b + first : vc + first, B, cnt, pad, mul, sign);
}

// --------------------------------------------------------------------------
template <typename T, int SINK>
__global__ void level0_kernel(const T *v0, long long N0, T *coef_out, QuantOut qo)
{
    next_begin();
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= N0) return;
    T x = v0[i];
    if (SINK == (int)Sink::STREAM) { coef_out[i] = x; return; }
    quant_emit(qo, i, x, rho64_of(qo.sc, 0));
}

template <typename T, int SRC>
__global__ void level0_in_kernel(const T *coef_in, SymIn symin, long long N0, T *v0)
{
    next_begin();
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= N0) return;
    v0[i] = (SRC == (int)WSrc::STREAM) ? coef_in[i] : dequant<T>(symin, i, 0);
}

// --------------------------------------------------------------------------
// max|u| and sum u^2, then the level bins by the last block to finish: fixed
// grid, fixed per-thread order and a fixed tree over the blocks' partials ->
// deterministic.  Binary64 issue is slow on this part (about two lanes per
// cycle and SM), so a magnitude is compared as an integer (the order of
// non-negative values, with every NaN above infinity) and binary64 fields
// spend one binary64 instruction a value, the multiply-add of the sum, where
// they spent four (500 x 500 x 100: 300 -> 107 us).

template <typename T> struct BitsOf;
template <> struct BitsOf<float> { using type = unsigned; };
template <> struct BitsOf<double> { using type = unsigned long long; };
__device__ __forceinline__ unsigned abs_bits(float x) { return __float_as_uint(x) & 0x7FFFFFFFu; }
// (by halves: masking the whole word is recognised as an absolute value and sent
// through the FP64 pipe, which is what bounds the norm of a binary64 field: 25
// million values 108 -> 61 us)
__device__ __forceinline__ unsigned long long abs_bits(double x)
{
    return (unsigned long long)((unsigned)__double2hiint(x) & 0x7FFFFFFFu) << 32 | (unsigned)__double2loint(x);
}
__device__ __forceinline__ double abs_value(unsigned b) { return (double)__uint_as_float(b); }
__device__ __forceinline__ double abs_value(unsigned long long b) { return __longlong_as_double((long long)b); }

// the bins from the partials, by one block of 256 threads
__device__ __forceinline__ void bins_body(const BinArgs &ba, const volatile double *partials, int nparts, Scalars *sc)
{
    __shared__ unsigned long long smx[256];
    __shared__ double sss[256];
    // five loads in flight, then the sums in the order of the partials
    unsigned long long mx = 0;
    double ss = 0.0;
    constexpr int U = 5;
    for (int i0 = threadIdx.x; i0 < nparts; i0 += U * 256) {
        double m[U], v[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int i = i0 + 256 * u;
            m[u] = i < nparts ? partials[2 * i] : 0.0;
            v[u] = i < nparts ? partials[2 * i + 1] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            mx = max(mx, abs_bits(m[u]));
            ss += v[u];
        }
    }
    smx[threadIdx.x] = mx;
    sss[threadIdx.x] = ss;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) {
            smx[threadIdx.x] = max(smx[threadIdx.x], smx[threadIdx.x + s]);
            sss[threadIdx.x] += sss[threadIdx.x + s];
        }
        __syncthreads();
    }
    const double mxv = abs_value(smx[0]);
    ss = sss[0];
    if (threadIdx.x == 0) {
        sc->maxabs = mxv;
        sc->sumsq = ss;
    }
    const int L = ba.L;
    bool ok = mxv <= DBL_MAX;
    double nrm = ba.mode == 0 ? mxv : sqrt(__ddiv_rn(ss, (double)ba.N));
    double tau = ba.tol_kind == 1 ? __dmul_rn(ba.tol, nrm) : ba.tol;
    if (threadIdx.x == 0) sc->tau_abs = tau;
    double tp = 0.0;
    if (ok && mxv > 0.0) {
        tp = __dsub_rn(tau, __dmul_rn(__dmul_rn(__dmul_rn(32.0, (double)(L + 1)), ba.eps), mxv));
        if (!(tp > 0.0)) ok = false;
    }
    // one level per thread (two FP64 divisions each)
    for (int l = threadIdx.x; l <= L; l += blockDim.x) {
        double q;
        if (!ok || mxv == 0.0) q = 1.0;
        else if (l == 0) q = __ddiv_rn(__dmul_rn(2.0, tp), (double)(L + 1));
        else q = __ddiv_rn(__dmul_rn(2.0, tp), __dmul_rn((double)(L + 1), __dadd_rn(1.0, ba.c[l])));
        sc->q[l] = q;
        double r = __ddiv_rn(1.0, q);
        sc->rho_d[l] = r;
        sc->rho_f[l] = __double2float_rn(r);
        sc->rho_lo[l] = __double2float_rn(__dsub_rn(r, (double)sc->rho_f[l]));
        sc->q_f[l] = __double2float_rn(q);
    }
    if (!ok && threadIdx.x == 0) atomicExch(&sc->status, (unsigned int)DS_ARG);
}

template <typename T>
__global__ void __launch_bounds__(256) norm_kernel(const T *u, long long N, double *partials, BinArgs ba,
                                                   Scalars *sc)
{
    next_begin();
    typename BitsOf<T>::type mx = 0;
    T ssT = (T)0;   // per-thread partial sum in T (binary64 arithmetic is slow on this part)
    double ss = 0.0;
    const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long nth = (long long)gridDim.x * blockDim.x;
    constexpr int V = 16 / sizeof(T);
    const bool vec = (((uintptr_t)u) & 15) == 0;
    long long nv = vec ? N / V : 0;
    if (vec) {
        typedef typename std::conditional<sizeof(T) == 4, float4, double2>::type VT;
        const VT *uv = reinterpret_cast<const VT *>(u);
        for (long long i = tid; i < nv; i += nth) {
            VT x = __ldcs(uv + i);
            const T *e = reinterpret_cast<const T *>(&x);
#pragma unroll
            for (int k = 0; k < V; k++) {
                mx = max(mx, abs_bits(e[k]));
                ssT = fma_rn(e[k], e[k], ssT);
            }
        }
    }
    for (long long i = nv * V + tid; i < N; i += nth) {
        T x = u[i];
        mx = max(mx, abs_bits(x));
        ssT = fma_rn(x, x, ssT);
    }
    ss = (double)ssT;
    for (int o = 16; o > 0; o >>= 1) {
        mx = max(mx, __shfl_down_sync(0xffffffffu, mx, o));
        ss += __shfl_down_sync(0xffffffffu, ss, o);
    }
    __shared__ typename BitsOf<T>::type smx[8];
    __shared__ double sss[8];
    __shared__ bool last;
    int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) { smx[w] = mx; sss[w] = ss; }
    __syncthreads();
    if (threadIdx.x == 0) {
        typename BitsOf<T>::type m = smx[0];
        double s = sss[0];
        for (int i = 1; i < (int)(blockDim.x >> 5); i++) { m = max(m, smx[i]); s += sss[i]; }
        partials[2 * blockIdx.x] = abs_value(m);
        partials[2 * blockIdx.x + 1] = s;
        __threadfence();
        last = atomicAdd(&sc->blocks_done, 1u) + 1 == gridDim.x;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    bins_body(ba, partials, (int)gridDim.x, sc);
}

// --------------------------------------------------------------------------
// The coarse levels in one CTA.  Every level l <= ls (the largest level whose
// working arrays fit in shared memory) and level 0 run in a single 512-thread
// block out of shared memory, instead of four or five launches per level.  A
// level of compression (Alg. 1) here:
//   1. w = v - P v_c on the new nodes (0 on kept ones; v_c are the kept nodes
//      of v), quantized or written to the stream;
//   2. b = (x)_k P^T M_l w, dimension 2, then 1, then 0 (5 taps each);
//   3. z = (x)_k M_{l-1}^{-1} b, Thomas sweeps along dimension 0, 1, then 2;
//      the last sweep writes v_{l-1} = v_c + z.
// Recomposition runs the levels upwards: w from the stream, b and z as above,
// the last sweep writing v_c = v_{l-1} - z, then v = P v_c + w.  P v_c is the
// multilinear interpolant, taken along dimension 2, then 1, then 0.
//
// One block on one SM: the time is the chain of phases and the latency inside
// each, not throughput.  So
//   - everything a phase reads is put in shared memory once, by copies that
//     overlap each other: the level tables, the top grid or the stream prefix
//     [0, N_ls) of levels 0..ls (dequantized on the way), the bins;
//   - a thread owns a coarse cell: it loads the cell's eight corners and forms
//     the interpolant of its up to seven new nodes from them, where a thread
//     per node met every combination of new and kept dimensions as its own
//     branch and loaded 27 corners for 8 nodes;
//   - binary32 coefficients are quantized in binary32 (quant_exact): the
//     binary64 decision ran at two lanes per cycle and was half of the kernel;
//   - lines are swept in batches loaded ahead of the recurrence, and indices
//     are split by a multiply-high with precomputed factors.
// Levels 4..1 and 0 of a 513^3 FP32 field: 58 -> 24 us down, 60 -> 26 us up; of
// 129^2: 67 -> 27 and 69 -> 26 us (64 bit index divisions, tables read in global
// memory on every use and the binary64 quantizer before).
constexpr int kCoarseThreads = 512;

// element counts of the shared arrays for top level ls (host and device)
template <typename T>
__host__ __device__ inline void coarse_sizes(const LevelGeom<T> &g, long long &nl, long long &nc, long long &r2,
                                             long long &r1)
{
    const long long m0 = g.dim[0].m, m1 = g.dim[1].m, m2 = g.dim[2].m;
    const long long c0 = g.dim[0].mc, c1 = g.dim[1].mc, c2 = g.dim[2].mc;
    nl = m0 * m1 * m2;
    nc = c0 * c1 * c2;
    r2 = m0 * m1 * c2;
    r1 = m0 * c1 * c2;
}

// One dimension of one level.  Tables: wl[m], wr[m], tap[5 mc], sub[mc],
// cp[mc], inv[mc], in this order when they are staged.
template <typename T>
struct CoarseDim {
    const T *wl, *wr, *tap, *sub, *cp, *inv;
    int m, mc;
    unsigned mmul, cmul;   // small_div factors of m and mc
};
struct CoarseExt {
    int m, mc, off;
    unsigned mmul, cmul;
};
__host__ __device__ inline int coarse_tab_elems(int m, int mc) { return 2 * m + 8 * mc; }

// dimension k of level l; STG: the tables sit at `extra` + their offset
template <typename T, bool STG>
__device__ __forceinline__ CoarseDim<T> coarse_dim(const CoarseArgs<T> &a, const CoarseExt &e, const T *extra, int l,
                                                   int k)
{
    CoarseDim<T> c;
    c.m = e.m; c.mc = e.mc; c.mmul = e.mmul; c.cmul = e.cmul;
    if (STG) {
        const T *t = extra + e.off;
        c.wl = t; c.wr = t + e.m; c.tap = t + 2 * e.m;
        c.sub = t + 2 * e.m + 5 * e.mc; c.cp = t + 2 * e.m + 6 * e.mc; c.inv = t + 2 * e.m + 7 * e.mc;
    } else {
        const DimTables<T> &g = a.g[l].dim[k];
        c.wl = g.wl; c.wr = g.wr; c.tap = g.tap; c.sub = g.sub; c.cp = g.cp; c.inv = g.inv_den;
    }
    return c;
}

// the coarse cell at (j0, j1, j2): whether a new node follows along each
// dimension, and the weights of that node
template <typename T>
struct CoarseCell {
    int p[3];
    bool h[3];
    T wl[3], wr[3];
};
template <typename T>
__device__ __forceinline__ CoarseCell<T> coarse_cell(const CoarseDim<T> *d, const int j[3])
{
    CoarseCell<T> c;
#pragma unroll
    for (int k = 0; k < 3; k++) {
        c.p[k] = cpos_of(d[k].m, d[k].mc, j[k]);
        c.h[k] = j[k] + 1 < d[k].mc && c.p[k] + 2 == cpos_of(d[k].m, d[k].mc, j[k] + 1);
        c.wl[k] = c.h[k] ? d[k].wl[c.p[k] + 1] : (T)0;
        c.wr[k] = c.h[k] ? d[k].wr[c.p[k] + 1] : (T)0;
    }
    return c;
}

// multilinear interpolant at the cell's nodes (index 4 q0 + 2 q1 + q2; q = 1:
// the new node of that dimension) from its corners X[o0][o1][o2] around X[0],
// the other corner of dimension k at offset s[k] (0 without a new node);
// dimension 2, then 1, then 0
template <typename T>
__device__ __forceinline__ void coarse_interp(const CoarseCell<T> &c, const T *X, const int s[3], T r[8])
{
    auto lerp = [&](int k, T x, T y) { return fma_rn(c.wr[k], y, mul_rn(c.wl[k], x)); };
    T v[2][2][2];   // [side of dimension 0][side of dimension 1][kept, new column]
#pragma unroll
    for (int a = 0; a < 2; a++)
#pragma unroll
        for (int b = 0; b < 2; b++) {
            const T *x = X + a * s[0] + b * s[1];
            const T x0 = x[0], x1 = x[s[2]];
            v[a][b][0] = x0;
            v[a][b][1] = lerp(2, x0, x1);
        }
#pragma unroll
    for (int q2 = 0; q2 < 2; q2++) {
        const T y0 = lerp(1, v[0][0][q2], v[0][1][q2]), y1 = lerp(1, v[1][0][q2], v[1][1][q2]);
        r[q2] = v[0][0][q2];
        r[2 + q2] = y0;
        r[4 + q2] = lerp(0, v[0][0][q2], v[1][0][q2]);
        r[6 + q2] = lerp(0, y0, y1);
    }
}

// f(q, p-offset, stream offset) for every new node of the cell: q as in
// coarse_interp, the node's flat index relative to the cell's kept node, and
// its index in the level's section of the stream
template <typename T, typename F>
__device__ __forceinline__ void coarse_new_nodes(const CoarseCell<T> &c, const int j[3], int m1, int m2, int c1, int c2,
                                                 F f)
{
    const int base = (c.p[0] * m1 + c.p[1]) * m2 + c.p[2];
#pragma unroll
    for (int q = 1; q < 8; q++) {
        const int q0 = q >> 2, q1 = (q >> 1) & 1, q2 = q & 1;
        if ((q0 && !c.h[0]) || (q1 && !c.h[1]) || (q2 && !c.h[2])) continue;
        const int off = (q0 * m1 + q1) * m2 + q2;
        // kept nodes before it: whole planes, then rows, then columns
        int cr = (j[0] + q0) * c1 * c2;
        if (!q0) cr += (j[1] + q1) * c2;
        if (!q0 && !q1) cr += j[2] + 1;
        f(q, off, base + off - cr);
    }
}

// out = in restricted along dimension k with the 5 taps of P^T M_l; in has
// extents n0 x n1 x n2 (extent k = m), out the same with extent k = mc;
// mul2, mul1: small_div factors of out's extents 2 and 1
template <typename T, int k>
__device__ __forceinline__ void coarse_restrict(const CoarseDim<T> &d, int n0, int n1, int n2, unsigned mul2,
                                                unsigned mul1, const T *in, T *out)
{
    const int m = d.m, mc = d.mc;
    const int o0 = k == 0 ? mc : n0, o1 = k == 1 ? mc : n1, o2 = k == 2 ? mc : n2;
    const int is = k == 0 ? n1 * n2 : k == 1 ? n2 : 1;
    const int tot = o0 * o1 * o2;
    const T *tap = d.tap;
    for (int idx = threadIdx.x; idx < tot; idx += blockDim.x) {
        const int r = small_div(idx, mul2), j2 = idx - r * o2, j0 = small_div(r, mul1), j1 = r - j0 * o1;
        const int jk = k == 0 ? j0 : k == 1 ? j1 : j2;
        const int c = cpos_of(m, mc, jk);
        const T *x = in + ((k == 0 ? c : j0) * n1 + (k == 1 ? c : j1)) * n2 + (k == 2 ? c : j2);
        T t[5], y[5];
#pragma unroll
        for (int o = -2; o <= 2; o++) {
            const bool inside = (unsigned)(c + o) < (unsigned)m;
            t[o + 2] = tap[jk * 5 + o + 2];
            y[o + 2] = x[inside ? o * is : 0];
        }
        T acc = (T)0;
#pragma unroll
        for (int o = -2; o <= 2; o++) {
            const T z = fma_rn(t[o + 2], y[o + 2], acc);
            acc = (unsigned)(c + o) < (unsigned)m ? z : acc;
        }
        out[idx] = acc;
    }
    __syncthreads();
}

// b = (x)_k P^T M_l W, then z = (x)_k M_{l-1}^{-1} b in place (R2, R1, B
// scratch).  out[j] = sign z + base at the coarse node (j0, j1, t) of flat index
// j, with base read at base0(j0, j1) + at(t) (the dimension-2 sweep always runs:
// a field's last dimension is active)
template <typename T, bool SUB, typename Base, typename At>
__device__ __forceinline__ void coarse_correct(const CoarseDim<T> *d, const T *W, T *R2, T *R1, T *B, T *out, Base base0,
                                               At at)
{
    const int c0 = d[0].mc, c1 = d[1].mc, c2 = d[2].mc, m0 = d[0].m, m1 = d[1].m;
    // an inactive dimension (one node) keeps its values: no pass
    T *const rhs = m0 > 1 ? B : m1 > 1 ? R1 : R2;
    coarse_restrict<T, 2>(d[2], m0, m1, d[2].m, d[2].cmul, d[1].mmul, W, R2);
    if (m1 > 1) coarse_restrict<T, 1>(d[1], m0, m1, c2, d[2].cmul, d[1].cmul, R2, R1);
    if (m0 > 1) coarse_restrict<T, 0>(d[0], m0, c1, c2, d[2].cmul, d[1].cmul, m1 > 1 ? R1 : R2, B);
    if (m0 > 1) {
        const int pl = c1 * c2;
        for (int i = threadIdx.x; i < pl; i += blockDim.x) {
            T *p = rhs + i;
            sweep_line<T>(p, pl, c0, d[0].sub, d[0].cp, d[0].inv, [&](int t, const auto &v) {
#pragma unroll
                for (int u = 0; u < (int)(sizeof(v) / sizeof(T)); u++) p[(t - u) * pl] = v[u];
            });
        }
        __syncthreads();
    }
    if (m1 > 1) {
        for (int i = threadIdx.x; i < c0 * c2; i += blockDim.x) {
            const int j0 = small_div(i, d[2].cmul);
            T *p = rhs + j0 * c1 * c2 + (i - j0 * c2);
            sweep_line<T>(p, c2, c1, d[1].sub, d[1].cp, d[1].inv, [&](int t, const auto &v) {
#pragma unroll
                for (int u = 0; u < (int)(sizeof(v) / sizeof(T)); u++) p[(t - u) * c2] = v[u];
            });
        }
        __syncthreads();
    }
    for (int i = threadIdx.x; i < c0 * c1; i += blockDim.x) {
        const int j0 = small_div(i, d[1].cmul), j1 = i - j0 * c1;
        const T *src = base0(j0, j1);
        T *dst = out + i * c2;
        sweep_line<T>(rhs + i * c2, 1, c2, d[2].sub, d[2].cp, d[2].inv, [&](int t, const auto &v) {
            constexpr int U = sizeof(v) / sizeof(T);
            T old[U];
#pragma unroll
            for (int u = 0; u < U; u++) old[u] = src[at(t - u)];
#pragma unroll
            for (int u = 0; u < U; u++) dst[t - u] = SUB ? sub_rn(old[u], v[u]) : add_rn(old[u], v[u]);
        });
    }
    __syncthreads();
}

// MODE 0: compression (quantize), 1: decomposition (coefficient stream),
// 2: decompression (symbols), 3: recomposition (coefficient stream)
template <typename T, int MODE, bool STG>
__device__ __forceinline__ void coarse_body(const CoarseArgs<T> &a)
{
    extern __shared__ __align__(16) unsigned char coarse_smem[];
    __shared__ CoarseExt sext[kCoarseMaxLevels + 1][3];
    __shared__ int snprev[kCoarseMaxLevels + 1];    // first stream index of every level
    __shared__ T sq[kCoarseMaxLevels + 1];          // MODE 2: q of every level
    const int ls = a.ls, tid = threadIdx.x, nt = blockDim.x, N0 = (int)a.N0;
    long long nl_, nc_, r2_, r1_;
    coarse_sizes<T>(a.g[ls], nl_, nc_, r2_, r1_);
    const int nl = (int)nl_, nc = (int)nc_;
    T *VA = reinterpret_cast<T *>(coarse_smem);   // [nl]
    T *VB = VA + nl;                                // [nc]
    T *W = VB + nc;                                 // [nl]
    T *R2 = W + nl;                                 // [r2]
    T *R1 = R2 + (int)r2_;                          // [r1]
    T *B = R1 + (int)r1_;                           // [nc]
    T *VK = B + nc;                                 // [nc]
    T *const extra = VK + nc;                       // staged stream prefix, staged tables
    const bool stream = MODE >= 2 && a.stream_off >= 0;
    const T *const S = extra + (stream ? a.stream_off : 0);

    // ---- staging
    for (int i = tid; i < 3 * ls; i += nt) {
        const int l = 1 + i / 3, k = i - (l - 1) * 3;
        const DimTables<T> &g = a.g[l].dim[k];
        sext[l][k] = {g.m, g.mc, a.tab_off[l][k], small_div_mul(g.m), small_div_mul(g.mc)};
    }
    if (tid <= ls) {
        snprev[tid] = tid ? (int)a.g[tid].Nprev : 0;
        if (MODE == 2) sq[tid] = q_of<T>(a.symin.sc, tid);
    }
    if (STG)
        for (int task = tid >> 5; task < 18 * ls; task += nt >> 5) {
            const int l = 1 + task / 18, r = task - (l - 1) * 18, k = r / 6, w = r - k * 6;
            const DimTables<T> &g = a.g[l].dim[k];
            if (!(g.m > 1)) continue;
            const T *src = w == 0 ? g.wl : w == 1 ? g.wr : w == 2 ? g.tap : w == 3 ? g.sub : w == 4 ? g.cp : g.inv_den;
            const int cnt = w < 2 ? g.m : w == 2 ? 5 * g.mc : g.mc;
            T *dst = extra + a.tab_off[l][k] + (w < 2 ? w * g.m : 2 * g.m + (w == 2 ? 0 : (w + 2) * g.mc));
            for (int i = tid & 31; i < cnt; i += 32) cp_async_elem(dst + i, src + i);
        }
    if (MODE <= 1) for (int i = tid; i < nl; i += nt) cp_async_elem(VA + i, a.v_in + i);
    if (MODE == 3 && stream) for (int i = tid; i < nl; i += nt) cp_async_elem(extra + a.stream_off + i, a.coef_in + i);
    if (MODE == 2 && stream) {
        // symbols, then the codes of the escaped ones: every load of a batch in
        // flight before the first use
        T *const So = extra + a.stream_off;
        constexpr int U = 10;
        bool first = true;
        for (int i0 = tid; i0 < nl || first; i0 += U * nt) {
            unsigned sv[U];
            long long ev[U];
#pragma unroll
            for (int u = 0; u < U; u++) sv[u] = i0 + u * nt < nl ? a.symin.sym[i0 + u * nt] : 1u;
#pragma unroll
            for (int u = 0; u < U; u++) ev[u] = sv[u] == 0u ? a.symin.esc[i0 + u * nt] : 0;
            if (first) __syncthreads();   // the bins and the level starts
            first = false;
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int i = i0 + u * nt;
                if (i >= nl) continue;
                int l = 0;
                while (l < ls && i >= snprev[l + 1]) l++;
                So[i] = sv[u] != 0u ? mul_rn(code_value<T>(sv[u], (int)(a.symin.D / 2)), sq[l]) : mul_rn(escape_value<T>(ev[u]), sq[l]);
            }
        }
    }
    cp_async_wait_all();
    __syncthreads();

    if (MODE <= 1) {
        T *V = VA, *Vn = VB;
        for (int l = ls; l >= 0; l--) {
            // quantization constants of this level, off the critical path of the phases
            double rho = 0.0;
            float rhi = 0.f, rlo = 0.f;
            if (MODE == 0) { rho = rho64_of(a.qo.sc, l); rhi = a.qo.sc->rho_f[l]; rlo = a.qo.sc->rho_lo[l]; }
            auto put = [&](long long si, T w) {
                if (MODE == 0) quant_emit_exact(a.qo, si, w, rho, rhi, rlo);
                else a.coef_out[si] = w;
            };
            if (l == 0) {
                for (int i = tid; i < N0; i += nt) put((long long)i, V[i]);
                break;
            }
            const CoarseDim<T> d[3] = {coarse_dim<T, STG>(a, sext[l][0], extra, l, 0),
                                       coarse_dim<T, STG>(a, sext[l][1], extra, l, 1),
                                       coarse_dim<T, STG>(a, sext[l][2], extra, l, 2)};
            const int m0 = d[0].m, m1 = d[1].m, m2 = d[2].m, c0 = d[0].mc, c1 = d[1].mc, c2 = d[2].mc;
            const int np = snprev[l];
            // 1. coefficients of the new nodes
#pragma unroll 1
            for (int i = tid; i < c0 * c1 * c2; i += nt) {
                const int r = small_div(i, d[2].cmul), j0 = small_div(r, d[1].cmul);
                const int j[3] = {j0, r - j0 * c1, i - r * c2};
                const CoarseCell<T> c = coarse_cell<T>(d, j);
                const int base = (c.p[0] * m1 + c.p[1]) * m2 + c.p[2];
                const int st[3] = {c.h[0] ? 2 * m1 * m2 : 0, c.h[1] ? 2 * m2 : 0, c.h[2] ? 2 : 0};
                T x[8];
                coarse_interp<T>(c, V + base, st, x);
                W[base] = (T)0;
                coarse_new_nodes<T>(c, j, m1, m2, c1, c2, [&](int q, int off, int so) {
                    const T w = sub_rn(V[base + off], x[q]);
                    W[base + off] = w;
                    put((long long)np + so, w);
                });
            }
            __syncthreads();
            // 2.-3.
            coarse_correct<T, false>(
                d, W, R2, R1, B, Vn,
                [&](int j0, int j1) { return V + (cpos_of(m0, c0, j0) * m1 + cpos_of(m1, c1, j1)) * m2; },
                [&](int t) { return cpos_of(m2, c2, t); });
            T *t = V; V = Vn; Vn = t;
        }
    } else {
        T *V = VA, *Vn = VB;
        // the same ping-pong as compression, run backwards: level l's grid lands
        // where compression read it (the top level's would be VA)
        if ((ls & 1) == 1) { V = VB; Vn = VA; }
        // value of stream index i of level l
        auto value = [&](int i, int l) -> T {
            if (stream) return S[i];
            if (MODE == 2) return dequant_sym<T>(a.symin, a.symin.sym[i], i, sq[l]);
            return a.coef_in[i];
        };
        for (int i = tid; i < N0; i += nt) V[i] = value(i, 0);
        for (int l = 1; l <= ls; l++) {
            const CoarseDim<T> d[3] = {coarse_dim<T, STG>(a, sext[l][0], extra, l, 0),
                                       coarse_dim<T, STG>(a, sext[l][1], extra, l, 1),
                                       coarse_dim<T, STG>(a, sext[l][2], extra, l, 2)};
            const int m1 = d[1].m, m2 = d[2].m, c0 = d[0].mc, c1 = d[1].mc, c2 = d[2].mc;
            const int np = snprev[l];
            auto cell = [&](int i, int j[3]) {
                const int r = small_div(i, d[2].cmul);
                j[0] = small_div(r, d[1].cmul);
                j[1] = r - j[0] * c1;
                j[2] = i - r * c2;
                return coarse_cell<T>(d, j);
            };
#pragma unroll 1
            for (int i = tid; i < c0 * c1 * c2; i += nt) {
                int j[3];
                const CoarseCell<T> c = cell(i, j);
                const int base = (c.p[0] * m1 + c.p[1]) * m2 + c.p[2];
                W[base] = (T)0;
                coarse_new_nodes<T>(c, j, m1, m2, c1, c2, [&](int, int off, int so) { W[base + off] = value(np + so, l); });
            }
            __syncthreads();
            coarse_correct<T, true>(
                d, W, R2, R1, B, VK, [&](int j0, int j1) { return V + (j0 * c1 + j1) * c2; }, [&](int t) { return t; });
            auto expand = [&](T *dst) {
#pragma unroll 1
                for (int i = tid; i < c0 * c1 * c2; i += nt) {
                    int j[3];
                    const CoarseCell<T> c = cell(i, j);
                    const int base = (c.p[0] * m1 + c.p[1]) * m2 + c.p[2];
                    const int st[3] = {c.h[0] ? c1 * c2 : 0, c.h[1] ? c2 : 0, c.h[2] ? 1 : 0};
                    T x[8];
                    coarse_interp<T>(c, VK + i, st, x);
                    dst[base] = x[0];
                    coarse_new_nodes<T>(c, j, m1, m2, c1, c2, [&](int q, int off, int) {
                        dst[base + off] = add_rn(W[base + off], x[q]);
                    });
                }
            };
            if (l == ls) { expand(a.v_out); break; }
            expand(Vn);
            __syncthreads();
            T *t = V; V = Vn; Vn = t;
        }
    }
}

template <typename T, int MODE>
__global__ void __launch_bounds__(kCoarseThreads, 1) coarse_kernel(CoarseArgs<T> a)
{
    next_begin();
    if (a.staged) coarse_body<T, MODE, true>(a);
    else coarse_body<T, MODE, false>(a);
}

// one field per block (compression)
template <typename T>
__global__ void __launch_bounds__(kCoarseThreads, 1) coarse_batch_kernel(const CoarseArgs<T> *jobs)
{
    const CoarseArgs<T> &a = jobs[blockIdx.x];
    if (a.staged) coarse_body<T, 0, true>(a);
    else coarse_body<T, 0, false>(a);
}

// The coarse levels of the adjoint of recomposition in one CTA, like
// coarse_kernel: for l = ls..1, from the level-l gradient g_l,
//   g_{l-1} = P^T g_l,   y = (x)_k M_{l-1}^{-1} g_{l-1},
//   g_{c_l} = g_l - (x)_k M_l P_k y at the new nodes,
// and g_{c_0} = g_0.  Latency-bound: five launches a level took 100 us with their
// gaps on grids this small (257^3, levels 4..1), one CTA takes 18 us.  The sums
// run in the order of the launches it replaces.  Tables per dimension: ptap[5 mc],
// sub[mc], cp[mc], inv[mc], etap[3 m], efirst[m].
__host__ __device__ inline int adjoint_tab_elems(int m, int mc) { return 4 * m + 8 * mc; }
template <typename T>
struct AdjointSizes {
    long long nl, nc, ra, rb, tab;   // level grid, coarse grid, the two scratch arrays, tables of levels 1..l
};
template <typename T>
__host__ __device__ inline AdjointSizes<T> adjoint_sizes(const LevelGeom<T> *g, int ls)
{
    AdjointSizes<T> z;
    long long r2, r1;
    coarse_sizes<T>(g[ls], z.nl, z.nc, r2, r1);
    const long long t2 = (long long)g[ls].dim[0].mc * g[ls].dim[1].m * g[ls].dim[2].m;
    const long long t1 = (long long)g[ls].dim[0].mc * g[ls].dim[1].mc * g[ls].dim[2].m;
    z.ra = r2 > t2 ? r2 : t2;
    z.rb = r1 > t1 ? r1 : t1;
    z.tab = 0;
    for (int l = 1; l <= ls; l++)
        for (int k = 0; k < 3; k++) z.tab += adjoint_tab_elems(g[l].dim[k].m, g[l].dim[k].mc);
    return z;
}

// out = (M_l P) in along dimension k; out has extents n0 x n1 x n2 (extent k =
// m), in the same with extent k = mc; fin(idx, v) takes the products
template <typename T, int k, typename Fin>
__device__ __forceinline__ void coarse_prolong(const T *etap, const int *efirst, int mc, int n0, int n1, int n2,
                                               unsigned mul2, unsigned mul1, const T *in, Fin fin)
{
    const int i1 = k == 1 ? mc : n1, i2 = k == 2 ? mc : n2;
    const int is = k == 0 ? i1 * i2 : k == 1 ? i2 : 1;
    for (int idx = threadIdx.x; idx < n0 * n1 * n2; idx += blockDim.x) {
        const int r = small_div(idx, mul2), p2 = idx - r * n2, p0 = small_div(r, mul1), p1 = r - p0 * n1;
        const int p = k == 0 ? p0 : k == 1 ? p1 : p2;
        const int f = efirst[p];
        const T *x = in + ((k == 0 ? f : p0) * i1 + (k == 1 ? f : p1)) * i2 + (k == 2 ? f : p2);
        T v = (T)0;
#pragma unroll
        for (int i = 0; i < 3; i++)
            if (f + i < mc) v = fma_rn(etap[p * 3 + i], x[i * is], v);
        fin(idx, p0, p1, p2, v);
    }
}

template <typename T>
__global__ void __launch_bounds__(kCoarseThreads, 1) coarse_adjoint_kernel(AdjointArgs<T> a)
{
    extern __shared__ __align__(16) unsigned char coarse_smem[];
    __shared__ CoarseExt sext[kCoarseMaxLevels + 1][3];
    const int ls = a.ls, tid = threadIdx.x, nt = blockDim.x;
    const AdjointSizes<T> z = adjoint_sizes<T>(a.g, ls);
    const int nl = (int)z.nl, nc = (int)z.nc;
    T *VA = reinterpret_cast<T *>(coarse_smem);   // [nl] the level's gradient, by turns
    T *VB = VA + nl;                                // [nc]
    T *Y = VB + nc;                                 // [nc]
    T *RA = Y + nc;                                 // [ra]
    T *RB = RA + z.ra;                              // [rb]
    T *tab = RB + z.rb;
    next_begin();
    // extents and offsets of every dimension (thread 0: a few dozen), then the tables
    if (tid == 0) {
        int off = 0;
        for (int l = 1; l <= ls; l++)
            for (int k = 0; k < 3; k++) {
                const int m = a.g[l].dim[k].m, mc = a.g[l].dim[k].mc;
                sext[l][k] = {m, mc, off, small_div_mul(m), small_div_mul(mc)};
                off += adjoint_tab_elems(m, mc);
            }
    }
    for (int i = tid; i < nl; i += nt) cp_async_elem(VA + i, a.g_in + i);
    __syncthreads();
    for (int task = tid >> 5; task < 18 * ls; task += nt >> 5) {
        const int l = 1 + task / 18, r = task - (l - 1) * 18, k = r / 6, w = r - k * 6;
        const DimTables<T> &g = a.g[l].dim[k];
        const CoarseExt &e = sext[l][k];
        T *t = tab + e.off;
        if (w == 5) {
            int *d = reinterpret_cast<int *>(t + 8 * e.mc + 3 * e.m);
            for (int i = tid & 31; i < e.m; i += 32) d[i] = g.efirst[i];
            continue;
        }
        const T *src = w == 0 ? g.ptap : w == 1 ? g.sub : w == 2 ? g.cp : w == 3 ? g.inv_den : g.etap;
        const int cnt = w == 0 ? 5 * e.mc : w < 4 ? e.mc : 3 * e.m;
        T *dst = t + (w == 0 ? 0 : w < 4 ? (4 + w) * e.mc : 8 * e.mc);
        for (int i = tid & 31; i < cnt; i += 32) cp_async_elem(dst + i, src + i);
    }
    cp_async_wait_all();
    __syncthreads();
    T *G = VA, *GC = VB;
    for (int l = ls; l >= 1; l--) {
        CoarseDim<T> d[3];
        const T *etap[3];
        const int *efirst[3];
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const CoarseExt &e = sext[l][k];
            const T *t = tab + e.off;
            d[k].m = e.m; d[k].mc = e.mc; d[k].mmul = e.mmul; d[k].cmul = e.cmul;
            d[k].wl = d[k].wr = nullptr;
            d[k].tap = t; d[k].sub = t + 5 * e.mc; d[k].cp = t + 6 * e.mc; d[k].inv = t + 7 * e.mc;
            etap[k] = t + 8 * e.mc;
            efirst[k] = reinterpret_cast<const int *>(t + 8 * e.mc + 3 * e.m);
        }
        const int m0 = d[0].m, m1 = d[1].m, m2 = d[2].m, c0 = d[0].mc, c1 = d[1].mc, c2 = d[2].mc;
        // g_{l-1} = P^T g_l
        coarse_restrict<T, 2>(d[2], m0, m1, m2, d[2].cmul, d[1].mmul, G, RA);
        coarse_restrict<T, 1>(d[1], m0, m1, c2, d[2].cmul, d[1].cmul, RA, RB);
        coarse_restrict<T, 0>(d[0], m0, c1, c2, d[2].cmul, d[1].cmul, RB, GC);
        // y
        for (int i = tid; i < c0 * c1 * c2; i += nt) Y[i] = GC[i];
        __syncthreads();
        if (m0 > 1) {
            const int pl = c1 * c2;
            for (int i = tid; i < pl; i += nt) {
                T *p = Y + i;
                sweep_line<T>(p, pl, c0, d[0].sub, d[0].cp, d[0].inv, [&](int t, const auto &v) {
#pragma unroll
                    for (int u = 0; u < (int)(sizeof(v) / sizeof(T)); u++) p[(t - u) * pl] = v[u];
                });
            }
            __syncthreads();
        }
        if (m1 > 1) {
            for (int i = tid; i < c0 * c2; i += nt) {
                const int j0 = small_div(i, d[2].cmul);
                T *p = Y + j0 * c1 * c2 + (i - j0 * c2);
                sweep_line<T>(p, c2, c1, d[1].sub, d[1].cp, d[1].inv, [&](int t, const auto &v) {
#pragma unroll
                    for (int u = 0; u < (int)(sizeof(v) / sizeof(T)); u++) p[(t - u) * c2] = v[u];
                });
            }
            __syncthreads();
        }
        for (int i = tid; i < c0 * c1; i += nt) {
            T *p = Y + i * c2;
            sweep_line<T>(p, 1, c2, d[2].sub, d[2].cp, d[2].inv, [&](int t, const auto &v) {
#pragma unroll
                for (int u = 0; u < (int)(sizeof(v) / sizeof(T)); u++) p[t - u] = v[u];
            });
        }
        __syncthreads();
        // the prolonged correction, taken from g_l at the new nodes
        coarse_prolong<T, 2>(etap[2], efirst[2], c2, c0, c1, m2, d[2].mmul, d[1].cmul, Y,
                             [&](int i, int, int, int, T v) { RB[i] = v; });
        __syncthreads();
        coarse_prolong<T, 1>(etap[1], efirst[1], c1, c0, m1, m2, d[2].mmul, d[1].mmul, RB,
                             [&](int i, int, int, int, T v) { RA[i] = v; });
        __syncthreads();
        const long long np = a.g[l].Nprev;
        coarse_prolong<T, 0>(etap[0], efirst[0], c0, m0, m1, m2, d[2].mmul, d[1].mmul, RA,
                             [&](int i, int p0, int p1, int p2, T v) {
                                 const bool k0 = kept_pos(m0, p0), k1 = kept_pos(m1, p1);
                                 if (k0 && k1 && kept_pos(m2, p2)) return;
                                 int cr = kept_before(p0) * c1 * c2;
                                 if (k0) cr += kept_before(p1) * c2 + (k1 ? kept_before(p2) : 0);
                                 a.coef_out[np + i - cr] = sub_rn(G[i], v);
                             });
        __syncthreads();
        T *t = G; G = GC; GC = t;
    }
    for (int i = tid; i < (int)a.N0; i += nt) a.coef_out[i] = G[i];
}

}  // namespace

int norm_parts() { return kNormBlocks; }

// Coarse planes per CTA (segment) for a grid of `tiles` x segments CTAs:
// fill whole waves of the resident CTAs (per_sm per SM) while keeping the
// dim-0 halo (two fine planes each side of a segment) small.
int choose_segment(int mc0, long long tiles, int per_sm)
{
    const int nsm = sm_count();
    const long long slots = (long long)nsm * std::max(1, per_sm);
    double best = -1.0;
    int best_seg = mc0;
    for (int gz = 1; gz <= mc0 && gz <= 512; gz++) {
        const int seg = (mc0 + gz - 1) / gz;
        const long long ctas = tiles * ((mc0 + seg - 1) / seg);
        const long long waves = (ctas + slots - 1) / slots;
        const double score = (double)ctas / (double)(waves * slots) * (2.0 * seg) / (2.0 * seg + 4.0);
        if (score > best + 1e-9) { best = score; best_seg = seg; }
    }
    return best_seg;
}


template <typename T>
cudaError_t launch_restrict(WSrc src, Sink sink, const RestrictArgs<T> &a, cudaStream_t s)
{
    // the field source (compression, decomposition) and the decompression-side
    // sources (symbols, a coefficient stream, a dense level grid) run in the
    // warp-specialised plane pipelines of decomp.cu
    if (src == WSrc::FIELD) return launch_decomp<T>(sink, a, s);
    return launch_restrict_planes<T>(src, a, s);
}

template <typename T>
cudaError_t launch_solves(const LevelGeom<T> &g, T *b, T *vc, int sign, cudaStream_t s, const T *src)
{
    if (!src) src = b;   // the first solve reads src, the others b
    const long long c0 = g.dim[0].mc, c1 = g.dim[1].mc, c2 = g.dim[2].mc;
    int last = -1;
    for (int k = 0; k < 3; k++) if (g.dim[k].mc > 1 && g.dim[k].m > 1) last = k;
    for (int k = 0; k < 3; k++) {
        const DimTables<T> &d = g.dim[k];
        if (!(d.m > 1)) continue;
        int sg = (k == last) ? sign : 0;
        cudaError_t e;
        // the streaming sweep keeps the three factor tables in shared memory
        // (at most the default 48 KB); longer lines take the strided kernel
        if (k < 2 && sg == 0 && 3 * (size_t)d.mc * sizeof(T) <= 48 * 1024) {
            // dim 0: lines (j1, j2), step c1*c2; dim 1: lines (j0, j2), step c2
            const long long st = (k == 0) ? c1 * c2 : c2;
            const long long outer = (k == 0) ? c1 : c0;
            const long long ostride = (k == 0) ? c2 : c1 * c2;
            const long long nlines = outer * c2;
            e = launch_next(solve_stream_kernel<T>, (unsigned)((nlines + kSolveThreads - 1) / kSolveThreads), kSolveThreads,
                            3 * (size_t)d.mc * sizeof(T), s, b, src, d.mc, st, ostride, c2, nlines, d.sub, d.cp, d.inv_den);
        } else if (k < 2) {
            long long stride = (k == 0) ? c1 * c2 : c2;
            long long nlines = (k == 0) ? c1 * c2 : c0 * c2;
            int n = d.mc;
            e = launch_next(solve_strided_kernel<T>, (unsigned)((nlines + 255) / 256), 256, 0, s, b, src, n, stride, nlines,
                            d.sub, d.cp, d.inv_den, vc, sg);
        } else {
            int n = d.mc;
            long long nlines = c0 * c1;
            // a tile of lines and the three factor tables in 100 KB, two or three CTAs per
            // SM; lines of which fewer than eight fit that take the SM's shared memory
            // where it holds more of them
            constexpr int V = 16 / sizeof(T);
            const bool pad = n % kContigPad == 0 && !(((uintptr_t)b | (uintptr_t)src | (uintptr_t)vc) & 15);
            const size_t line = (size_t)(pad ? n + V : n) * sizeof(T), fixed = 3 * (size_t)n * sizeof(T) + 96;
            const auto lines_in = [&](size_t kb) {
                return kb * 1024 > fixed ? std::min<size_t>(kContigRows, (kb * 1024 - fixed) / line) : 0;
            };
            size_t rows = lines_in(100);
            if (rows < 8 && lines_in(kContigMaxKb) > 2 * rows) rows = lines_in(kContigMaxKb);
            // One or two lines an SM pay a sweep's latency alone (55 ns a step in binary64, 11
            // in binary32) once per wave; the strided kernel has every line in flight at about
            // a microsecond a step (9000x9501 binary64: 20.6 ms with tiles of two, 16.7
            // with the strided kernel on its finest level; 2000x9501 4.6 with tiles).
            if (rows <= 2 && nlines > (sizeof(T) == 8 ? 8 : 40) * (long long)rows * sm_count()) rows = 0;
            if (rows < 1) {
                e = launch_next(solve_strided_kernel<T>, (unsigned)((nlines + 255) / 256), 256, 0, s, b, src, n, 1, nlines,
                                d.sub, d.cp, d.inv_den, vc, sg);
            } else {
                static PerDeviceOnce attr;
                cudaError_t ea = once_per_device(attr, [] {
                    return cudaFuncSetAttribute(solve_contig_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                (int)(kContigMaxKb * 1024));
                });
                if (ea != cudaSuccess) return ea;
                e = launch_next(solve_contig_kernel<T>, (unsigned)((nlines + rows - 1) / rows), kContigThreads,
                                fixed + rows * line, s, b, src, n, nlines, (int)rows, pad, d.sub, d.cp, d.inv_den, vc, sg);
            }
        }
        src = b;
        count_launch();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <typename T>
cudaError_t launch_expand(WSrc src, const LevelGeom<T> &g, const T *vc, const T *coef_in,
                          const SymIn &symin, T *out, cudaStream_t s)
{
    return launch_expand_planes<T>(src, g, vc, coef_in, symin, out, s);
}

template <typename T>
cudaError_t launch_level0(Sink sink, const T *v0, long long N0, T *coef_out, const QuantOut &qo,
                          cudaStream_t s)
{
    unsigned blocks = (unsigned)((N0 + 255) / 256);
    count_launch();
    return launch_next(sink == Sink::STREAM ? level0_kernel<T, 1> : level0_kernel<T, 2>, blocks, 256, 0, s, v0, N0, coef_out,
                       qo);
}

template <typename T>
cudaError_t launch_level0_in(WSrc src, const T *coef_in, const SymIn &symin, long long N0, T *v0,
                             cudaStream_t s)
{
    unsigned blocks = (unsigned)((N0 + 255) / 256);
    count_launch();
    return launch_next(src == WSrc::STREAM ? level0_in_kernel<T, 1> : level0_in_kernel<T, 2>, blocks, 256, 0, s, coef_in, symin,
                       N0, v0);
}

template <typename T>
cudaError_t launch_norm(const T *u, long long N, double *partials, const BinArgs &ba, Scalars *sc, cudaStream_t s)
{
    // a block per 256 16-byte vectors, at most norm_parts() of them: with fewer
    // vectors than the full grid has threads the smaller grid gives every value
    // the same thread, and the blocks left out would add zeros
    const long long need = (N * (long long)sizeof(T) / 16 + 255) / 256 + 1;
    const int blocks = (((uintptr_t)u) & 15) == 0 && need < kNormBlocks ? (int)need : kNormBlocks;
    count_launch();
    return launch_next(norm_kernel<T>, blocks, 256, 0, s, u, N, partials, ba, sc);
}

template <typename T>
size_t coarse_smem_bytes(const LevelGeom<T> &g)
{
    long long nl, nc, r2, r1;
    coarse_sizes<T>(g, nl, nc, r2, r1);
    return (size_t)(2 * nl + 3 * nc + r2 + r1) * sizeof(T);
}

template <typename T>
int coarse_top(const Plan *P, const LevelGeom<T> *geo)
{
    int ls = 0;
    for (int l = 1; l <= P->L && l <= kCoarseMaxLevels; l++)
        if (coarse_smem_bytes<T>(geo[l]) <= kCoarseSmem) ls = l;
        else break;
    return ls;
}

template <typename T>
CoarseArgs<T> coarse_args(int mode, const Plan *P, const LevelGeom<T> *geo, int ls, const T *v_in, T *v_out,
                          const QuantOut &qo, T *coef_out, const SymIn &symin, const T *coef_in, size_t *smem)
{
    CoarseArgs<T> a;
    memset(&a, 0, sizeof(a));
    for (int l = 1; l <= ls && l <= kCoarseMaxLevels; l++) a.g[l] = geo[l];
    a.ls = ls;
    a.N0 = P->N[0];
    a.v_in = v_in; a.v_out = v_out; a.qo = qo; a.coef_out = coef_out; a.symin = symin; a.coef_in = coef_in;
    a.stream_off = -1;
    size_t bytes = 0;
    if (ls >= 1 && ls <= kCoarseMaxLevels) {
        // the stream prefix, then the tables of every level and dimension, as far
        // as the block's shared memory takes them (long thin grids read theirs in
        // global memory)
        const size_t work = coarse_smem_bytes<T>(geo[ls]);
        const size_t room = work < kCoarseSmemMax ? (kCoarseSmemMax - work) / sizeof(T) : 0;
        const size_t nl = (size_t)geo[ls].dim[0].m * geo[ls].dim[1].m * geo[ls].dim[2].m;
        size_t n = 0, tab = 0;
        for (int l = 1; l <= ls; l++)
            for (int k = 0; k < 3; k++)
                if (geo[l].dim[k].m > 1) tab += coarse_tab_elems(geo[l].dim[k].m, geo[l].dim[k].mc);
        a.staged = tab <= room;
        if (a.staged)
            for (int l = 1; l <= ls; l++)
                for (int k = 0; k < 3; k++) {
                    a.tab_off[l][k] = (int)n;
                    if (geo[l].dim[k].m > 1) n += coarse_tab_elems(geo[l].dim[k].m, geo[l].dim[k].mc);
                }
        if (mode >= 2 && n + nl <= room) { a.stream_off = (int)n; n += nl; }
        bytes = work + n * sizeof(T);
    }
    if (smem) *smem = bytes;
    return a;
}

template <typename T>
cudaError_t launch_coarse_batch(const CoarseArgs<T> *jobs, int n, size_t smem, cudaStream_t s)
{
    if (n < 1) return cudaSuccess;
    static PerDeviceOnce attr;
    cudaError_t e = once_per_device(attr, [] {
        return cudaFuncSetAttribute(coarse_batch_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)kCoarseSmemMax);
    });
    if (e != cudaSuccess) return e;
    coarse_batch_kernel<T><<<n, kCoarseThreads, smem, s>>>(jobs);
    count_launch();
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_coarse(int mode, const Plan *P, const LevelGeom<T> *geo, int ls, const T *v_in, T *v_out,
                          const QuantOut &qo, T *coef_out, const SymIn &symin, const T *coef_in, cudaStream_t s)
{
    if (ls < 1 || ls > kCoarseMaxLevels) return cudaErrorInvalidValue;
    size_t sm = 0;
    const CoarseArgs<T> a = coarse_args<T>(mode, P, geo, ls, v_in, v_out, qo, coef_out, symin, coef_in, &sm);
    static PerDeviceOnce attr[4];
    auto go = [&](auto kern) -> cudaError_t {
        cudaError_t e = once_per_device(attr[mode], [&] {
            return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCoarseSmemMax);
        });
        if (e != cudaSuccess) return e;
        count_launch();
        return launch_next(kern, 1, kCoarseThreads, sm, s, a);
    };
    switch (mode) {
    case 0: return go(coarse_kernel<T, 0>);
    case 1: return go(coarse_kernel<T, 1>);
    case 2: return go(coarse_kernel<T, 2>);
    default: return go(coarse_kernel<T, 3>);
    }
}

template <typename T>
int coarse_adjoint_top(const Plan &P, const LevelGeom<T> *geo)
{
    int ls = 0;
    for (int l = 1; l <= P.L && l <= kCoarseMaxLevels; l++) {
        const AdjointSizes<T> z = adjoint_sizes<T>(geo, l);
        // small_div takes indices below 2^16
        if (z.nl >= 65536 || (size_t)(z.nl + 2 * z.nc + z.ra + z.rb + z.tab) * sizeof(T) > kCoarseSmemMax) break;
        ls = l;
    }
    return ls;
}

template <typename T>
cudaError_t launch_coarse_adjoint(const Plan &P, const LevelGeom<T> *geo, int ls, const T *g_in, T *coef_out,
                                  cudaStream_t s)
{
    if (ls < 1 || ls > kCoarseMaxLevels) return cudaErrorInvalidValue;
    AdjointArgs<T> a;
    memset(&a, 0, sizeof(a));
    for (int l = 1; l <= ls; l++) a.g[l] = geo[l];
    a.ls = ls;
    a.N0 = P.N[0];
    a.g_in = g_in;
    a.coef_out = coef_out;
    const AdjointSizes<T> z = adjoint_sizes<T>(geo, ls);
    static PerDeviceOnce attr;
    cudaError_t e = once_per_device(attr, [] {
        return cudaFuncSetAttribute(coarse_adjoint_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)kCoarseSmemMax);
    });
    if (e != cudaSuccess) return e;
    count_launch();
    return launch_next(coarse_adjoint_kernel<T>, 1, kCoarseThreads,
                       (size_t)(z.nl + 2 * z.nc + z.ra + z.rb + z.tab) * sizeof(T), s, a);
}

#define INST(T)                                                                                   \
    template cudaError_t launch_restrict<T>(WSrc, Sink, const RestrictArgs<T> &, cudaStream_t);  \
    template cudaError_t launch_solves<T>(const LevelGeom<T> &, T *, T *, int, cudaStream_t, const T *); \
    template cudaError_t launch_expand<T>(WSrc, const LevelGeom<T> &, const T *, const T *,       \
                                          const SymIn &, T *, cudaStream_t);                     \
    template cudaError_t launch_level0<T>(Sink, const T *, long long, T *, const QuantOut &,      \
                                          cudaStream_t);                                         \
    template cudaError_t launch_level0_in<T>(WSrc, const T *, const SymIn &, long long, T *,      \
                                             cudaStream_t);                                      \
    template cudaError_t launch_norm<T>(const T *, long long, double *, const BinArgs &, Scalars *, cudaStream_t); \
    template int coarse_top<T>(const Plan *, const LevelGeom<T> *);                              \
    template cudaError_t launch_coarse<T>(int, const Plan *, const LevelGeom<T> *, int, const T *, T *, \
                                          const QuantOut &, T *, const SymIn &, const T *, cudaStream_t); \
    template CoarseArgs<T> coarse_args<T>(int, const Plan *, const LevelGeom<T> *, int, const T *, T *,         \
                                          const QuantOut &, T *, const SymIn &, const T *, size_t *);      \
    template int coarse_adjoint_top<T>(const Plan &, const LevelGeom<T> *);                      \
    template cudaError_t launch_coarse_adjoint<T>(const Plan &, const LevelGeom<T> *, int, const T *, T *, cudaStream_t); \
    template cudaError_t launch_coarse_batch<T>(const CoarseArgs<T> *, int, size_t, cudaStream_t);
INST(float)
INST(double)

}  // namespace hpdr
