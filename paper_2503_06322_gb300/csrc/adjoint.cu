// adjoint.cu -- transposes of recomposition and decomposition (the maps are
// linear, so backward passes need no saved forward state).
//
// One level of recomposition is  v_l = P (v_{l-1} - S c_l) + E_new c_l  with
// S = (x)M_{l-1}^{-1} (x)P^T M_l E_new; its transpose, from the level-l
// gradient g_l, is
//     g_{l-1} = P^T g_l,      g_{c_l} = g_l|new - E_new^T ((x)M_l P) (x)M_{l-1}^{-1} P^T g_l.
// One level of decomposition is  c_l = (v - P v|kept)|new,
// v_{l-1} = v|kept + S c_l; its transpose, from g_{c_l} and g_{v_{l-1}}, is
//     h = g_{c_l} + E_new^T ((x)M_l P) (x)M_{l-1}^{-1} g_{v_{l-1}},
//     g_{v_l} = E_new h + E_kept (g_{v_{l-1}} - P^T E_new h).
// P^T is the restriction kernel with the interpolation taps, M_{l-1}^{-1} the
// Thomas solves, and (x)M_l P runs in one pass over the fine grid below.
#include <cstring>
#include "internal.cuh"
#include "levels.cuh"
#include "levels_dev.cuh"

namespace hpdr {
namespace {

enum { MP_RT_FINAL = 1, MP_DT_FINAL = 2 };

// y_f = (x)_k M_l P_k y on the level-l grid, only at its new nodes:
//   MP_RT_FINAL: stream[rank(p)] = gsrc[p] - y_f(p)
//   MP_DT_FINAL: out[p] = coef[rank(p)] + y_f(p)
// One pass over the fine grid is all it needs from memory (a pass per dimension,
// through two partial grids, moved 2.6 times the bytes and took 173 us for the
// finest level of 257^3; this takes 62, bound by the latency of its sixteen cached
// loads a plane at 42% of the issue slots: 78 with the window's edges tested at every
// node).  A warp owns coarse row j1 of a tile and lane l coarse column j2 (or, on thin
// grids, four rows and eight columns), and the CTA marches along the coarse planes of
// its segment; for each plane a lane forms the dimension-2, then the dimension-1
// products at its 2 x 2 fine nodes (rows Ra, Ra + 1, columns Ca, Ca + 1) from the four
// rows and four columns of y around it (cached loads, coalesced per row) and keeps the
// last three planes' for the dimension-0 products.  Every value sums its taps in a
// fixed order, so nothing depends on the tiling.
constexpr int kMpWarps = 8;
// The tiles of a coarse plane, LC columns wide, run along gridDim.x, columns first:
// gridDim.y ends at 65535, and a tall field has more row tiles.
__host__ __device__ inline int tile_cols(int mc2, int LC) { return (mc2 + LC - 1) / LC; }
__host__ __device__ inline int tile_rows(int LC) { return kMpWarps * (32 / LC); }
__host__ __device__ inline long long plane_tiles(int mc1, int mc2, int LC)
{
    return (long long)tile_cols(mc2, LC) * ((mc1 + tile_rows(LC) - 1) / tile_rows(LC));
}
// first coarse row and column of tile b
struct PlaneTile {
    int j1, j2;
};
__host__ __device__ inline PlaneTile plane_tile(unsigned b, int mc2, int LC)
{
    const unsigned cols = (unsigned)tile_cols(mc2, LC), r = b / cols;
    return {(int)r * tile_rows(LC), (int)(b - r * cols) * LC};
}
// BIG: planes of 2^31 nodes and more, whose offsets take 64 bits.  LC: a warp takes
// 32 columns of one coarse row, or 8 of four rows, which leaves fewer lanes without a
// column on grids that are thin in the last dimension.
template <typename T, int MODE, int LC, bool BIG>
__global__ void __launch_bounds__(32 * kMpWarps)
prolong_kernel(LevelGeom<T> g, const T *y, const T *gsrc, T *__restrict__ stream, const T *coef, T *__restrict__ out,
               int seg_len)
{
    const DimTables<T> &d0 = g.dim[0], &d1 = g.dim[1], &d2 = g.dim[2];
    const int m0 = d0.m, m1 = d1.m, m2 = d2.m, mc0 = d0.mc, mc1 = d1.mc, mc2 = d2.mc;
    const int lane = threadIdx.x & 31, warp = warp_index();
    constexpr int RW = 32 / LC;   // rows of a warp
    const PlaneTile tile = plane_tile(blockIdx.x, mc2, LC);
    const int w1 = tile.j1 + warp * RW, j2 = tile.j2 + lane % LC, j1 = w1 + (RW > 1 ? lane / LC : 0);
    const int J0a = blockIdx.y * seg_len, J0b = min(J0a + seg_len, mc0);
    next_begin();
    if (J0a >= J0b || w1 >= mc1) return;
    const bool live = j2 < mc2 && (RW == 1 || j1 < mc1);
    const int Ca = cpos_of(m2, mc2, min(j2, mc2 - 1)), Ra = cpos_of(m1, mc1, RW == 1 ? j1 : min(j1, mc1 - 1));
    const bool hb = Ca + 1 < m2 && !kept_pos(m2, Ca + 1), hr = Ra + 1 < m1 && !kept_pos(m1, Ra + 1);
    // taps of the two fine columns and rows; the second ones start at the same
    // coarse index or one later
    T e2[2][3], e1[2][3];
    const int c2 = d2.efirst[Ca], c1 = d1.efirst[Ra];
    const bool s2 = hb && d2.efirst[Ca + 1] != c2, s1 = hr && d1.efirst[Ra + 1] != c1;
#pragma unroll
    for (int i = 0; i < 3; i++) {
        e2[0][i] = d2.etap[Ca * 3ll + i];
        e2[1][i] = hb ? d2.etap[(Ca + 1) * 3ll + i] : (T)0;
        e1[0][i] = d1.etap[Ra * 3ll + i];
        e1[1][i] = hr ? d1.etap[(Ra + 1) * 3ll + i] : (T)0;
    }
    const int nc2 = mc2 - c2, nc1 = mc1 - c1;   // columns and rows from the first on
    // away from the grid's edges the window is whole and the second taps start one later
    const bool inner = __all_sync(0xffffffffu, s2 && s1 && nc2 >= 4 && nc1 >= 4);
    if (!live) return;
    const long long cplane = (long long)mc1 * mc2;
    // offsets inside a coarse plane, a fine plane, and a kept plane of the stream
    using Off = typename std::conditional<BIG, unsigned long long, unsigned>::type;
    const PlaneRows<Off> rows = plane_rows<Off>(m2, mc2, Ra);
    const Off oy = (Off)c1 * mc2 + c2;
    const Off ox0 = rows.x[0] + Ca, ox1 = rows.x[1] + Ca, ok0 = rows.k[0] + (Ca >> 1), ok1 = rows.k[1] + Ca;
    struct D4 { T v[2][2]; };
    // dimension-2 and -1 products of coarse plane j at the lane's nodes
    auto plane = [&](int j) -> D4 {
        const T *p = y + j * cplane;
        T r2[4][2];   // rows c1.., the two columns
        D4 d;
        if (inner) {
#pragma unroll
            for (int r = 0; r < 4; r++) {
                const T *q = p + (oy + (Off)r * mc2);
                const T x0 = q[0], x1 = q[1], x2 = q[2], x3 = q[3];
                r2[r][0] = fma_rn(e2[0][2], x2, fma_rn(e2[0][1], x1, fma_rn(e2[0][0], x0, (T)0)));
                r2[r][1] = fma_rn(e2[1][2], x3, fma_rn(e2[1][1], x2, fma_rn(e2[1][0], x1, (T)0)));
            }
#pragma unroll
            for (int c = 0; c < 2; c++) {
                d.v[0][c] = fma_rn(e1[0][2], r2[2][c], fma_rn(e1[0][1], r2[1][c], fma_rn(e1[0][0], r2[0][c], (T)0)));
                d.v[1][c] = fma_rn(e1[1][2], r2[3][c], fma_rn(e1[1][1], r2[2][c], fma_rn(e1[1][0], r2[1][c], (T)0)));
            }
            return d;
        }
#pragma unroll
        for (int r = 0; r < 4; r++) {
            T x[4];
            const T *q = p + (oy + (Off)r * mc2);
#pragma unroll
            for (int c = 0; c < 4; c++) x[c] = r < nc1 && c < nc2 ? q[c] : (T)0;
            T a = (T)0, b = (T)0;
#pragma unroll
            for (int i = 0; i < 3; i++) {
                if (i < nc2) a = fma_rn(e2[0][i], x[i], a);
                if (i + (s2 ? 1 : 0) < nc2) b = fma_rn(e2[1][i], s2 ? x[i + 1] : x[i], b);
            }
            r2[r][0] = a;
            r2[r][1] = b;
        }
#pragma unroll
        for (int c = 0; c < 2; c++) {
            T a = (T)0, b = (T)0;
#pragma unroll
            for (int i = 0; i < 3; i++) {
                if (i < nc1) a = fma_rn(e1[0][i], r2[i][c], a);
                if (i + (s1 ? 1 : 0) < nc1) b = fma_rn(e1[1][i], s1 ? r2[i + 1][c] : r2[i][c], b);
            }
            d.v[0][c] = a;
            d.v[1][c] = b;
        }
        return d;
    };
    // fine plane P from the products A, B, C of coarse planes j - 1, j, j + 1: its
    // three taps start at plane j - 1, or one later (the start of the grid, a new
    // plane) or earlier (its end), where the tap that falls outside is zero
    D4 A, B, C;
    auto emit = [&](int P, int j) {
        const bool k0 = kept_pos(m0, P);
        const int o = d0.efirst[P] - (j - 1);
        const T *e = d0.etap + P * 3ll;
        const T tA = o == 0 ? e[0] : o < 0 ? e[1] : (T)0, tB = o == 0 ? e[1] : o < 0 ? e[2] : e[0];
        const T tC = o == 0 ? e[2] : o < 0 ? (T)0 : e[1];
        const bool useA = j > 0 && o <= 0, useC = j + 1 < mc0 && o >= 0;
        const long long fp = (long long)P * m1 * m2, sp = plane_base_of(g, P);
#pragma unroll
        for (int r = 0; r < 2; r++) {
            if (r && !hr) continue;
            const bool rownew = !k0 || r;
            const Off f = r ? ox1 : ox0, k = k0 ? (r ? ok1 : ok0) : f;   // of column Ca, or the row's first new one
            const T *gp = MODE == MP_RT_FINAL ? gsrc + fp + f : coef + sp + k;
            T *op = MODE == MP_RT_FINAL ? stream + sp + k : out + fp + f;
#pragma unroll
            for (int c = 0; c < 2; c++) {
                if ((c && !hb) || (!rownew && !c)) continue;
                T v = (T)0;
                if (useA) v = fma_rn(tA, A.v[r][c], v);
                v = fma_rn(tB, B.v[r][c], v);
                if (useC) v = fma_rn(tC, C.v[r][c], v);
                const int ks = rownew ? c : 0;   // the stream's step to column Ca + c
                if (MODE == MP_RT_FINAL) op[ks] = sub_rn(gp[c], v);
                else op[c] = add_rn(gp[ks], v);
            }
        }
    };
    A = plane(J0a > 0 ? J0a - 1 : 0);
    B = J0a > 0 ? plane(J0a) : A;
    for (int j = J0a; j < J0b; j++) {
        if (j + 1 < mc0) C = plane(j + 1);
        const int P = cpos_of(m0, mc0, j);
        emit(P, j);
        // the new plane between j and j + 1
        if (P + 1 < m0 && !kept_pos(m0, P + 1)) emit(P + 1, j);
        A = B;
        B = C;
    }
}

// decompose transpose: G(kept node of coarse q) = gv[q] - R[q]
template <typename T>
__global__ void set_kept_kernel(T *G, const T *gv, const T *R, LevelGeom<T> g)
{
    next_begin();
    const long long c1 = g.dim[1].mc, c2 = g.dim[2].mc;
    const long long n = (long long)g.dim[0].mc * c1 * c2;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        long long q0, q1, q2;
        if (n < (1LL << 31)) {   // 32-bit divisions
            const unsigned u = (unsigned)q, t = u / (unsigned)c2;
            q2 = u - t * (unsigned)c2;
            q0 = t / (unsigned)c1;
            q1 = t - (unsigned)q0 * (unsigned)c1;
        } else {
            const long long t = q / c2;
            q2 = q - t * c2;
            q1 = t % c1;
            q0 = t / c1;
        }
        const long long p0 = cpos_of(g.dim[0].m, g.dim[0].mc, (int)q0);
        const long long p1 = cpos_of(g.dim[1].m, g.dim[1].mc, (int)q1);
        const long long p2 = cpos_of(g.dim[2].m, g.dim[2].mc, (int)q2);
        G[(p0 * g.dim[1].m + p1) * g.dim[2].m + p2] = sub_rn(gv[q], R[q]);
    }
}

template <typename T>
__global__ void copy_kernel(T *dst, const T *src, long long n)
{
    next_begin();
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = src[i];
}

unsigned grid_for(long long n) { return (unsigned)std::min<long long>((n + 255) / 256, 152LL * 16); }

template <typename T, int MODE>
cudaError_t launch_prolong(const LevelGeom<T> &g, const T *y, T *out, const T *gsrc, T *stream, const T *coef,
                           cudaStream_t s)
{
    const int mc0 = g.dim[0].mc, mc1 = g.dim[1].mc, mc2 = g.dim[2].mc;
    // Eight columns below 64 and where tiles of 32 have over a quarter more lanes
    // (recomposition's adjoint, binary64, 32 or 8 columns: 1000x1000x15 2668 or 1639 us,
    // x63 2840 or 2738, x65 4318 or 3610, x80 4540 or 4185; 200x200x127 460 or 477,
    // 100x200x400 635 or 644).
    const bool big = big_planes(g), thin = !big && (mc2 < 64 || 4 * 32 * tile_cols(mc2, 32) > 5 * 8 * tile_cols(mc2, 8));
    const auto kern = big ? prolong_kernel<T, MODE, 32, true>
                    : thin ? prolong_kernel<T, MODE, 8, false> : prolong_kernel<T, MODE, 32, false>;
    const long long tiles = plane_tiles(mc1, mc2, thin ? 8 : 32);
    const int seg = choose_segment(mc0, tiles, resident_ctas(kern, 32 * kMpWarps, 0));
    count_launch();
    return launch_next(kern, dim3((unsigned)tiles, (mc0 + seg - 1) / seg), 32 * kMpWarps, 0, s, g, y, gsrc, stream, coef, out,
                       seg);
}

}  // namespace

template <typename T>
cudaError_t recompose_adjoint_run(const Plan &P, const LevelGeom<T> *geo, const T *gu, T *gcoef, T *ga, T *gb,
                                  T *y, unsigned *status, cudaStream_t s)
{
    const int L = P.L;
    const T *gl = gu;
    const int ls = coarse_adjoint_top<T>(P, geo);
    for (int l = L; l > ls; l--) {
        const LevelGeom<T> &g = geo[l];
        T *gc = ((L - l) % 2 == 0) ? ga : gb;   // g_{l-1} = P^T g_l
        RestrictArgs<T> a;
        memset(&a, 0, sizeof(a));
        a.g = g;
        a.v = gl;
        a.use_ptap = 1;
        a.dense_new_only = 0;
        a.b = gc;
        a.status = status;
        cudaError_t e = launch_restrict<T>(WSrc::DENSE, Sink::NONE, a, s);
        if (e != cudaSuccess) return e;
        e = launch_solves<T>(g, y, nullptr, 0, s, gc);
        if (e != cudaSuccess) return e;
        e = launch_prolong<T, MP_RT_FINAL>(g, y, nullptr, gl, gcoef, nullptr, s);
        if (e != cudaSuccess) return e;
        gl = gc;
    }
    if (ls >= 1) return launch_coarse_adjoint<T>(P, geo, ls, gl, gcoef, s);
    count_launch();
    return launch_next(copy_kernel<T>, grid_for(P.N[0]), 256, 0, s, gcoef, gl, P.N[0]);
}

template <typename T>
cudaError_t decompose_adjoint_run(const Plan &P, const LevelGeom<T> *geo, const T *gcoef, T *gu, T *ga, T *gb,
                                  T *y, T *R, unsigned *status, cudaStream_t s)
{
    const int L = P.L;
    T *gv = (L == 0) ? gu : ((L % 2 == 1) ? ga : gb);
    count_launch();
    cudaError_t e = launch_next(copy_kernel<T>, grid_for(P.N[0]), 256, 0, s, gv, gcoef, P.N[0]);
    if (e != cudaSuccess) return e;
    for (int l = 1; l <= L; l++) {
        const LevelGeom<T> &g = geo[l];
        T *G = (l == L) ? gu : (((L - l) % 2 == 1) ? ga : gb);
        const long long nc = P.N[l - 1];
        e = launch_solves<T>(g, y, nullptr, 0, s, gv);
        if (e != cudaSuccess) return e;
        // new nodes: G = h = g_c + ((x)M_l P) y
        e = launch_prolong<T, MP_DT_FINAL>(g, y, G, nullptr, nullptr, gcoef, s);
        if (e != cudaSuccess) return e;
        // kept nodes: G = gv - P^T E_new h
        RestrictArgs<T> a;
        memset(&a, 0, sizeof(a));
        a.g = g;
        a.v = G;
        a.use_ptap = 1;
        a.dense_new_only = 1;
        a.b = R;
        a.status = status;
        e = launch_restrict<T>(WSrc::DENSE, Sink::NONE, a, s);
        if (e != cudaSuccess) return e;
        count_launch();
        e = launch_next(set_kept_kernel<T>, grid_for(nc), 256, 0, s, G, gv, R, g);
        if (e != cudaSuccess) return e;
        gv = G;
    }
    return cudaGetLastError();
}

#define INST(T)                                                                                                    \
    template cudaError_t recompose_adjoint_run<T>(const Plan &, const LevelGeom<T> *, const T *, T *, T *, T *, T *, \
                                                  unsigned *, cudaStream_t);                                       \
    template cudaError_t decompose_adjoint_run<T>(const Plan &, const LevelGeom<T> *, const T *, T *, T *, T *, T *, \
                                                  T *, unsigned *, cudaStream_t);
INST(float)
INST(double)

}  // namespace hpdr
