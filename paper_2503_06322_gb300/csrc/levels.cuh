// levels.cuh -- launchers of the per-level kernels (levels.cu).
#pragma once
#include "internal.cuh"

namespace hpdr {

// Where a restriction reads its fine-level values w from.
enum class WSrc : int {
    FIELD = 0,     // w = new-node coefficients computed from a level-l field (Alg. 1 lerp)
    STREAM = 1,    // w = coefficients read from a level-major stream (type T)
    SYMBOLS = 2,   // w = dequantized symbols of a level-major stream
    DENSE = 3,     // w = a dense level-l array (all nodes; used by the transposes)
};
// What the FIELD source does with the coefficients it computes.
enum class Sink : int { NONE = 0, STREAM = 1, QUANT = 2 };

struct QuantOut {
    uint16_t *sym;                 // stream of symbols
    unsigned long long *hist;      // global histogram [D]
    long long *esc;                // [N] code k at every escaped stream position (symbol 0)
    unsigned int D;
    Scalars *sc;
};

struct SymIn {
    const uint16_t *sym;
    unsigned int D;
    const Scalars *sc;               // q per level
    const long long *esc;            // [N] code k at every escaped stream position
    unsigned int *status;
    const double *deq;               // binary64: value of every symbol on every level, [L + 1][D], or null
};
// The expansion of binary64 fields dequantizes symbols through a table per
// level for alphabets whose table leaves two blocks an SM
constexpr unsigned kDeqMaxD = 8192;

template <typename T>
struct RestrictArgs {
    LevelGeom<T> g;
    const T *v;          // FIELD / DENSE: level-l array
    const T *coef_in;    // STREAM source
    SymIn symin;         // SYMBOLS source
    T *coef_out;         // Sink::STREAM
    QuantOut qo;         // Sink::QUANT
    T *b;                // coarse output (level l-1 grid)
    T *vc;               // coarse copy of v (FIELD with a sink), may be null
    int use_ptap;        // 0: P^T M_l taps, 1: P^T taps
    int dense_new_only;  // DENSE: 1 = use only the new nodes (E_new^T of the input)
    const void *src_end; // one past the last byte of the staged source (FIELD: v, SYMBOLS: sym)
    unsigned int *status;  // device status word (timeouts)
    int wait_limit;      // polls of a pipeline wait before it gives up (0: use the library's limit)
};

template <typename T>
cudaError_t launch_restrict(WSrc src, Sink sink, const RestrictArgs<T> &a, cudaStream_t s);

// decomp.cu: the level kernel of decomposition and compression (FIELD
// source; Sink::QUANT or Sink::STREAM) and the restriction of decompression
// (SYMBOLS source), warp-specialised plane pipelines.
template <typename T>
cudaError_t launch_decomp(Sink sink, const RestrictArgs<T> &a, cudaStream_t s);
// the plane pipeline over any decompression-side source: SYMBOLS,
// STREAM (a coefficient stream) or DENSE (a level-l grid, all or new nodes)
template <typename T>
cudaError_t launch_restrict_planes(WSrc src, const RestrictArgs<T> &a, cudaStream_t s);
template <typename T>
cudaError_t launch_expand_planes(WSrc src, const LevelGeom<T> &g, const T *vc, const T *coef_in,
                                 const SymIn &symin, T *out, cudaStream_t s);

// Polls of a bounded pipeline wait before the kernel gives up with
// DS_TIMEOUT (set through hpdr_debug_set_wait_limit; default kWaitPolls).
// The drain of copies in flight after a give-up always uses kWaitPolls.
extern int g_wait_limit;

// Solve (x)_k M_{l-1} along every active dimension of the coarse array b, in
// place; the last solve optionally adds (sign=+1) or subtracts (sign=-1) the
// result into vc instead of storing it into b.  src non-null: the right-hand
// side is read there and left as it is (b need not be set).
template <typename T>
cudaError_t launch_solves(const LevelGeom<T> &g, T *b, T *vc, int sign, cudaStream_t s, const T *src = nullptr);

// Recomposition of level l: out (level-l grid) = kept nodes from vc (level
// l-1 grid), new nodes = coefficient + interpolant of vc.
template <typename T>
cudaError_t launch_expand(WSrc src, const LevelGeom<T> &g, const T *vc, const T *coef_in,
                          const SymIn &symin, T *out, cudaStream_t s);

// Level 0: quantize (Sink::QUANT) or copy (Sink::STREAM) the coarsest grid.
template <typename T>
cudaError_t launch_level0(Sink sink, const T *v0, long long N0, T *coef_out, const QuantOut &qo,
                          cudaStream_t s);
// Level 0 of recomposition: v0 = coefficient stream entries [0, N0).
template <typename T>
cudaError_t launch_level0_in(WSrc src, const T *coef_in, const SymIn &symin, long long N0, T *v0,
                             cudaStream_t s);

// max|u| and sum u^2 (deterministic), then the bins, in one launch; sc must be
// zero before (its blocks_done counts the blocks), partials holds 2 norm_parts().
struct BinArgs {
    int L;
    double c[kMaxLevels + 1];
    double tol;
    int tol_kind, mode;
    double eps;
    long long N;
};
template <typename T>
cudaError_t launch_norm(const T *u, long long N, double *partials, const BinArgs &ba, Scalars *sc, cudaStream_t s);

int norm_parts();

// The coarse levels in one CTA (levels.cu): levels 1..ls and level 0, with
// ls = coarse_top(), the largest level whose shared arrays fit kCoarseSmem.
// mode 0: compression (v_in -> symbols), 1: decomposition (v_in -> coef_out),
// 2: decompression (symbols -> v_out), 3: recomposition (coef_in -> v_out).
constexpr int kCoarseMaxLevels = 16;
constexpr size_t kCoarseSmem = 200 * 1024;      // working arrays (fixes ls)
constexpr size_t kCoarseSmemMax = 220 * 1024;   // with the staged tables and stream
template <typename T>
int coarse_top(const Plan *P, const LevelGeom<T> *geo);
template <typename T>
struct CoarseArgs {
    LevelGeom<T> g[kCoarseMaxLevels + 1];   // levels 1..ls
    int ls;
    long long N0;
    const T *v_in;       // compression / decomposition: the level-ls grid
    T *v_out;            // recomposition: the level-ls grid
    QuantOut qo;         // compression
    T *coef_out;         // decomposition
    SymIn symin;         // decompression
    const T *coef_in;    // recomposition
    // past the working arrays: element offsets of the staged tables (staged) and
    // of the staged stream prefix (-1: read in global memory)
    bool staged;
    int stream_off;
    int tab_off[kCoarseMaxLevels + 1][3];
};
template <typename T>
cudaError_t launch_coarse(int mode, const Plan *P, const LevelGeom<T> *geo, int ls, const T *v_in, T *v_out,
                          const QuantOut &qo, T *coef_out, const SymIn &symin, const T *coef_in, cudaStream_t s);
// the arguments of that launch (host), and its dynamic shared memory
template <typename T>
CoarseArgs<T> coarse_args(int mode, const Plan *P, const LevelGeom<T> *geo, int ls, const T *v_in, T *v_out,
                          const QuantOut &qo, T *coef_out, const SymIn &symin, const T *coef_in, size_t *smem);
// the coarse levels of n compressions in one launch (one block per field; jobs:
// device [n]; smem: the largest of the fields' shared-memory sizes)
template <typename T>
cudaError_t launch_coarse_batch(const CoarseArgs<T> *jobs, int n, size_t smem, cudaStream_t s);

// The coarse levels ls..1 and 0 of the adjoint of recomposition in one CTA: g_in
// is the gradient on the level-ls grid, coef_out the coefficient gradient's
// stream.  ls = coarse_adjoint_top(), the largest level that fits (0: none).
template <typename T>
struct AdjointArgs {
    LevelGeom<T> g[kCoarseMaxLevels + 1];
    int ls;
    long long N0;
    const T *g_in;
    T *coef_out;
};
template <typename T>
int coarse_adjoint_top(const Plan &P, const LevelGeom<T> *geo);
template <typename T>
cudaError_t launch_coarse_adjoint(const Plan &P, const LevelGeom<T> *geo, int ls, const T *g_in, T *coef_out,
                                  cudaStream_t s);

// adjoint.cu: transposes of recomposition / decomposition over all levels.
// ga, gb, y, R hold N_{L-1} elements.
template <typename T>
cudaError_t recompose_adjoint_run(const Plan &P, const LevelGeom<T> *geo, const T *gu, T *gcoef, T *ga, T *gb,
                                  T *y, unsigned *status, cudaStream_t s);
template <typename T>
cudaError_t decompose_adjoint_run(const Plan &P, const LevelGeom<T> *geo, const T *gcoef, T *gu, T *ga, T *gb,
                                  T *y, T *R, unsigned *status, cudaStream_t s);

}  // namespace hpdr
