// api.cu -- extern "C" entry points declared in include/hpdr.h.
//
// compress  = norm pre-pass -> bins -> for l = L..1 { fused coefficients +
//             quantization + histogram + restriction; Thomas solves + add }
//             -> level 0 -> codebook -> encode -> header   (Alg. 1, Alg. 2)
// decompress = header -> decode tables -> chunk-parallel decode -> level 0 ->
//             for l = 1..L { restriction of the dequantized level; solves and
//             subtract; expand }  (the inverse of Alg. 1)
#include <cstring>
#include <cstdio>
#include <cmath>
#include <new>
#include <algorithm>
#include "internal.cuh"
#include "levels.cuh"
#include "huffman.cuh"

using namespace hpdr;

namespace {

struct DevGuard {
    int prev = -1;
    bool changed = false;
    explicit DevGuard(int d)
    {
        cudaGetDevice(&prev);
        if (prev != d) { changed = cudaSetDevice(d) == cudaSuccess; }
    }
    ~DevGuard() { if (changed) cudaSetDevice(prev); }
};

struct Carver {
    char *p;
    size_t used = 0;
    explicit Carver(void *base) : p((char *)base) {}
    template <typename T> T *take(size_t count)
    {
        size_t off = (used + 255) & ~size_t(255);
        used = off + count * sizeof(T);
        return reinterpret_cast<T *>(p ? p + off : nullptr);
    }
};

hpdr_status map_device_status(unsigned st)
{
    switch (st) {
    case DS_OK: return HPDR_OK;
    case DS_ARG: return HPDR_ERR_ARG;
    case DS_CAPACITY: return HPDR_ERR_CAPACITY;
    case DS_FORMAT: return HPDR_ERR_FORMAT;
    case DS_LENGTH: return HPDR_ERR_CAPACITY;
    case DS_TIMEOUT: return HPDR_ERR_TIMEOUT;
    default: return HPDR_ERR_CUDA;
    }
}

// K = 0 after validation: chosen from the field size (chunk_of)
bool valid_cfg(const hpdr_config *cfg, unsigned &D, unsigned &K)
{
    D = cfg ? cfg->dict_size : 8192;
    K = cfg ? cfg->chunk : 0;
    if (cfg && D == 0) D = 8192;
    if (D < 4 || D > 65536 || (D & 1)) return false;
    if (K != 0 && (K < 128 || K > 32768 || (K % 128))) return false;
    return true;
}

// Symbols per decode chunk when the caller leaves it to the library: every
// chunk is one thread's sequential decode, so smaller fields take shorter
// chunks to keep the GPU's threads busy (about 2^17 chunks or more).
unsigned chunk_of(unsigned K, unsigned long long N)
{
    if (K) return K;
    if (N >= (1ULL << 27)) return 1024;
    if (N >= (1ULL << 26)) return 512;
    return 256;
}

long long total_of(int ndim, const size_t *dims)
{
    long long n = 1;
    for (int k = 0; k < ndim; k++) n *= (long long)dims[k];
    return n;
}

// workspace of one field: scalars, hist, partials, level buffers, symbols,
// escaped codes, chunk tables, Huffman scratch
struct Ws {
    Scalars *sc;
    double *partials;
    unsigned long long *hist;
    void *va, *vb, *b;
    uint16_t *sym;
    long long *esc;
    unsigned long long *chunk_bits;
    unsigned long long *bsum;
    void *huff;
    DevHdr *dh;   // a container header parsed on the device
    double *deq;  // binary64 fields: symbol values per level (null for binary32 and large alphabets)
};

size_t carve_ws(void *base, const Plan *P, size_t esz, unsigned D, unsigned K, bool need_sym, Ws *w)
{
    Carver c(base);
    long long N = P->N[P->L];
    long long Nl1 = P->L >= 1 ? P->N[P->L - 1] : 1;
    unsigned long long nch = (N + K - 1) / K;
    w->sc = c.take<Scalars>(1);
    w->hist = c.take<unsigned long long>(D);
    w->partials = c.take<double>(2 * norm_parts());
    w->va = c.take<char>(Nl1 * esz);
    w->vb = c.take<char>(Nl1 * esz);
    w->b = c.take<char>(Nl1 * esz);
    w->sym = need_sym ? c.take<uint16_t>(N + 8) : nullptr;
    w->esc = need_sym ? c.take<long long>(N) : nullptr;
    w->chunk_bits = c.take<unsigned long long>(nch + 2);
    w->bsum = c.take<unsigned long long>(1024);
    w->huff = c.take<char>(huff_scratch_bytes(D));
    w->dh = c.take<DevHdr>(1);
    w->deq = esz == 8 && need_sym && D <= kDeqMaxD ? c.take<double>((size_t)(P->L + 1) * D) : nullptr;
    return c.used + 256;
}

// diagnostics group names of the levels below the finest
#define LN(p) {p "_l0", p "_l1", p "_l2", p "_l3", p "_l4", p "_l5", p "_l6", p "_l7", p "_l8", p "_l9", \
               p "_l10", p "_l11", p "_l12", p "_l13", p "_l14", p "_l15", p "_l16", p "_l17", p "_l18", \
               p "_l19", p "_l20", p "_l21", p "_l22", p "_l23", p "_l24", p "_l25", p "_l26", p "_l27", \
               p "_l28", p "_l29", p "_l30", p "_l31", p "_l32", p "_l33", p "_l34", p "_l35", p "_l36", \
               p "_l37", p "_l38", p "_l39", p "_l40"}
const char *const kLevelName[5][kMaxLevels + 1] = {LN("c_restrict_quant"), LN("c_solves"), LN("d_restrict_sym"),
                                                   LN("d_solves"), LN("d_expand")};
#undef LN

template <typename T> const LevelGeom<T> &geom(const Plan *P, int l);
template <> const LevelGeom<float> &geom<float>(const Plan *P, int l) { return P->gf[l]; }
template <> const LevelGeom<double> &geom<double>(const Plan *P, int l) { return P->gd[l]; }

#define CK(x)                                                    \
    do {                                                         \
        cudaError_t _e = (x);                                    \
        if (_e != cudaSuccess) { return HPDR_ERR_CUDA; }         \
    } while (0)

// ----- statistical L2 bins (mode 2) ----------------------------------------
// The paper names an L2 mode without a bin rule; the rule taken here bounds
// the expected squared L2 error.  Coefficient errors on the new nodes of
// level l enter the reconstruction as (I - Q_{l-1}) f_l, f_l their level-l
// piecewise-linear function; the components are L2-orthogonal across levels,
// so E||u - u~||^2 <= sum_l (q_l^2 / 12) S_l for independent uniform errors,
// S_l = the level-l mass-matrix diagonal summed over the level's new nodes.
// The budget tau'^2 T (T = trace of the finest mass matrix) is split evenly:
//     q_l = sqrt(12 tau'^2 T / ((L+1) S_l)).
// The diagonal is a product of 1-D diagonals, so the sum over all nodes of a
// level is a product of 1-D sums A_k and the sum over its kept nodes a
// product of sums B_k over the kept positions: S_l = prod A_k - prod B_k
// (S_0 = prod A_k), T = prod A_k on the finest level.
struct L2sArgs {
    int L;
    double eps, T;
    double S[kMaxLevels + 1];
};

void l2s_weights(const Plan *P, L2sArgs &a)
{
    const int L = P->L, pad = 3 - P->ndim;
    double A[3][kMaxLevels + 1], B[3][kMaxLevels + 1];
    size_t co = 0;
    for (int k = 0; k < 3; k++) {
        for (int l = 0; l <= L; l++) A[k][l] = B[k][l] = 1.0;
        if (k < pad) continue;
        const int n = (int)P->n[k];
        std::vector<double> x(n);
        for (int i = 0; i < n; i++) x[i] = P->coords.empty() ? (double)i : P->coords[co + i];
        co += n;
        auto diag = [&](int i) {
            double h = 0.0;
            if (i > 0) h += x[i] - x[i - 1];
            if (i + 1 < (int)x.size()) h += x[i + 1] - x[i];
            return h / 3.0;
        };
        for (int l = L; l >= 0; l--) {
            const int m = (int)x.size(), mc = l > 0 ? P->m[k][l - 1] : 0;
            double sa = 0.0, sb = 0.0;
            for (int i = 0; i < m; i++) sa += diag(i);
            for (int j = 0; j < mc; j++) sb += diag(cpos_of(m, mc, j));
            A[k][l] = sa;
            B[k][l] = sb;
            if (l > 0) {
                std::vector<double> xc(mc);
                for (int j = 0; j < mc; j++) xc[j] = x[cpos_of(m, mc, j)];
                x.swap(xc);
            }
        }
    }
    a.L = L;
    for (int l = 0; l <= L; l++) {
        const double pa = A[0][l] * A[1][l] * A[2][l];
        a.S[l] = l == 0 ? pa : pa - B[0][l] * B[1][l] * B[2][l];
        if (l == L) a.T = pa;
    }
}

// runs after the norm pass (which set the norm, tau and the status of the
// bound) and replaces its bins; a rejected bound or a zero field keeps them
__global__ void bins_l2s_kernel(L2sArgs a, Scalars *sc)
{
    next_begin();
    if (sc->status) return;
    const double mx = sc->maxabs;
    if (!(mx > 0.0)) return;
    const double tp = __dsub_rn(sc->tau_abs, __dmul_rn(__dmul_rn(__dmul_rn(32.0, (double)(a.L + 1)), a.eps), mx));
    for (int l = threadIdx.x; l <= a.L; l += blockDim.x) {
        const double q = __dsqrt_rn(__ddiv_rn(__dmul_rn(__dmul_rn(12.0, __dmul_rn(tp, tp)), a.T),
                                              __dmul_rn((double)(a.L + 1), a.S[l])));
        sc->q[l] = q;
        const double r = __ddiv_rn(1.0, q);
        sc->rho_d[l] = r;
        sc->rho_f[l] = __double2float_rn(r);
        sc->rho_lo[l] = __double2float_rn(__dsub_rn(r, (double)sc->rho_f[l]));
        sc->q_f[l] = __double2float_rn(q);
    }
}

// the container header's fields of one compression
template <typename T>
HeaderArgs header_args(const Plan *P, int ndim, const size_t *dims, double tol, int tol_kind, int mode, unsigned D,
                       unsigned K, const Ws &w)
{
    HeaderArgs h;
    memset(&h, 0, sizeof(h));
    h.dtype = sizeof(T) == 4 ? 0 : 1;
    h.ndim = ndim;
    h.L = P->L;
    h.mode = mode;
    h.tol_kind = tol_kind;
    for (int k = 0; k < 3; k++) h.dims[k] = k < ndim ? dims[k] : 1;
    h.D = D; h.K = K; h.tol = tol; h.N = (unsigned long long)P->N[P->L]; h.hist = w.hist;
    h.coords = P->coords_dev; h.ncoord = P->coords.size();
    return h;
}

// the phases of one compression; the batched path runs each phase for all
// of its fields before the next (the single-block phases as one launch)
enum : int { kPhLevels = 1, kPhCoarse = 2, kPhCodebook = 4, kPhEncode = 8, kPhHeader = 16, kPhAll = 31 };

// the whole compression of one field (or the selected phases of it),
// enqueued on s without any host wait; the container size and status stay
// in w.sc (device), and in the device pair size_status where the caller gives one
template <typename T>
hpdr_status compress_core(hpdr_ctx *ctx, const Plan *P, const T *u, int ndim, const size_t *dims, double tol,
                          int tol_kind, int mode, unsigned D, unsigned K, uint8_t *out, size_t cap, const Ws &w,
                          cudaStream_t s, int phases = kPhAll, unsigned long long *size_status = nullptr)
{
    const int L = P->L;
    const long long N = P->N[L];
    QuantOut qo;
    qo.sym = w.sym; qo.hist = w.hist; qo.esc = w.esc;
    qo.D = D; qo.sc = w.sc;
    const LevelGeom<T> *geo = &geom<T>(P, 0);
    const int ls = coarse_top<T>(P, geo);
    // the level-ls grid the coarse levels start from
    const T *vtop = (ls >= L) ? u : (const T *)(((L - ls - 1) % 2 == 0) ? w.va : w.vb);
    HuffScratch hs;
    huff_scratch_carve(w.huff, D, w.sc, &hs);
    if (phases & kPhLevels) {
    // the scalars and the histogram are neighbours in the workspace
    CK(cudaMemsetAsync(w.sc, 0, (size_t)((char *)(w.hist + D) - (char *)w.sc), s));
    BinArgs ba;
    memset(&ba, 0, sizeof(ba));
    ba.L = L;
    for (int l = 0; l <= L; l++) ba.c[l] = P->corr_norm[l];
    ba.tol = tol;
    ba.tol_kind = tol_kind;
    ba.mode = mode == 2 ? 1 : mode;   // both L2 modes take the RMS norm
    ba.eps = sizeof(T) == 4 ? ldexp(1.0, -24) : ldexp(1.0, -53);
    ba.N = N;
    {
    ProfScope ps(ctx, "norm", s);
    CK(launch_norm<T>(u, N, w.partials, ba, w.sc, s));
    }
    if (mode == 2) {
        L2sArgs la;
        memset(&la, 0, sizeof(la));
        l2s_weights(P, la);
        la.eps = ba.eps;
        count_launch();
        CK(launch_next(bins_l2s_kernel, 1, 32, 0, s, la, w.sc));
    }

    const T *v = u;
    for (int l = L; l > ls; l--) {
        T *vc = (T *)(((L - l) % 2 == 0) ? w.va : w.vb);
        RestrictArgs<T> a;
        memset(&a, 0, sizeof(a));
        a.g = geom<T>(P, l);
        a.v = v;
        a.src_end = v + P->N[l];
        a.status = &w.sc->status;
        a.qo = qo;
        a.b = (T *)w.b;
        a.vc = vc;
        {
        ProfScope ps(ctx, l == L ? "c_restrict_quant_L" : kLevelName[0][l], s);
        CK(launch_restrict<T>(WSrc::FIELD, Sink::QUANT, a, s));
        }
        {
        ProfScope ps(ctx, l == L ? "c_solves_L" : kLevelName[1][l], s);
        CK(launch_solves<T>(a.g, (T *)w.b, vc, +1, s));
        }
        v = vc;
    }
    }
    // levels 1..ls and level 0 in one CTA (ls = 0: none fits; level 0 alone)
    if (phases & kPhCoarse) {
        if (ls >= 1) {
            ProfScope ps(ctx, "c_coarse", s);
            SymIn none;
            memset(&none, 0, sizeof(none));
            CK(launch_coarse<T>(0, P, geo, ls, vtop, nullptr, qo, nullptr, none, nullptr, s));
        } else {
            CK(launch_level0<T>(Sink::QUANT, vtop, P->N[0], nullptr, qo, s));
        }
    }
    if (phases & kPhCodebook) {
        ProfScope ps(ctx, "c_codebook", s);
        CK(launch_codebook(w.hist, D, hs, s));
    }
    if (!(phases & (kPhEncode | kPhHeader))) return HPDR_OK;
    EncodeArgs ea;
    memset(&ea, 0, sizeof(ea));
    ea.sym = w.sym; ea.N = (unsigned long long)N; ea.D = D; ea.K = K;
    ea.len = hs.len; ea.code = hs.code; ea.pack = hs.pack;
    ea.esc = w.esc;
    ea.chunk_bits = w.chunk_bits; ea.sc = w.sc;
    ea.bsum = w.bsum;
    ea.container = out; ea.L = L; ea.capacity = cap;
    ea.ncoord = P->coords.size();
    if (phases & kPhEncode) {
        ProfScope ps(ctx, "c_encode", s);
        CK(launch_encode(ea, s));
    }
    if (!(phases & kPhHeader)) return HPDR_OK;
    HeaderJob hj;
    hj.h = header_args<T>(P, ndim, dims, tol, tol_kind, mode, D, K, w);
    hj.len = hs.len;
    hj.sc = w.sc;
    hj.out = out;
    hj.size_status = size_status;
    CK(launch_header(hj, s));
    return HPDR_OK;
}

// h_size_status == null: synchronize and return the size in *out_bytes;
// otherwise the call is left in flight and {size, device status} are copied
// into the pinned host pair h_size_status when the stream gets there
template <typename T>
hpdr_status compress_t(hpdr_ctx *ctx, const Plan *P, const T *u, int ndim, const size_t *dims,
                       double tol, int tol_kind, int mode, unsigned D, unsigned K, uint8_t *out,
                       size_t cap, size_t *out_bytes, cudaStream_t s,
                       unsigned long long *h_size_status = nullptr, unsigned long long *d_pair = nullptr)
{
    K = chunk_of(K, (unsigned long long)P->N[P->L]);
    Ws w;
    size_t need = carve_ws(nullptr, P, sizeof(T), D, K, true, &w);
    hpdr_status st = ensure_workspace(ctx, need);
    if (st != HPDR_OK) return st;
    carve_ws(ctx->ws.base, P, sizeof(T), D, K, true, &w);
    st = compress_core<T>(ctx, P, u, ndim, dims, tol, tol_kind, mode, D, K, out, cap, w, s, kPhAll,
                          h_size_status ? d_pair : nullptr);
    if (st != HPDR_OK) return st;
    if (h_size_status) {
        CK(cudaMemcpyAsync(h_size_status, d_pair, 2 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
        return HPDR_OK;
    }
    Scalars *hsc = (Scalars *)ctx->host_pinned;
    CK(cudaMemcpyAsync(hsc, w.sc, sizeof(Scalars), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (hsc->status) return map_device_status(hsc->status);
    *out_bytes = (size_t)hsc->out_bytes;
    return HPDR_OK;
}

// ----- container header (host side) --------------------------------------
struct Hdr {
    int dtype, ndim, L, mode, tol_kind;
    size_t dims[3];
    unsigned D, K, s_lo, s_hi, esc_w;
    unsigned long long N, n_esc, bits, nch, nwords;
    unsigned long long ncoord;   // node coordinates after q (0: unit spacing)
    unsigned long long off_len, off_chunk, off_bits, total;
    double q[kMaxLevels + 1];
};

uint32_t crc32_host(const uint8_t *p, int n)
{
    uint32_t c = 0xFFFFFFFFu;
    for (int i = 0; i < n; i++) {
        c ^= p[i];
        for (int b = 0; b < 8; b++) c = (c >> 1) ^ (0xEDB88320u & (0u - (c & 1u)));
    }
    return c ^ 0xFFFFFFFFu;
}
uint32_t rd32(const uint8_t *p) { uint32_t v = 0; for (int i = 0; i < 4; i++) v |= (uint32_t)p[i] << (8 * i); return v; }
uint64_t rd64(const uint8_t *p) { uint64_t v = 0; for (int i = 0; i < 8; i++) v |= (uint64_t)p[i] << (8 * i); return v; }

hpdr_status parse_header(const uint8_t *b, size_t avail, size_t in_bytes, Hdr *h)
{
    if (in_bytes < 128 || avail < 128) return HPDR_ERR_FORMAT;
    if (memcmp(b, "HPDR", 4) != 0 || rd32(b + 4) != 3) return HPDR_ERR_FORMAT;
    if (crc32_host(b, 124) != rd32(b + 124)) return HPDR_ERR_FORMAT;
    h->dtype = (int)rd32(b + 8);
    h->ndim = (int)rd32(b + 12);
    if (h->dtype < 0 || h->dtype > 1 || h->ndim < 1 || h->ndim > 3) return HPDR_ERR_FORMAT;
    for (int k = 0; k < 3; k++) h->dims[k] = (size_t)rd64(b + 16 + 8 * k);
    for (int k = 0; k < h->ndim; k++) if (h->dims[k] < 2 || h->dims[k] > (1u << 30)) return HPDR_ERR_FORMAT;
    h->L = (int)rd32(b + 40);
    h->mode = (int)rd32(b + 44);
    const uint32_t tk = rd32(b + 48);
    if (tk & ~0x101u) return HPDR_ERR_FORMAT;
    h->tol_kind = (int)(tk & 1u);
    h->D = rd32(b + 52);
    h->K = rd32(b + 56);
    h->s_lo = rd32(b + 60);
    h->N = rd64(b + 96);
    h->n_esc = rd64(b + 104);
    h->bits = rd64(b + 112);
    h->s_hi = rd32(b + 120) & 0xFFFFu;
    h->esc_w = (rd32(b + 120) >> 16) & 0xFFu;
    if (rd32(b + 120) >> 24) return HPDR_ERR_FORMAT;
    if (levels_of(h->ndim, h->dims) != h->L || h->L > kMaxLevels) return HPDR_ERR_FORMAT;
    if ((long long)h->N != total_of(h->ndim, h->dims)) return HPDR_ERR_FORMAT;
    if (h->D < 4 || h->D > 65536 || (h->D & 1) || h->K < 128 || h->K > 32768 || (h->K % 128))
        return HPDR_ERR_FORMAT;
    if (h->s_hi >= h->D || h->s_lo > h->s_hi || h->n_esc > h->N) return HPDR_ERR_FORMAT;
    if (h->esc_w > 63 || (h->n_esc > 0) != (h->esc_w > 0)) return HPDR_ERR_FORMAT;
    // at most 63 code bits per symbol plus the payload of every escape
    if (h->bits > 63ULL * h->N + (unsigned long long)h->esc_w * h->n_esc || h->bits < h->N)
        return HPDR_ERR_FORMAT;
    h->nch = (h->N + h->K - 1) / h->K;
    h->nwords = (h->bits + 31) / 32;
    h->ncoord = 0;
    if (tk & 0x100u) for (int k = 0; k < h->ndim; k++) h->ncoord += h->dims[k];
    h->off_len = a16(128 + 8ULL * (h->L + 1) + 8ULL * h->ncoord);
    h->off_chunk = a16(h->off_len + (h->s_hi - h->s_lo + 1));
    h->off_bits = a16(h->off_chunk + 8 * h->nch);
    h->total = h->off_bits + 4 * h->nwords;
    if (h->total > in_bytes) return HPDR_ERR_FORMAT;
    if (avail >= 128 + 8ULL * (h->L + 1))
        for (int l = 0; l <= h->L; l++) {
            uint64_t u = rd64(b + 128 + 8 * l);
            memcpy(&h->q[l], &u, 8);
            if (!(h->q[l] > 0.0) || !std::isfinite(h->q[l])) return HPDR_ERR_FORMAT;
        }
    return HPDR_OK;
}

// status of one decompression OR-ed into an accumulated word
__global__ void accumulate_status_kernel(const Scalars *sc, unsigned *acc)
{
    next_begin();
    if (sc->status) atomicOr(acc, sc->status);
}

// err_acc == null: synchronize and report this call's status; otherwise the
// call is left in flight and its status OR-ed into *err_acc on the device
// the levels of one decompression, after its symbols are decoded (Sec. IV-A:
// the inverse of Alg. 1 -- dequantization, mass_trans, tridiag and the
// correction, then the interpolation up to the next level)
template <typename T>
hpdr_status decompress_levels(hpdr_ctx *ctx, const Plan *P, unsigned D, unsigned long long N, const Ws &w, T *out,
                              cudaStream_t s)
{
    const int L = P->L;
    SymIn si;
    si.sym = w.sym; si.D = D; si.sc = w.sc; si.esc = w.esc;
    si.status = &w.sc->status;
    si.deq = w.deq;
    // level buffers: v_{l-1} in X, v_l written to Y (or to out at l = L)
    T *bufs[2] = {(T *)w.va, (T *)w.vb};
    const LevelGeom<T> *geo = &geom<T>(P, 0);
    const int ls = coarse_top<T>(P, geo);
    T *v;
    if (ls >= 1) {
        // levels 0..ls in one CTA, level ls written where level ls + 1 reads it
        v = (ls == L) ? out : bufs[ls % 2];
        ProfScope ps(ctx, "d_coarse", s);
        QuantOut none;
        memset(&none, 0, sizeof(none));
        CK(launch_coarse<T>(2, P, geo, ls, nullptr, v, none, nullptr, si, nullptr, s));
    } else {
        v = L == 0 ? out : bufs[0];
        CK(launch_level0_in<T>(WSrc::SYMBOLS, nullptr, si, P->N[0], v, s));
    }
    for (int l = ls + 1; l <= L; l++) {
        const LevelGeom<T> &g = geom<T>(P, l);
        RestrictArgs<T> a;
        memset(&a, 0, sizeof(a));
        a.g = g;
        a.symin = si;
        a.src_end = w.sym + N + 8;
        a.status = &w.sc->status;
        a.b = (T *)w.b;
        {
        ProfScope ps(ctx, l == L ? "d_restrict_sym_L" : kLevelName[2][l], s);
        CK(launch_restrict<T>(WSrc::SYMBOLS, Sink::NONE, a, s));
        }
        {
        ProfScope ps(ctx, l == L ? "d_solves_L" : kLevelName[3][l], s);
        CK(launch_solves<T>(g, (T *)w.b, v, -1, s));
        }
        T *dst = (l == L) ? out : bufs[l % 2];
        {
        ProfScope ps(ctx, l == L ? "d_expand_L" : kLevelName[4][l], s);
        CK(launch_expand<T>(WSrc::SYMBOLS, g, v, nullptr, si, dst, s));
        }
        v = dst;
    }
    return HPDR_OK;
}

template <typename T>
hpdr_status decompress_t(hpdr_ctx *ctx, const Plan *P, const Hdr &h, const uint8_t *in, T *out,
                         cudaStream_t s, unsigned *err_acc = nullptr)
{
    Ws w;
    size_t need = carve_ws(nullptr, P, sizeof(T), h.D, h.K, true, &w);
    hpdr_status st = ensure_workspace(ctx, need);
    if (st != HPDR_OK) return st;
    carve_ws(ctx->ws.base, P, sizeof(T), h.D, h.K, true, &w);
    const int L = P->L;
    Scalars *hsc = (Scalars *)ctx->host_pinned;
    HuffScratch hs;
    huff_scratch_carve(w.huff, h.D, w.sc, &hs);
    {
    // the decoder-side scalars come with the launch parameters (no host staging
    // buffer, so calls need not wait)
    ProfScope ps(ctx, "d_tables", s);
    TabArgs ta;
    ta.lenb = in + h.off_len; ta.s_lo = h.s_lo; ta.s_hi = h.s_hi; ta.D = h.D;
    ta.sc = w.sc;
    ta.set_scalars = true;
    ta.deq = w.deq;
    for (int l = 0; l <= L; l++) ta.si.q[l] = h.q[l];
    ta.si.L = L;
    ta.si.n_esc = h.n_esc;
    ta.si.esc_w = h.esc_w;
    ta.si.total_bits = h.bits;
    CK(launch_decode_tables(ta, hs, s));
    }
    DecodeArgs da;
    da.words = (const uint32_t *)(in + h.off_bits);
    da.nwords = h.nwords;
    da.chunk = (const unsigned long long *)(in + h.off_chunk);
    da.N = h.N; da.total_bits = h.bits; da.K = h.K; da.sym = w.sym;
    da.esc = h.esc_w ? w.esc : nullptr; da.esc_w = h.esc_w; da.n_esc = h.n_esc;
    {
    ProfScope ps(ctx, "d_decode", s);
    CK(launch_decode(da, hs, s));
    }
    st = decompress_levels<T>(ctx, P, h.D, h.N, w, out, s);
    if (st != HPDR_OK) return st;
    if (err_acc) {
        count_launch();
        CK(launch_next(accumulate_status_kernel, 1, 1, 0, s, w.sc, err_acc));
        return HPDR_OK;
    }
    CK(cudaMemcpyAsync(hsc, w.sc, sizeof(Scalars), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (hsc->status) return map_device_status(hsc->status);
    return HPDR_OK;
}

// {status} of one call into a device word
__global__ void status_out_kernel(const Scalars *sc, unsigned long long *dst)
{
    next_begin();
    dst[0] = sc->status;
}

// decompression whose header is read on the device: no host wait
template <typename T>
hpdr_status decompress_dev(hpdr_ctx *ctx, const Plan *P, int dtype, int ndim, const size_t *dims, unsigned D,
                           unsigned K, const uint8_t *in, size_t in_bytes, T *out, unsigned long long *d_result,
                           cudaStream_t s)
{
    K = chunk_of(K, (unsigned long long)P->N[P->L]);
    Ws w;
    size_t need = carve_ws(nullptr, P, sizeof(T), D, K, true, &w);
    hpdr_status st = ensure_workspace(ctx, need);
    if (st != HPDR_OK) return st;
    carve_ws(ctx->ws.base, P, sizeof(T), D, K, true, &w);
    HuffScratch hs;
    huff_scratch_carve(w.huff, D, w.sc, &hs);
    TabArgs ta;
    ta.D = D;
    ta.sc = w.sc;
    ta.base = in; ta.in_bytes = in_bytes; ta.dh = w.dh;
    ta.deq = w.deq;
    HdrExpect &ex = ta.ex;
    ex.dtype = dtype;
    ex.ndim = ndim;
    ex.L = P->L;
    for (int k = 0; k < 3; k++) ex.dims[k] = k < ndim ? dims[k] : 1;
    ex.N = (unsigned long long)P->N[P->L];
    ex.D = D;
    ex.K = K;
    {
    ProfScope ps(ctx, "d_tables", s);
    CK(launch_decode_tables(ta, hs, s));
    }
    DecodeArgs da;
    da.words = nullptr; da.nwords = 0; da.chunk = nullptr; da.total_bits = 0; da.esc_w = 0;
    da.N = ex.N; da.K = K; da.sym = w.sym; da.esc = w.esc;
    da.base = in; da.dh = w.dh;
    {
    ProfScope ps(ctx, "d_decode", s);
    CK(launch_decode(da, hs, s));
    }
    st = decompress_levels<T>(ctx, P, D, ex.N, w, out, s);
    if (st != HPDR_OK) return st;
    count_launch();
    CK(launch_next(status_out_kernel, 1, 1, 0, s, w.sc, d_result));
    return HPDR_OK;
}

// node coordinates of a container (empty with unit spacing) from a host copy
// that holds at least its first 128 + 8 (L + 1 + ncoord) bytes
void read_coords(const uint8_t *b, const Hdr &h, std::vector<double> &co)
{
    co.resize(h.ncoord);
    for (unsigned long long i = 0; i < h.ncoord; i++) {
        uint64_t u = rd64(b + 128 + 8 * (h.L + 1) + 8 * i);
        memcpy(&co[i], &u, 8);
    }
}

// Decompression of a container whose header the caller already holds in
// host memory (hdr_host, hdr_bytes): no header read-back, and with err_acc the
// call does not wait (status OR-ed into *err_acc on the device).
hpdr_status decompress_with_header(hpdr_ctx *ctx, const uint8_t *hdr_host, size_t hdr_bytes, const void *d_in,
                                   size_t in_bytes, void *d_out, size_t out_capacity, cudaStream_t s,
                                   unsigned *err_acc)
{
    Hdr h;
    hpdr_status st = parse_header(hdr_host, hdr_bytes, in_bytes, &h);
    if (st != HPDR_OK) return st;
    if (hdr_bytes < 128 + 8ULL * (h.L + 1 + h.ncoord)) return HPDR_ERR_FORMAT;
    const size_t esz = h.dtype == 0 ? 4 : 8;
    if (out_capacity < h.N * esz) return HPDR_ERR_CAPACITY;
    std::vector<double> co;
    read_coords(hdr_host, h, co);
    Plan *P;
    st = get_plan(ctx, h.ndim, h.dims, h.dtype == 1, &P, co.empty() ? nullptr : co.data());
    if (st != HPDR_OK) return st;
    if (h.dtype == 0) return decompress_t<float>(ctx, P, h, (const uint8_t *)d_in, (float *)d_out, s, err_acc);
    return decompress_t<double>(ctx, P, h, (const uint8_t *)d_in, (double *)d_out, s, err_acc);
}

template <typename T>
hpdr_status decompose_t(hpdr_ctx *ctx, const Plan *P, const T *u, T *coef, cudaStream_t s)
{
    Ws w;
    size_t need = carve_ws(nullptr, P, sizeof(T), 4, 128, false, &w);
    hpdr_status st = ensure_workspace(ctx, need);
    if (st != HPDR_OK) return st;
    carve_ws(ctx->ws.base, P, sizeof(T), 4, 128, false, &w);
    const int L = P->L;
    const T *v = u;
    CK(cudaMemsetAsync(w.sc, 0, sizeof(Scalars), s));
    QuantOut qo;
    memset(&qo, 0, sizeof(qo));
    const LevelGeom<T> *geo = &geom<T>(P, 0);
    const int ls = coarse_top<T>(P, geo);
    for (int l = L; l > ls; l--) {
        T *vc = (T *)(((L - l) % 2 == 0) ? w.va : w.vb);
        RestrictArgs<T> a;
        memset(&a, 0, sizeof(a));
        a.g = geom<T>(P, l);
        a.v = v;
        a.src_end = v + P->N[l];
        a.status = &w.sc->status;
        a.coef_out = coef;
        a.b = (T *)w.b;
        a.vc = vc;
        CK(launch_restrict<T>(WSrc::FIELD, Sink::STREAM, a, s));
        CK(launch_solves<T>(a.g, (T *)w.b, vc, +1, s));
        v = vc;
    }
    if (ls >= 1) {
        SymIn none;
        memset(&none, 0, sizeof(none));
        CK(launch_coarse<T>(1, P, geo, ls, v, nullptr, qo, coef, none, nullptr, s));
    } else {
        CK(launch_level0<T>(Sink::STREAM, v, P->N[0], coef, qo, s));
    }
    return HPDR_OK;
}

template <typename T>
hpdr_status recompose_t(hpdr_ctx *ctx, const Plan *P, const T *coef, T *out, cudaStream_t s)
{
    Ws w;
    size_t need = carve_ws(nullptr, P, sizeof(T), 4, 128, false, &w);
    hpdr_status st = ensure_workspace(ctx, need);
    if (st != HPDR_OK) return st;
    carve_ws(ctx->ws.base, P, sizeof(T), 4, 128, false, &w);
    const int L = P->L;
    SymIn si;
    memset(&si, 0, sizeof(si));
    T *bufs[2] = {(T *)w.va, (T *)w.vb};
    const LevelGeom<T> *geo = &geom<T>(P, 0);
    const int ls = coarse_top<T>(P, geo);
    T *v;
    if (ls >= 1) {
        v = (ls == L) ? out : bufs[ls % 2];
        QuantOut none;
        memset(&none, 0, sizeof(none));
        CK(launch_coarse<T>(3, P, geo, ls, nullptr, v, none, nullptr, si, coef, s));
    } else {
        v = L == 0 ? out : bufs[0];
        CK(launch_level0_in<T>(WSrc::STREAM, coef, si, P->N[0], v, s));
    }
    for (int l = ls + 1; l <= L; l++) {
        const LevelGeom<T> &g = geom<T>(P, l);
        RestrictArgs<T> a;
        memset(&a, 0, sizeof(a));
        a.g = g;
        a.coef_in = coef;
        a.b = (T *)w.b;
        CK(launch_restrict<T>(WSrc::STREAM, Sink::NONE, a, s));
        CK(launch_solves<T>(g, (T *)w.b, v, -1, s));
        T *dst = (l == L) ? out : bufs[l % 2];
        CK(launch_expand<T>(WSrc::STREAM, g, v, coef, si, dst, s));
        v = dst;
    }
    return HPDR_OK;
}

template <typename T> const LevelGeom<T> *geos(const Plan *P);
template <> const LevelGeom<float> *geos<float>(const Plan *P) { return P->gf; }
template <> const LevelGeom<double> *geos<double>(const Plan *P) { return P->gd; }

template <typename T>
hpdr_status adjoint_t(hpdr_ctx *ctx, const Plan *P, const T *in, T *out, bool recompose, cudaStream_t s)
{
    const int L = P->L;
    const size_t n1 = L >= 1 ? (size_t)P->N[L - 1] : 1;
    Carver c(nullptr);
    c.take<Scalars>(1);
    for (int i = 0; i < 4; i++) c.take<T>(n1);
    hpdr_status st = ensure_workspace(ctx, c.used + 256);
    if (st != HPDR_OK) return st;
    Carver w(ctx->ws.base);
    Scalars *sc = w.take<Scalars>(1);
    T *ga = w.take<T>(n1), *gb = w.take<T>(n1), *y = w.take<T>(n1), *R = w.take<T>(n1);
    CK(cudaMemsetAsync(sc, 0, sizeof(Scalars), s));
    if (recompose) {
        ProfScope ps(ctx, "adj_recompose", s);
        CK(recompose_adjoint_run<T>(*P, geos<T>(P), in, out, ga, gb, y, &sc->status, s));
    } else {
        ProfScope ps(ctx, "adj_decompose", s);
        CK(decompose_adjoint_run<T>(*P, geos<T>(P), in, out, ga, gb, y, R, &sc->status, s));
    }
    return HPDR_OK;
}

// ---- batched compression ------------------------------------------------

struct BatchPlan {
    int nfields = 0;
    std::vector<Plan *> plans;
    std::vector<size_t> ws_off, out_off, bound;
    size_t ws_total = 0;
    void *ws = nullptr;
    unsigned long long *sizes = nullptr;   // device [nfields][2]: container bytes, status
    cudaGraphExec_t exec = nullptr;
    int streams = 0;
    double tuned_ms = 0.0;
    unsigned long long last_use = 0;   // call counter of the last replay (least recently used goes first)
    // device job arrays of the single-block phases (one block per field)
    void *jobs = nullptr;
    CoarseArgs<float> *coarse32 = nullptr;
    CoarseArgs<double> *coarse64 = nullptr;
    int n32 = 0, n64 = 0;
    size_t sm32 = 0, sm64 = 0;
    std::vector<int> coarse_ls;          // per field: coarse_top (0: level 0 alone, in its field's phase)
    CodebookJob *codebooks = nullptr;    // [nfields]
    HeaderJob *headers = nullptr;        // [nfields]
};

// Captured batches kept per context: a graph holds the pointers it was
// captured with, so a batch over other buffers is another entry; beyond this
// many the least recently used entry is destroyed (graph, workspace, sizes).
constexpr size_t kMaxBatchPlans = 4;
void free_batch_plan(BatchPlan *bp)
{
    if (bp->exec) cudaGraphExecDestroy(bp->exec);
    cudaFree(bp->jobs);
    cudaFree(bp->ws);
    cudaFree(bp->sizes);
    delete bp;
}

struct BatchRes {
    cudaStream_t origin = nullptr;
    std::vector<cudaStream_t> workers;
    cudaEvent_t fork = nullptr;
    std::vector<cudaEvent_t> join;
    std::map<std::string, BatchPlan *> plans;
    unsigned long long calls = 0;
};

hpdr_status batch_res(hpdr_ctx *ctx, BatchRes *&r, int nworkers)
{
    if (!ctx->batch_res) {
        r = new BatchRes();
        if (cudaStreamCreateWithFlags(&r->origin, cudaStreamNonBlocking) != cudaSuccess) return HPDR_ERR_CUDA;
        if (cudaEventCreateWithFlags(&r->fork, cudaEventDisableTiming) != cudaSuccess) return HPDR_ERR_CUDA;
        ctx->batch_res = r;
    }
    r = (BatchRes *)ctx->batch_res;
    while ((int)r->workers.size() < nworkers) {
        cudaStream_t st;
        cudaEvent_t ev;
        if (cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking) != cudaSuccess) return HPDR_ERR_CUDA;
        if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) return HPDR_ERR_CUDA;
        r->workers.push_back(st);
        r->join.push_back(ev);
    }
    return HPDR_OK;
}

// fields assigned largest first to the least-loaded of K streams
std::vector<std::vector<int>> schedule(const hpdr_field *f, int n, int K)
{
    std::vector<int> order(n);
    for (int i = 0; i < n; i++) order[i] = i;
    auto work = [&](int i) {
        double w = f[i].dtype == HPDR_F64 ? 8.0 : 4.0;
        for (int k = 0; k < f[i].ndim; k++) w *= (double)f[i].dims[k];
        return w;
    };
    std::sort(order.begin(), order.end(), [&](int a, int b) { return work(a) > work(b); });
    std::vector<std::vector<int>> q(K);
    std::vector<double> load(K, 0.0);
    for (int i : order) {
        int k = (int)(std::min_element(load.begin(), load.end()) - load.begin());
        q[k].push_back(i);
        load[k] += work(i);
    }
    return q;
}

// the field's workspace inside the batch's workspace
Ws batch_ws(const BatchPlan *bp, const hpdr_field *f, int i, unsigned D, unsigned K)
{
    const Plan *P = bp->plans[i];
    const unsigned Ki = chunk_of(K, (unsigned long long)P->N[P->L]);
    Ws w;
    carve_ws((char *)bp->ws + bp->ws_off[i], P, f[i].dtype == HPDR_F64 ? 8 : 4, D, Ki, true, &w);
    return w;
}

// the job arrays of the single-block phases, built once per batch plan
template <typename T>
void batch_field_jobs(const BatchPlan *bp, const hpdr_field *f, int i, unsigned D, unsigned K, uint8_t *d_out,
                      std::vector<CoarseArgs<T>> &coarse, size_t &smem, int &ls, CodebookJob &cb, HeaderJob &hj)
{
    const Plan *P = bp->plans[i];
    const unsigned Ki = chunk_of(K, (unsigned long long)P->N[P->L]);
    const Ws w = batch_ws(bp, f, i, D, K);
    const int L = P->L;
    const LevelGeom<T> *geo = &geom<T>(P, 0);
    ls = coarse_top<T>(P, geo);
    QuantOut qo;
    qo.sym = w.sym; qo.hist = w.hist; qo.esc = w.esc;
    qo.D = D; qo.sc = w.sc;
    HuffScratch hs;
    huff_scratch_carve(w.huff, D, w.sc, &hs);
    if (ls >= 1) {
        const T *vtop = (ls >= L) ? (const T *)f[i].d_in : (const T *)(((L - ls - 1) % 2 == 0) ? w.va : w.vb);
        SymIn none;
        memset(&none, 0, sizeof(none));
        size_t sm = 0;
        coarse.push_back(coarse_args<T>(0, P, geo, ls, vtop, nullptr, qo, nullptr, none, nullptr, &sm));
        smem = std::max(smem, sm);
    }
    cb.hist = w.hist;
    cb.D = D;
    cb.hs = hs;
    hj.h = header_args<T>(P, f[i].ndim, f[i].dims, f[i].tol, f[i].tol_kind, f[i].mode, D, Ki, w);
    hj.len = hs.len;
    hj.sc = w.sc;
    hj.out = d_out + bp->out_off[i];
    hj.size_status = bp->sizes + 2 * i;
}

hpdr_status build_batch_jobs(BatchPlan *bp, const hpdr_field *f, unsigned D, unsigned K, uint8_t *d_out)
{
    const int n = bp->nfields;
    std::vector<CoarseArgs<float>> c32;
    std::vector<CoarseArgs<double>> c64;
    std::vector<CodebookJob> cb(n);
    std::vector<HeaderJob> hj(n);
    bp->coarse_ls.assign(n, 0);
    for (int i = 0; i < n; i++) {
        if (f[i].dtype == HPDR_F64)
            batch_field_jobs<double>(bp, f, i, D, K, d_out, c64, bp->sm64, bp->coarse_ls[i], cb[i], hj[i]);
        else
            batch_field_jobs<float>(bp, f, i, D, K, d_out, c32, bp->sm32, bp->coarse_ls[i], cb[i], hj[i]);
    }
    bp->n32 = (int)c32.size();
    bp->n64 = (int)c64.size();
    auto al = [](size_t x) { return (x + 255) & ~size_t(255); };
    const size_t b32 = al(sizeof(CoarseArgs<float>) * c32.size()), b64 = al(sizeof(CoarseArgs<double>) * c64.size());
    const size_t bcb = al(sizeof(CodebookJob) * n), bhj = al(sizeof(HeaderJob) * n);
    if (cudaMalloc(&bp->jobs, b32 + b64 + bcb + bhj) != cudaSuccess) { cudaGetLastError(); return HPDR_ERR_NOMEM; }
    char *p = (char *)bp->jobs;
    bp->coarse32 = (CoarseArgs<float> *)p;
    bp->coarse64 = (CoarseArgs<double> *)(p + b32);
    bp->codebooks = (CodebookJob *)(p + b32 + b64);
    bp->headers = (HeaderJob *)(p + b32 + b64 + bcb);
    // pageable sources: synchronous copies, done before any capture
    if ((c32.size() && cudaMemcpy(bp->coarse32, c32.data(), sizeof(CoarseArgs<float>) * c32.size(),
                                  cudaMemcpyHostToDevice) != cudaSuccess) ||
        (c64.size() && cudaMemcpy(bp->coarse64, c64.data(), sizeof(CoarseArgs<double>) * c64.size(),
                                  cudaMemcpyHostToDevice) != cudaSuccess) ||
        cudaMemcpy(bp->codebooks, cb.data(), sizeof(CodebookJob) * n, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(bp->headers, hj.data(), sizeof(HeaderJob) * n, cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaGetLastError();
        return HPDR_ERR_CUDA;
    }
    return HPDR_OK;
}

// The batch in four phases, each over all fields: (A) per field on the K
// worker streams, norm, bins and the large levels (and level 0 when no level
// fits one CTA); (B) on the origin stream, the coarse levels of every field
// in one launch per element type, then every field's codebook in one launch;
// (C) per field on the workers, the encoder; (D) every header and every
// {bytes, status} pair in one launch.  Each field meets the same kernels in
// the same order as hpdr_compress, so its container is byte-identical.
hpdr_status enqueue_batch(hpdr_ctx *ctx, BatchRes *r, BatchPlan *bp, const hpdr_field *f, unsigned D, unsigned K,
                          uint8_t *d_out, int nstreams)
{
    std::vector<std::vector<int>> q = schedule(f, bp->nfields, nstreams);
    auto fork = [&]() -> bool {
        if (cudaEventRecord(r->fork, r->origin) != cudaSuccess) return false;
        for (int k = 0; k < nstreams; k++)
            if (cudaStreamWaitEvent(r->workers[k], r->fork, 0) != cudaSuccess) return false;
        return true;
    };
    auto join = [&]() -> bool {
        for (int k = 0; k < nstreams; k++) {
            if (cudaEventRecord(r->join[k], r->workers[k]) != cudaSuccess) return false;
            if (cudaStreamWaitEvent(r->origin, r->join[k], 0) != cudaSuccess) return false;
        }
        return true;
    };
    auto field = [&](int i, int phases, cudaStream_t st) -> hpdr_status {
        const Plan *P = bp->plans[i];
        const unsigned Ki = chunk_of(K, (unsigned long long)P->N[P->L]);
        const Ws w = batch_ws(bp, f, i, D, K);
        if (f[i].dtype == HPDR_F64)
            return compress_core<double>(ctx, P, (const double *)f[i].d_in, f[i].ndim, f[i].dims, f[i].tol,
                                         f[i].tol_kind, f[i].mode, D, Ki, d_out + bp->out_off[i], bp->bound[i], w,
                                         st, phases);
        return compress_core<float>(ctx, P, (const float *)f[i].d_in, f[i].ndim, f[i].dims, f[i].tol,
                                    f[i].tol_kind, f[i].mode, D, Ki, d_out + bp->out_off[i], bp->bound[i], w, st,
                                    phases);
    };
    // (A)
    if (!fork()) return HPDR_ERR_CUDA;
    for (int k = 0; k < nstreams; k++)
        for (int i : q[k]) {
            const hpdr_status st = field(i, kPhLevels | (bp->coarse_ls[i] < 1 ? kPhCoarse : 0), r->workers[k]);
            if (st != HPDR_OK) return st;
        }
    if (!join()) return HPDR_ERR_CUDA;
    // (B)
    CK(launch_coarse_batch<float>(bp->coarse32, bp->n32, bp->sm32, r->origin));
    CK(launch_coarse_batch<double>(bp->coarse64, bp->n64, bp->sm64, r->origin));
    if (codebook_fused(D)) {
        CK(launch_codebook_batch(bp->codebooks, bp->nfields, r->origin));
    } else {
        for (int i = 0; i < bp->nfields; i++) {
            const hpdr_status st = field(i, kPhCodebook, r->origin);
            if (st != HPDR_OK) return st;
        }
    }
    // (C)
    if (!fork()) return HPDR_ERR_CUDA;
    for (int k = 0; k < nstreams; k++)
        for (int i : q[k]) {
            const hpdr_status st = field(i, kPhEncode, r->workers[k]);
            if (st != HPDR_OK) return st;
        }
    if (!join()) return HPDR_ERR_CUDA;
    // (D)
    CK(launch_header_batch(bp->headers, bp->nfields, r->origin));
    return HPDR_OK;
}
hpdr_status capture_batch(hpdr_ctx *ctx, BatchRes *r, BatchPlan *bp, const hpdr_field *f, unsigned D, unsigned K,
                          uint8_t *d_out, int nstreams, cudaGraphExec_t *exec)
{
    cudaGraph_t g = nullptr;
    if (cudaStreamBeginCapture(r->origin, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return HPDR_ERR_CUDA;
    hpdr_status st = enqueue_batch(ctx, r, bp, f, D, K, d_out, nstreams);
    cudaError_t e = cudaStreamEndCapture(r->origin, &g);
    if (st != HPDR_OK) { if (g) cudaGraphDestroy(g); return st; }
    if (e != cudaSuccess) { cudaGetLastError(); return HPDR_ERR_CUDA; }
    e = cudaGraphInstantiate(exec, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) { cudaGetLastError(); return HPDR_ERR_CUDA; }
    return HPDR_OK;
}

bool is_device_ptr(const void *p)
{
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) { cudaGetLastError(); return false; }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

// ----- lossless container (HPDL) -------------------------------------------
// byte keys travel as 16-bit symbols through the Huffman kernels
__global__ void widen_keys_kernel(const uint8_t *in, unsigned long long n, uint16_t *out)
{
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x)
        out[i] = in[i];
}
__global__ void narrow_keys_kernel(const uint16_t *in, unsigned long long n, uint8_t *out)
{
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x)
        out[i] = (uint8_t)in[i];
}

constexpr unsigned kLosslessHdr = 64;
struct LosslessHdr {
    unsigned key_bytes, D, K;
    unsigned long long n, bits, nch, off_chunk, off_bits, total;
};
void lossless_layout(LosslessHdr *h)
{
    h->nch = (h->n + h->K - 1) / h->K;
    h->off_chunk = a16(kLosslessHdr + h->D);
    h->off_bits = a16(h->off_chunk + 8 * h->nch);
    h->total = h->off_bits + 4 * ((h->bits + 31) / 32);
}
uint32_t rd32l(const uint8_t *p) { uint32_t v = 0; for (int i = 0; i < 4; i++) v |= (uint32_t)p[i] << (8 * i); return v; }
uint64_t rd64l(const uint8_t *p) { uint64_t v = 0; for (int i = 0; i < 8; i++) v |= (uint64_t)p[i] << (8 * i); return v; }

hpdr_status parse_lossless(const uint8_t *b, size_t in_bytes, LosslessHdr *h)
{
    if (in_bytes < kLosslessHdr || memcmp(b, "HPDL", 4) != 0 || rd32l(b + 4) != 1) return HPDR_ERR_FORMAT;
    if (crc32_host(b, 60) != rd32l(b + 60)) return HPDR_ERR_FORMAT;
    h->key_bytes = rd32l(b + 8);
    h->D = rd32l(b + 12);
    h->K = rd32l(b + 16);
    h->n = rd64l(b + 24);
    h->bits = rd64l(b + 32);
    if ((h->key_bytes != 1 && h->key_bytes != 2) || h->D != (h->key_bytes == 1 ? 256u : 65536u)) return HPDR_ERR_FORMAT;
    if (h->K < 128 || h->K > 32768 || (h->K % 128) || h->n == 0 || h->n > (1ull << 40)) return HPDR_ERR_FORMAT;
    if (h->bits > 63ull * h->n) return HPDR_ERR_FORMAT;
    lossless_layout(h);
    if (rd64l(b + 40) != h->off_chunk || rd64l(b + 48) != h->off_bits || h->total > in_bytes) return HPDR_ERR_FORMAT;
    return HPDR_OK;
}

}  // namespace

namespace hpdr {
hpdr_status decompress_in_flight(hpdr_ctx *ctx, const uint8_t *hdr_host, size_t hdr_bytes, const void *d_in,
                                 size_t in_bytes, void *d_out, size_t out_capacity, cudaStream_t s,
                                 unsigned *err_acc)
{
    return decompress_with_header(ctx, hdr_host, hdr_bytes, d_in, in_bytes, d_out, out_capacity, s, err_acc);
}
hpdr_status status_of_device(unsigned st) { return map_device_status(st); }
hpdr_status compress_in_flight(hpdr_ctx *ctx, const void *d_in, hpdr_dtype dtype, int ndim, const size_t *dims,
                               double tol, hpdr_tol_kind tol_kind, hpdr_mode mode, const hpdr_config *cfg,
                               void *d_out, size_t out_capacity, unsigned long long *h_size_status,
                               unsigned long long *d_pair, cudaStream_t s)
{
    unsigned D, K;
    if (!ctx || !d_in || !d_out || !h_size_status || !d_pair || !valid_cfg(cfg, D, K)) return HPDR_ERR_ARG;
    if ((dtype != HPDR_F32 && dtype != HPDR_F64) || (mode != HPDR_LINF && mode != HPDR_L2 && mode != HPDR_L2_STAT) ||
        (tol_kind != HPDR_ABS && tol_kind != HPDR_REL) || !(tol > 0.0) || !std::isfinite(tol))
        return HPDR_ERR_ARG;
    if (((uintptr_t)d_in & 15) || ((uintptr_t)d_out & 15)) return HPDR_ERR_ARG;
    Plan *P;
    hpdr_status st = get_plan(ctx, ndim, dims, dtype == HPDR_F64, &P);
    if (st != HPDR_OK) return st;
    size_t unused = 0;
    if (dtype == HPDR_F32)
        return compress_t<float>(ctx, P, (const float *)d_in, ndim, dims, tol, tol_kind, mode, D, K,
                                 (uint8_t *)d_out, out_capacity, &unused, s, h_size_status, d_pair);
    return compress_t<double>(ctx, P, (const double *)d_in, ndim, dims, tol, tol_kind, mode, D, K,
                              (uint8_t *)d_out, out_capacity, &unused, s, h_size_status, d_pair);
}
}  // namespace hpdr

extern "C" {

hpdr_status hpdr_ctx_create(hpdr_ctx **ctx, int device)
{
    if (!ctx) return HPDR_ERR_ARG;
    *ctx = nullptr;
    int n = 0;
    if (cudaGetDeviceCount(&n) != cudaSuccess) { cudaGetLastError(); return HPDR_ERR_CUDA; }
    if (device < 0 || device >= n) return HPDR_ERR_ARG;
    hpdr_ctx *c = new (std::nothrow) hpdr_ctx();
    if (!c) return HPDR_ERR_NOMEM;
    c->device = device;
    DevGuard g(device);
    if (cudaMallocHost(&c->host_pinned, 64 * 1024) != cudaSuccess) {
        cudaGetLastError();
        delete c;
        return HPDR_ERR_CUDA;
    }
    *ctx = c;
    return HPDR_OK;
}

hpdr_status hpdr_ctx_destroy(hpdr_ctx *ctx)
{
    if (!ctx) return HPDR_ERR_ARG;
    DevGuard g(ctx->device);
    destroy_stream_res(ctx);
    if (ctx->batch_res) {
        BatchRes *r = (BatchRes *)ctx->batch_res;
        for (auto &kv : r->plans) free_batch_plan(kv.second);
        for (auto st : r->workers) cudaStreamDestroy(st);
        for (auto ev : r->join) cudaEventDestroy(ev);
        if (r->fork) cudaEventDestroy(r->fork);
        if (r->origin) cudaStreamDestroy(r->origin);
        delete r;
    }
    for (auto &kv : ctx->plans) { cudaFree(kv.second->tables); delete kv.second; }
    if (ctx->ws.base) cudaFree(ctx->ws.base);
    if (ctx->host_pinned) cudaFreeHost(ctx->host_pinned);
    delete ctx;
    return HPDR_OK;
}

size_t hpdr_compress_bound(int ndim, const size_t *dims, hpdr_dtype dtype, const hpdr_config *cfg)
{
    unsigned D, K;
    if (!dims || ndim < 1 || ndim > 3 || !valid_cfg(cfg, D, K)) return 0;
    if (dtype != HPDR_F32 && dtype != HPDR_F64) return 0;
    for (int k = 0; k < ndim; k++) if (dims[k] < 2 || dims[k] > (1u << 30)) return 0;
    int L = levels_of(ndim, dims);
    unsigned long long N = (unsigned long long)total_of(ndim, dims);
    K = chunk_of(K, N);
    // a Huffman code is never longer in total than the fixed-length code of
    // ceil(log2 D) bits per symbol; an escape payload takes at most 32 bits
    // while |k| < 2^31
    unsigned bpsym = 1;
    while ((1ULL << bpsym) < D) bpsym++;
    // room for node coordinates (sum of dims doubles) whether given or not
    unsigned long long nco = 0;
    for (int k = 0; k < ndim; k++) nco += dims[k];
    unsigned long long b = a16(128 + 8ULL * (L + 1) + 8 * nco);
    b = a16(b + D);
    b = a16(b + 8 * ((N + K - 1) / K));
    b += 4 * (((bpsym + 32ULL) * N + 31) / 32);
    return (size_t)b;
}

hpdr_status hpdr_compress(hpdr_ctx *ctx, const void *d_in, hpdr_dtype dtype, int ndim,
                          const size_t *dims, double tol, hpdr_tol_kind tol_kind, hpdr_mode mode,
                          const hpdr_config *cfg, void *d_out, size_t out_capacity,
                          size_t *out_bytes, void *stream)
{
    return hpdr_compress_coords(ctx, d_in, dtype, ndim, dims, nullptr, tol, tol_kind, mode, cfg, d_out,
                                out_capacity, out_bytes, stream);
}

hpdr_status hpdr_compress_coords(hpdr_ctx *ctx, const void *d_in, hpdr_dtype dtype, int ndim,
                                 const size_t *dims, const double *coords, double tol, hpdr_tol_kind tol_kind,
                                 hpdr_mode mode, const hpdr_config *cfg, void *d_out, size_t out_capacity,
                                 size_t *out_bytes, void *stream)
{
    unsigned D, K;
    if (!ctx || !d_in || !d_out || !out_bytes || !valid_cfg(cfg, D, K)) return HPDR_ERR_ARG;
    if ((dtype != HPDR_F32 && dtype != HPDR_F64) || (mode != HPDR_LINF && mode != HPDR_L2 && mode != HPDR_L2_STAT) ||
        (tol_kind != HPDR_ABS && tol_kind != HPDR_REL) || !(tol > 0.0) || !std::isfinite(tol))
        return HPDR_ERR_ARG;
    if (((uintptr_t)d_in & 15) || ((uintptr_t)d_out & 15)) return HPDR_ERR_ARG;
    DevGuard g(ctx->device);
    Plan *P;
    hpdr_status st = get_plan(ctx, ndim, dims, dtype == HPDR_F64, &P, coords);
    if (st != HPDR_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    if (dtype == HPDR_F32)
        return compress_t<float>(ctx, P, (const float *)d_in, ndim, dims, tol, tol_kind, mode, D, K,
                                 (uint8_t *)d_out, out_capacity, out_bytes, s);
    return compress_t<double>(ctx, P, (const double *)d_in, ndim, dims, tol, tol_kind, mode, D, K,
                              (uint8_t *)d_out, out_capacity, out_bytes, s);
}

hpdr_status hpdr_inspect(const void *in, size_t in_bytes, hpdr_dtype *dtype, int *ndim, size_t *dims)
{
    if (!in || !dtype || !ndim || !dims) return HPDR_ERR_ARG;
    // the fixed header and the bin widths q[0..L]: the checks of hpdr_decompress
    uint8_t hb[128 + 8 * (kMaxLevels + 1)];
    if (in_bytes < 128) return HPDR_ERR_FORMAT;
    const size_t rd = in_bytes < sizeof(hb) ? in_bytes : sizeof(hb);
    if (is_device_ptr(in)) {
        if (cudaMemcpy(hb, in, rd, cudaMemcpyDeviceToHost) != cudaSuccess) return HPDR_ERR_CUDA;
    } else {
        memcpy(hb, in, rd);
    }
    Hdr h;
    hpdr_status st = parse_header(hb, rd, in_bytes, &h);
    if (st != HPDR_OK) return st;
    if (rd < 128 + 8ULL * (h.L + 1)) return HPDR_ERR_FORMAT;
    *dtype = (hpdr_dtype)h.dtype;
    *ndim = h.ndim;
    for (int k = 0; k < 3; k++) dims[k] = k < h.ndim ? h.dims[k] : 1;
    return HPDR_OK;
}

hpdr_status hpdr_decompress(hpdr_ctx *ctx, const void *d_in, size_t in_bytes, void *d_out,
                            size_t out_capacity, void *stream)
{
    if (!ctx || !d_in || !d_out) return HPDR_ERR_ARG;
    DevGuard g(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    uint8_t *hb = (uint8_t *)ctx->host_pinned + 32 * 1024;
    size_t hdr_bytes = 128 + 8 * (kMaxLevels + 1);
    size_t rd = in_bytes < hdr_bytes ? in_bytes : hdr_bytes;
    if (in_bytes < 128) return HPDR_ERR_FORMAT;
    CK(cudaMemcpyAsync(hb, d_in, rd, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    Hdr h;
    hpdr_status st = parse_header(hb, rd, in_bytes, &h);
    if (st != HPDR_OK) return st;
    if (rd < 128 + 8ULL * (h.L + 1)) return HPDR_ERR_FORMAT;
    size_t esz = h.dtype == 0 ? 4 : 8;
    if (out_capacity < h.N * esz) return HPDR_ERR_CAPACITY;
    std::vector<double> co;
    if (h.ncoord) {
        // the coordinate section follows q; its size is bounded by the
        // container size that parse_header checked
        const size_t cb = 128 + 8 * (h.L + 1 + h.ncoord);
        std::vector<uint8_t> full(cb);
        CK(cudaMemcpy(full.data(), d_in, cb, cudaMemcpyDeviceToHost));
        read_coords(full.data(), h, co);
    }
    Plan *P;
    st = get_plan(ctx, h.ndim, h.dims, h.dtype == 1, &P, co.empty() ? nullptr : co.data());
    if (st != HPDR_OK) return st;
    if (h.dtype == 0) return decompress_t<float>(ctx, P, h, (const uint8_t *)d_in, (float *)d_out, s);
    return decompress_t<double>(ctx, P, h, (const uint8_t *)d_in, (double *)d_out, s);
}

hpdr_status hpdr_compress_async(hpdr_ctx *ctx, const void *d_in, hpdr_dtype dtype, int ndim, const size_t *dims,
                                double tol, hpdr_tol_kind tol_kind, hpdr_mode mode, const hpdr_config *cfg,
                                void *d_out, size_t out_capacity, uint64_t *d_result, void *stream)
{
    unsigned D, K;
    if (!ctx || !d_in || !d_out || !d_result || !dims || !valid_cfg(cfg, D, K)) return HPDR_ERR_ARG;
    if ((dtype != HPDR_F32 && dtype != HPDR_F64) || (mode != HPDR_LINF && mode != HPDR_L2 && mode != HPDR_L2_STAT) ||
        (tol_kind != HPDR_ABS && tol_kind != HPDR_REL) || !(tol > 0.0) || !std::isfinite(tol))
        return HPDR_ERR_ARG;
    if (((uintptr_t)d_in & 15) || ((uintptr_t)d_out & 15) || ((uintptr_t)d_result & 7)) return HPDR_ERR_ARG;
    DevGuard g(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    Plan *P;
    hpdr_status st = get_plan(ctx, ndim, dims, dtype == HPDR_F64, &P);
    if (st != HPDR_OK) return st;
    K = chunk_of(K, (unsigned long long)P->N[P->L]);
    Ws w;
    size_t need = carve_ws(nullptr, P, dtype == HPDR_F64 ? 8 : 4, D, K, true, &w);
    st = ensure_workspace(ctx, need);
    if (st != HPDR_OK) return st;
    carve_ws(ctx->ws.base, P, dtype == HPDR_F64 ? 8 : 4, D, K, true, &w);
    if (dtype == HPDR_F32)
        st = compress_core<float>(ctx, P, (const float *)d_in, ndim, dims, tol, tol_kind, mode, D, K,
                                  (uint8_t *)d_out, out_capacity, w, s, kPhAll, (unsigned long long *)d_result);
    else
        st = compress_core<double>(ctx, P, (const double *)d_in, ndim, dims, tol, tol_kind, mode, D, K,
                                   (uint8_t *)d_out, out_capacity, w, s, kPhAll, (unsigned long long *)d_result);
    return st;
}

hpdr_status hpdr_device_status(uint64_t code) { return map_device_status((unsigned)code); }

hpdr_status hpdr_decompress_async(hpdr_ctx *ctx, const void *d_in, size_t in_capacity, hpdr_dtype dtype, int ndim,
                                  const size_t *dims, const hpdr_config *cfg, void *d_out, size_t out_capacity,
                                  uint64_t *d_result, void *stream)
{
    unsigned D, K;
    if (!ctx || !d_in || !d_out || !d_result || !dims || !valid_cfg(cfg, D, K)) return HPDR_ERR_ARG;
    if ((dtype != HPDR_F32 && dtype != HPDR_F64) || ((uintptr_t)d_in & 15) || ((uintptr_t)d_result & 7))
        return HPDR_ERR_ARG;
    DevGuard g(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    Plan *P;
    hpdr_status st = get_plan(ctx, ndim, dims, dtype == HPDR_F64, &P);
    if (st != HPDR_OK) return st;
    const size_t esz = dtype == HPDR_F64 ? 8 : 4;
    if (out_capacity < (size_t)P->N[P->L] * esz) return HPDR_ERR_CAPACITY;
    if (dtype == HPDR_F32)
        return decompress_dev<float>(ctx, P, 0, ndim, dims, D, K, (const uint8_t *)d_in, in_capacity, (float *)d_out,
                                     (unsigned long long *)d_result, s);
    return decompress_dev<double>(ctx, P, 1, ndim, dims, D, K, (const uint8_t *)d_in, in_capacity, (double *)d_out,
                                  (unsigned long long *)d_result, s);
}

hpdr_status hpdr_decompose(hpdr_ctx *ctx, const void *d_u, void *d_coef, hpdr_dtype dtype,
                           int ndim, const size_t *dims, void *stream)
{
    return hpdr_decompose_coords(ctx, d_u, d_coef, dtype, ndim, dims, nullptr, stream);
}

hpdr_status hpdr_decompose_coords(hpdr_ctx *ctx, const void *d_u, void *d_coef, hpdr_dtype dtype,
                                  int ndim, const size_t *dims, const double *coords, void *stream)
{
    if (!ctx || !d_u || !d_coef || (dtype != HPDR_F32 && dtype != HPDR_F64)) return HPDR_ERR_ARG;
    if ((uintptr_t)d_u & 15) return HPDR_ERR_ARG;
    DevGuard g(ctx->device);
    Plan *P;
    hpdr_status st = get_plan(ctx, ndim, dims, dtype == HPDR_F64, &P, coords);
    if (st != HPDR_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    if (dtype == HPDR_F32) return decompose_t<float>(ctx, P, (const float *)d_u, (float *)d_coef, s);
    return decompose_t<double>(ctx, P, (const double *)d_u, (double *)d_coef, s);
}

hpdr_status hpdr_recompose(hpdr_ctx *ctx, const void *d_coef, void *d_u, hpdr_dtype dtype,
                           int ndim, const size_t *dims, void *stream)
{
    return hpdr_recompose_coords(ctx, d_coef, d_u, dtype, ndim, dims, nullptr, stream);
}

hpdr_status hpdr_recompose_coords(hpdr_ctx *ctx, const void *d_coef, void *d_u, hpdr_dtype dtype,
                                  int ndim, const size_t *dims, const double *coords, void *stream)
{
    if (!ctx || !d_u || !d_coef || (dtype != HPDR_F32 && dtype != HPDR_F64)) return HPDR_ERR_ARG;
    DevGuard g(ctx->device);
    Plan *P;
    hpdr_status st = get_plan(ctx, ndim, dims, dtype == HPDR_F64, &P, coords);
    if (st != HPDR_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    if (dtype == HPDR_F32) return recompose_t<float>(ctx, P, (const float *)d_coef, (float *)d_u, s);
    return recompose_t<double>(ctx, P, (const double *)d_coef, (double *)d_u, s);
}

hpdr_status hpdr_huffman_encode(hpdr_ctx *ctx, const uint16_t *d_symbols, uint64_t N, uint32_t D,
                                uint32_t K, uint8_t *d_lengths, uint64_t *d_chunk_bits,
                                uint32_t *d_words, uint64_t words_capacity, uint64_t *total_bits,
                                void *stream)
{
    hpdr_config cfg = {D, K};
    unsigned Dv, Kv;
    if (!ctx || !d_symbols || !d_lengths || !d_chunk_bits || !d_words || !total_bits || N == 0 || K == 0 ||
        !valid_cfg(&cfg, Dv, Kv) || ((uintptr_t)d_symbols & 15))
        return HPDR_ERR_ARG;
    DevGuard g(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    unsigned long long nch = (N + K - 1) / K;
    Carver c(nullptr);
    c.take<Scalars>(1); c.take<unsigned long long>(D); c.take<unsigned long long>(nch + 2);
    c.take<unsigned long long>(1024);
    c.take<char>(huff_scratch_bytes(D));
    hpdr_status st = ensure_workspace(ctx, c.used + 256);
    if (st != HPDR_OK) return st;
    Carver w(ctx->ws.base);
    Scalars *sc = w.take<Scalars>(1);
    unsigned long long *hist = w.take<unsigned long long>(D);
    unsigned long long *cb = w.take<unsigned long long>(nch + 2);
    unsigned long long *bs = w.take<unsigned long long>(1024);
    void *hb = w.take<char>(huff_scratch_bytes(D));
    CK(cudaMemsetAsync(sc, 0, sizeof(Scalars), s));
    CK(cudaMemsetAsync(hist, 0, 8ULL * D, s));
    CK(launch_histogram(d_symbols, N, D, hist, &sc->status, s));
    HuffScratch hs;
    huff_scratch_carve(hb, D, sc, &hs);
    CK(launch_codebook(hist, D, hs, s));
    EncodeArgs ea;
    memset(&ea, 0, sizeof(ea));
    ea.sym = d_symbols; ea.N = N; ea.D = D; ea.K = K; ea.len = hs.len; ea.code = hs.code; ea.pack = hs.pack;
    ea.chunk_bits = cb; ea.sc = sc; ea.bsum = bs;
    ea.chunk_out = (unsigned long long *)d_chunk_bits;
    ea.words_out = d_words;
    ea.words_cap = words_capacity;
    CK(launch_encode(ea, s));
    CK(cudaMemcpyAsync(d_lengths, hs.len, D, cudaMemcpyDeviceToDevice, s));
    Scalars *hsc = (Scalars *)ctx->host_pinned;
    CK(cudaMemcpyAsync(hsc, sc, sizeof(Scalars), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (hsc->status) return map_device_status(hsc->status);
    *total_bits = hsc->total_bits;
    return HPDR_OK;
}

size_t hpdr_lossless_bound(uint64_t n, int key_bytes, uint32_t K)
{
    if (n == 0 || (key_bytes != 1 && key_bytes != 2)) return 0;
    LosslessHdr h;
    h.key_bytes = (unsigned)key_bytes;
    h.D = key_bytes == 1 ? 256u : 65536u;
    hpdr_config cfg = {h.D, K};
    unsigned Dv, Kv;
    if (!valid_cfg(&cfg, Dv, Kv)) return 0;
    h.K = chunk_of(Kv, n);
    h.n = n;
    h.bits = n * 8ull * (unsigned)key_bytes;   // never above the fixed-length code
    lossless_layout(&h);
    return (size_t)h.total;
}

hpdr_status hpdr_lossless_compress(hpdr_ctx *ctx, const void *d_keys, uint64_t n, int key_bytes, uint32_t K,
                                   void *d_out, size_t out_capacity, size_t *out_bytes, void *stream)
{
    if (!ctx || !d_keys || !d_out || !out_bytes || n == 0 || (key_bytes != 1 && key_bytes != 2)) return HPDR_ERR_ARG;
    LosslessHdr h;
    h.key_bytes = (unsigned)key_bytes;
    h.D = key_bytes == 1 ? 256u : 65536u;
    hpdr_config cfg = {h.D, K};
    unsigned Dv, Kv;
    if (!valid_cfg(&cfg, Dv, Kv) || ((uintptr_t)d_out & 15) || (key_bytes == 2 && ((uintptr_t)d_keys & 15)))
        return HPDR_ERR_ARG;
    h.K = chunk_of(Kv, n);
    h.n = n;
    h.bits = 0;
    lossless_layout(&h);
    if (h.off_bits > out_capacity) return HPDR_ERR_CAPACITY;
    DevGuard g(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    const unsigned D = h.D;
    // byte keys are counted and encoded where they are; a pointer that does not
    // start on 16 bytes has them widened in the workspace first
    const bool bytes = key_bytes == 1 && ((uintptr_t)d_keys & 15) == 0, widen = key_bytes == 1 && !bytes;
    Carver c(nullptr);
    const auto carve = [&](Carver &w, Scalars *&sc, unsigned long long *&hist, unsigned long long *&cb,
                           unsigned long long *&bs, void *&hb, uint16_t *&wide) {
        sc = w.take<Scalars>(1);
        hist = w.take<unsigned long long>(D);
        cb = w.take<unsigned long long>(h.nch + 2);
        bs = w.take<unsigned long long>(1024);
        hb = w.take<char>(huff_scratch_bytes(D));
        wide = widen ? w.take<uint16_t>(n + 8) : nullptr;
    };
    Scalars *sc;
    unsigned long long *hist, *cb, *bs;
    void *hb;
    uint16_t *wide;
    carve(c, sc, hist, cb, bs, hb, wide);
    hpdr_status st = ensure_workspace(ctx, c.used + 256);
    if (st != HPDR_OK) return st;
    Carver w(ctx->ws.base);
    carve(w, sc, hist, cb, bs, hb, wide);
    if (widen) {
        widen_keys_kernel<<<152 * 8, 256, 0, s>>>((const uint8_t *)d_keys, n, wide);
        count_launch();
        CK(cudaGetLastError());
    }
    uint8_t *out = (uint8_t *)d_out;
    // the scalars and the histogram are neighbours in the workspace
    CK(cudaMemsetAsync(sc, 0, (size_t)((char *)(hist + D) - (char *)sc), s));
    if (bytes) CK(launch_histogram_bytes((const uint8_t *)d_keys, n, hist, s));
    else CK(launch_histogram(widen ? wide : (const uint16_t *)d_keys, n, D, hist, &sc->status, s));
    HuffScratch hs;
    huff_scratch_carve(hb, D, sc, &hs);
    CK(launch_codebook(hist, D, hs, s));
    EncodeArgs ea;
    memset(&ea, 0, sizeof(ea));
    ea.sym = widen ? wide : d_keys; ea.bytes = bytes;
    ea.N = n; ea.D = D; ea.K = h.K; ea.len = hs.len; ea.code = hs.code; ea.pack = hs.pack;
    ea.chunk_bits = cb; ea.sc = sc; ea.bsum = bs;
    ea.chunk_out = (unsigned long long *)(out + h.off_chunk);
    ea.words_out = (uint32_t *)(out + h.off_bits);
    ea.words_cap = (out_capacity - h.off_bits) / 4;
    CK(launch_encode(ea, s));
    LosslessHeader lh = {h.key_bytes, h.D, h.K, h.n, h.nch, h.off_chunk, h.off_bits};
    CK(launch_lossless_header(lh, hs.len, sc, out, s));
    Scalars *hsc = (Scalars *)ctx->host_pinned;
    CK(cudaMemcpyAsync(hsc, sc, sizeof(Scalars), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (hsc->status) return map_device_status(hsc->status);
    h.bits = hsc->total_bits;
    lossless_layout(&h);
    *out_bytes = (size_t)h.total;
    return HPDR_OK;
}

hpdr_status hpdr_lossless_decompress(hpdr_ctx *ctx, const void *d_in, size_t in_bytes, void *d_keys,
                                     size_t keys_capacity, void *stream)
{
    if (!ctx || !d_in || !d_keys || ((uintptr_t)d_in & 15)) return HPDR_ERR_ARG;
    if (in_bytes < kLosslessHdr) return HPDR_ERR_FORMAT;
    DevGuard g(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    uint8_t *hb = (uint8_t *)ctx->host_pinned + 48 * 1024;
    CK(cudaMemcpyAsync(hb, d_in, kLosslessHdr, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    LosslessHdr h;
    hpdr_status st = parse_lossless(hb, in_bytes, &h);
    if (st != HPDR_OK) return st;
    if (h.n * h.key_bytes > keys_capacity) return HPDR_ERR_CAPACITY;
    if (h.key_bytes == 2 && ((uintptr_t)d_keys & 15)) return HPDR_ERR_ARG;
    const unsigned D = h.D;
    Carver c(nullptr);
    // bytes are decoded in place; a pointer that does not start on 8 bytes takes
    // them from 16-bit symbols in the workspace
    const bool bytes = h.key_bytes == 1 && ((uintptr_t)d_keys & 7) == 0, narrow = h.key_bytes == 1 && !bytes;
    c.take<Scalars>(1); c.take<char>(huff_scratch_bytes(D));
    if (narrow) c.take<uint16_t>(h.n + 8);
    st = ensure_workspace(ctx, c.used + 256);
    if (st != HPDR_OK) return st;
    Carver w(ctx->ws.base);
    Scalars *sc = w.take<Scalars>(1);
    void *hsb = w.take<char>(huff_scratch_bytes(D));
    uint16_t *wide = narrow ? w.take<uint16_t>(h.n + 8) : nullptr;
    const uint8_t *in = (const uint8_t *)d_in;
    CK(cudaMemsetAsync(sc, 0, sizeof(Scalars), s));
    HuffScratch hs;
    huff_scratch_carve(hsb, D, sc, &hs);
    TabArgs ta;
    ta.lenb = in + kLosslessHdr; ta.s_hi = D - 1; ta.D = D;
    CK(launch_decode_tables(ta, hs, s));
    DecodeArgs da;
    da.words = (const uint32_t *)(in + h.off_bits);
    da.nwords = (h.bits + 31) / 32;
    da.chunk = (const unsigned long long *)(in + h.off_chunk);
    da.N = h.n; da.K = h.K; da.sym = narrow ? wide : d_keys; da.bytes = bytes; da.total_bits = h.bits; da.esc = nullptr; da.esc_w = 0;
    CK(launch_decode(da, hs, s));
    if (narrow) {
        narrow_keys_kernel<<<152 * 8, 256, 0, s>>>(wide, h.n, (uint8_t *)d_keys);
        count_launch();
        CK(cudaGetLastError());
    }
    Scalars *hsc = (Scalars *)ctx->host_pinned;
    CK(cudaMemcpyAsync(hsc, sc, sizeof(Scalars), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (hsc->status) return map_device_status(hsc->status);
    return HPDR_OK;
}

hpdr_status hpdr_lossless_inspect(const void *in, size_t in_bytes, int *key_bytes, uint64_t *n)
{
    if (!in || !key_bytes || !n) return HPDR_ERR_ARG;
    if (in_bytes < kLosslessHdr) return HPDR_ERR_FORMAT;
    uint8_t hb[kLosslessHdr];
    if (is_device_ptr(in)) {
        if (cudaMemcpy(hb, in, kLosslessHdr, cudaMemcpyDeviceToHost) != cudaSuccess) return HPDR_ERR_CUDA;
    } else {
        memcpy(hb, in, kLosslessHdr);
    }
    LosslessHdr h;
    hpdr_status st = parse_lossless(hb, in_bytes, &h);
    if (st != HPDR_OK) return st;
    *key_bytes = (int)h.key_bytes;
    *n = h.n;
    return HPDR_OK;
}

hpdr_status hpdr_huffman_decode(hpdr_ctx *ctx, const uint32_t *d_words, uint64_t total_bits,
                                const uint64_t *d_chunk_bits, uint64_t N, uint32_t D, uint32_t K,
                                const uint8_t *d_lengths, uint16_t *d_symbols, void *stream)
{
    hpdr_config cfg = {D, K};
    unsigned Dv, Kv;
    if (!ctx || !d_words || !d_chunk_bits || !d_lengths || !d_symbols || N == 0 || K == 0 ||
        !valid_cfg(&cfg, Dv, Kv) || ((uintptr_t)d_symbols & 15))
        return HPDR_ERR_ARG;
    DevGuard g(ctx->device);
    cudaStream_t s = (cudaStream_t)stream;
    Carver c(nullptr);
    c.take<Scalars>(1); c.take<char>(huff_scratch_bytes(D));
    hpdr_status st = ensure_workspace(ctx, c.used + 256);
    if (st != HPDR_OK) return st;
    Carver w(ctx->ws.base);
    Scalars *sc = w.take<Scalars>(1);
    void *hb = w.take<char>(huff_scratch_bytes(D));
    CK(cudaMemsetAsync(sc, 0, sizeof(Scalars), s));
    HuffScratch hs;
    huff_scratch_carve(hb, D, sc, &hs);
    TabArgs ta;
    ta.lenb = d_lengths; ta.s_hi = D - 1; ta.D = D;
    CK(launch_decode_tables(ta, hs, s));
    DecodeArgs da;
    da.words = d_words; da.nwords = (total_bits + 31) / 32;
    da.chunk = (const unsigned long long *)d_chunk_bits;
    da.N = N; da.K = K; da.sym = d_symbols; da.total_bits = total_bits; da.esc = nullptr; da.esc_w = 0;
    Scalars *hsc = (Scalars *)ctx->host_pinned;
    CK(launch_decode(da, hs, s));
    CK(cudaMemcpyAsync(hsc, sc, sizeof(Scalars), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (hsc->status) return map_device_status(hsc->status);
    return HPDR_OK;
}

hpdr_status hpdr_recompose_adjoint(hpdr_ctx *ctx, const void *d_grad_u, void *d_grad_coef,
                                   hpdr_dtype dtype, int ndim, const size_t *dims, void *stream)
{
    return hpdr_recompose_adjoint_coords(ctx, d_grad_u, d_grad_coef, dtype, ndim, dims, nullptr, stream);
}

hpdr_status hpdr_recompose_adjoint_coords(hpdr_ctx *ctx, const void *d_grad_u, void *d_grad_coef, hpdr_dtype dtype,
                                          int ndim, const size_t *dims, const double *coords, void *stream)
{
    if (!ctx || !d_grad_u || !d_grad_coef || (dtype != HPDR_F32 && dtype != HPDR_F64)) return HPDR_ERR_ARG;
    DevGuard g(ctx->device);
    Plan *P;
    hpdr_status st = get_plan(ctx, ndim, dims, dtype == HPDR_F64, &P, coords);
    if (st != HPDR_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    if (dtype == HPDR_F32)
        return adjoint_t<float>(ctx, P, (const float *)d_grad_u, (float *)d_grad_coef, true, s);
    return adjoint_t<double>(ctx, P, (const double *)d_grad_u, (double *)d_grad_coef, true, s);
}

hpdr_status hpdr_decompose_adjoint(hpdr_ctx *ctx, const void *d_grad_coef, void *d_grad_u,
                                   hpdr_dtype dtype, int ndim, const size_t *dims, void *stream)
{
    return hpdr_decompose_adjoint_coords(ctx, d_grad_coef, d_grad_u, dtype, ndim, dims, nullptr, stream);
}

hpdr_status hpdr_decompose_adjoint_coords(hpdr_ctx *ctx, const void *d_grad_coef, void *d_grad_u, hpdr_dtype dtype,
                                          int ndim, const size_t *dims, const double *coords, void *stream)
{
    if (!ctx || !d_grad_u || !d_grad_coef || (dtype != HPDR_F32 && dtype != HPDR_F64)) return HPDR_ERR_ARG;
    DevGuard g(ctx->device);
    Plan *P;
    hpdr_status st = get_plan(ctx, ndim, dims, dtype == HPDR_F64, &P, coords);
    if (st != HPDR_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    if (dtype == HPDR_F32)
        return adjoint_t<float>(ctx, P, (const float *)d_grad_coef, (float *)d_grad_u, false, s);
    return adjoint_t<double>(ctx, P, (const double *)d_grad_coef, (double *)d_grad_u, false, s);
}

hpdr_status hpdr_profile_enable(hpdr_ctx *ctx, int on)
{
    if (!ctx) return HPDR_ERR_ARG;
    DevGuard g(ctx->device);
    if (on && ctx->prof_pool.empty()) {
        ctx->prof_pool.resize(65536);
        for (auto &e : ctx->prof_pool)
            if (cudaEventCreate(&e) != cudaSuccess) return HPDR_ERR_CUDA;
    }
    ctx->prof_on = on != 0;
    return HPDR_OK;
}

int hpdr_profile_read(hpdr_ctx *ctx, const char **names, double *ms, long long *count, int cap)
{
    if (!ctx) return -1;
    DevGuard g(ctx->device);
    for (auto &r : ctx->prof_recs) {
        float t = 0.f;
        if (cudaEventSynchronize(r.b) == cudaSuccess && cudaEventElapsedTime(&t, r.a, r.b) == cudaSuccess) {
            ctx->prof_ms[r.id] += t;
            ctx->prof_cnt[r.id] += 1;
        } else {
            cudaGetLastError();
        }
    }
    ctx->prof_recs.clear();
    ctx->prof_used = 0;
    int n = (int)ctx->prof_names.size();
    for (int i = 0; i < n && i < cap; i++) {
        if (names) names[i] = ctx->prof_names[i].c_str();
        if (ms) ms[i] = ctx->prof_ms[i];
        if (count) count[i] = ctx->prof_cnt[i];
    }
    for (int i = 0; i < n; i++) { ctx->prof_ms[i] = 0.0; ctx->prof_cnt[i] = 0; }
    return n;
}

unsigned long long hpdr_launch_count(void) { return g_launches; }

int hpdr_debug_set_wait_limit(int polls)
{
    const int prev = g_wait_limit;
    if (polls >= 0) g_wait_limit = polls;
    return prev;
}

hpdr_status hpdr_compress_batched(hpdr_ctx *ctx, int nfields, const hpdr_field *fields, const hpdr_config *cfg,
                                  void *d_out, size_t out_capacity, size_t *out_offsets, size_t *out_sizes,
                                  void *stream)
{
    unsigned D, K;
    if (!ctx || nfields < 1 || !fields || !d_out || !out_offsets || !out_sizes || !valid_cfg(cfg, D, K))
        return HPDR_ERR_ARG;
    if ((uintptr_t)d_out & 15) return HPDR_ERR_ARG;
    DevGuard g(ctx->device);
    // key: everything the captured graph depends on
    std::string key = std::to_string(nfields) + "|" + std::to_string(D) + "|" + std::to_string(K) + "|" +
                      std::to_string((uintptr_t)d_out);
    size_t off = 0;
    for (int i = 0; i < nfields; i++) {
        const hpdr_field &f = fields[i];
        if (!f.d_in || ((uintptr_t)f.d_in & 15) || (f.dtype != HPDR_F32 && f.dtype != HPDR_F64) ||
            (f.mode != HPDR_LINF && f.mode != HPDR_L2 && f.mode != HPDR_L2_STAT) || (f.tol_kind != HPDR_ABS && f.tol_kind != HPDR_REL) ||
            !(f.tol > 0.0) || !std::isfinite(f.tol))
            return HPDR_ERR_ARG;
        const size_t b = hpdr_compress_bound(f.ndim, f.dims, f.dtype, cfg);
        if (!b) return HPDR_ERR_ARG;
        out_offsets[i] = off;
        off = (off + b + 255) & ~size_t(255);
        char buf[160];
        snprintf(buf, sizeof(buf), "|%p,%d,%d,%zu,%zu,%zu,%.17g,%d,%d", f.d_in, (int)f.dtype, f.ndim, f.dims[0],
                 f.ndim > 1 ? f.dims[1] : 1, f.ndim > 2 ? f.dims[2] : 1, f.tol, (int)f.tol_kind, (int)f.mode);
        key += buf;
    }
    out_offsets[nfields] = off;
    if (off > out_capacity) return HPDR_ERR_CAPACITY;
    BatchRes *r = nullptr;
    hpdr_status st = batch_res(ctx, r, 16);
    if (st != HPDR_OK) return st;
    cudaStream_t user = (cudaStream_t)stream;
    BatchPlan *bp;
    auto it = r->plans.find(key);
    if (it != r->plans.end()) {
        bp = it->second;
    } else {
        bp = new BatchPlan();
        bp->nfields = nfields;
        bp->plans.resize(nfields);
        bp->ws_off.resize(nfields);
        bp->out_off.resize(nfields);
        bp->bound.resize(nfields);
        size_t wsz = 0;
        for (int i = 0; i < nfields; i++) {
            const hpdr_field &f = fields[i];
            st = get_plan(ctx, f.ndim, f.dims, f.dtype == HPDR_F64, &bp->plans[i]);
            if (st != HPDR_OK) { delete bp; return st; }
            Ws w;
            const unsigned Ki = chunk_of(K, (unsigned long long)bp->plans[i]->N[bp->plans[i]->L]);
            const size_t need = carve_ws(nullptr, bp->plans[i], f.dtype == HPDR_F64 ? 8 : 4, D, Ki, true, &w);
            bp->ws_off[i] = wsz;
            wsz = (wsz + need + 255) & ~size_t(255);
            bp->out_off[i] = out_offsets[i];
            bp->bound[i] = out_offsets[i + 1 <= nfields ? i + 1 : i] - out_offsets[i];
        }
        bp->ws_total = wsz;
        if (cudaMalloc(&bp->ws, wsz) != cudaSuccess || cudaMalloc(&bp->sizes, 16ull * nfields) != cudaSuccess) {
            cudaGetLastError();
            free_batch_plan(bp);
            return HPDR_ERR_NOMEM;
        }
        st = build_batch_jobs(bp, fields, D, K, (uint8_t *)d_out);
        if (st != HPDR_OK) {
            free_batch_plan(bp);
            return st;
        }
        // one eager run (sets kernel attributes, warms the plans), then the
        // autotuner: capture the batch for every stream count and keep the fastest replay
        const bool prof = ctx->prof_on;
        ctx->prof_on = false;
        st = enqueue_batch(ctx, r, bp, fields, D, K, (uint8_t *)d_out, 1);
        if (st == HPDR_OK && cudaStreamSynchronize(r->origin) != cudaSuccess) st = HPDR_ERR_CUDA;
        cudaEvent_t t0, t1;
        cudaEventCreate(&t0);
        cudaEventCreate(&t1);
        const int cand[5] = {1, 2, 4, 8, 16};
        for (int ci = 0; ci < 5 && st == HPDR_OK; ci++) {
            const int ns = cand[ci];
            if (ns > nfields && ns > 1) break;
            cudaGraphExec_t ex = nullptr;
            st = capture_batch(ctx, r, bp, fields, D, K, (uint8_t *)d_out, ns, &ex);
            if (st != HPDR_OK) break;
            cudaGraphLaunch(ex, r->origin);
            cudaEventRecord(t0, r->origin);
            cudaGraphLaunch(ex, r->origin);
            cudaEventRecord(t1, r->origin);
            if (cudaEventSynchronize(t1) != cudaSuccess) { st = HPDR_ERR_CUDA; cudaGraphExecDestroy(ex); break; }
            float ms = 0.f;
            cudaEventElapsedTime(&ms, t0, t1);
            if (!bp->exec || ms < bp->tuned_ms) {
                if (bp->exec) cudaGraphExecDestroy(bp->exec);
                bp->exec = ex;
                bp->streams = ns;
                bp->tuned_ms = ms;
            } else {
                cudaGraphExecDestroy(ex);
            }
        }
        cudaEventDestroy(t0);
        cudaEventDestroy(t1);
        ctx->prof_on = prof;
        if (st != HPDR_OK) {
            free_batch_plan(bp);
            return st;
        }
        // every earlier replay has completed (each call waits for its sizes)
        while (r->plans.size() >= kMaxBatchPlans) {
            auto lru = r->plans.begin();
            for (auto jt = r->plans.begin(); jt != r->plans.end(); ++jt)
                if (jt->second->last_use < lru->second->last_use) lru = jt;
            free_batch_plan(lru->second);
            r->plans.erase(lru);
        }
        r->plans[key] = bp;
    }
    bp->last_use = ++r->calls;
    // replay: the caller's stream orders the graph before and after
    cudaEvent_t ev = r->fork;
    CK(cudaEventRecord(ev, user));
    CK(cudaStreamWaitEvent(r->origin, ev, 0));
    {
        ProfScope ps(ctx, "batched_graph", r->origin);
        CK(cudaGraphLaunch(bp->exec, r->origin));
    }
    count_launch();
    std::vector<unsigned long long> sizes(2 * (size_t)nfields);
    CK(cudaMemcpyAsync(sizes.data(), bp->sizes, 16ull * nfields, cudaMemcpyDeviceToHost, r->origin));
    CK(cudaStreamSynchronize(r->origin));
    for (int i = 0; i < nfields; i++) {
        if (sizes[2 * i + 1]) return map_device_status((unsigned)sizes[2 * i + 1]);
        out_sizes[i] = (size_t)sizes[2 * i];
    }
    return HPDR_OK;
}

int hpdr_batched_streams(hpdr_ctx *ctx)
{
    if (!ctx || !ctx->batch_res) return 0;
    BatchRes *r = (BatchRes *)ctx->batch_res;
    // the stream count of the most recently replayed batch
    int s = 0;
    unsigned long long last = 0;
    for (auto &kv : r->plans)
        if (kv.second->last_use >= last) { last = kv.second->last_use; s = kv.second->streams; }
    return s;
}

int hpdr_batched_cached(hpdr_ctx *ctx)
{
    if (!ctx || !ctx->batch_res) return 0;
    return (int)((BatchRes *)ctx->batch_res)->plans.size();
}

const char *hpdr_status_string(hpdr_status st)
{
    switch (st) {
    case HPDR_OK: return "ok";
    case HPDR_ERR_ARG: return "invalid argument";
    case HPDR_ERR_CUDA: return "CUDA error";
    case HPDR_ERR_CAPACITY: return "output buffer too small";
    case HPDR_ERR_FORMAT: return "malformed container";
    case HPDR_ERR_TIMEOUT: return "device wait timed out";
    case HPDR_ERR_NOMEM: return "device allocation failed";
    default: return "unknown status";
    }
}

}  // extern "C"
