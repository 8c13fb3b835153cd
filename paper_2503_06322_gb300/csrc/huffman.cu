// huffman.cu -- Huffman stage of Sec. IV-B (Alg. 2) for sm_103a: SortByKey of
// the frequencies, filter of zero frequencies, code lengths (tree_build),
// canonical codewords, encode + serialize, and the chunk-parallel decoder.
//
// Code lengths follow the two-queue Huffman rule (leaves sorted by
// (frequency, symbol); on equal weights a leaf is picked before a merged
// node).  It is computed here in rounds instead of one pick at a time: if w
// is the smallest weight left, every node created from now on weighs at least
// 2w, so all leaves and merged nodes of weight <= 2w are picked next, in
// merged order, before any new node; a round pairs an even number of them in
// parallel.  This yields exactly the picks of the sequential rule.
#include <cstdio>
#include "huffman.cuh"

namespace hpdr {
namespace {

constexpr int kRankBlocks = 152 * 2;
constexpr int kSmemKeys = 12288;     // keys one block stages in shared memory (96 KB)
constexpr int kSmemCodes = 16384;    // codewords staged by the encoder

__device__ __forceinline__ unsigned warp_sum(unsigned v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ unsigned long long warp_sum64(unsigned long long v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// keys (frequency << 16) | s of the present symbols, in increasing symbol order
__global__ void __launch_bounds__(1024)
compact_kernel(const unsigned long long *hist, unsigned D, unsigned long long *keys, unsigned *nsym, unsigned *s_lo,
               unsigned *s_hi)
{
    __shared__ unsigned wcnt[32], wpre[32];
    __shared__ unsigned base, lo, hi;
    const unsigned lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) { base = 0; lo = 0xFFFFFFFFu; hi = 0; }
    __syncthreads();
    for (unsigned t0 = 0; t0 < D; t0 += 1024) {
        unsigned s = t0 + threadIdx.x;
        unsigned long long f = 0;
        if (s < D) f = hist[s];
        bool p = f != 0;
        unsigned ball = __ballot_sync(0xffffffffu, p);
        if (lane == 0) wcnt[w] = __popc(ball);
        __syncthreads();
        if (w == 0) {
            unsigned v = wcnt[lane], x = v;
            for (int o = 1; o < 32; o <<= 1) {
                unsigned y = __shfl_up_sync(0xffffffffu, x, o);
                if ((int)lane >= o) x += y;
            }
            wpre[lane] = x - v;
        }
        __syncthreads();
        if (p) {
            keys[base + wpre[w] + __popc(ball & ((1u << lane) - 1))] = (f << 16) | s;
            atomicMin(&lo, s);
            atomicMax(&hi, s);
        }
        __syncthreads();
        if (threadIdx.x == 0) base += wpre[31] + wcnt[31];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        *nsym = base;
        *s_lo = base ? lo : 0;
        *s_hi = base ? hi : 0;
    }
}

// rank of every key among the n (unique) keys; scatter into sorted[] and/or rank[]
__global__ void __launch_bounds__(256)
rank_kernel(const unsigned long long *keys, const unsigned *nsym, unsigned long long *sorted,
            unsigned *rank_out)
{
    extern __shared__ unsigned long long sk[];
    const unsigned n = *nsym;
    const unsigned long long *K = keys;
    if (n <= (unsigned)kSmemKeys) {
        for (unsigned i = threadIdx.x; i < n; i += blockDim.x) sk[i] = keys[i];
        __syncthreads();
        K = sk;
    }
    const unsigned lane = threadIdx.x & 31;
    const unsigned wg = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const unsigned nw = gridDim.x * (blockDim.x >> 5);
    for (unsigned i = wg; i < n; i += nw) {
        const unsigned long long ki = K[i];
        unsigned c = 0;
        for (unsigned j = lane; j < n; j += 32) c += K[j] < ki ? 1u : 0u;
        c = warp_sum(c);
        if (lane == 0) {
            if (sorted) sorted[c] = ki;
            if (rank_out) rank_out[i] = c;
        }
    }
}

// all threads of a block take the same decision even if another block
// raises the status meanwhile
__device__ bool block_skip(const unsigned *status)
{
    __shared__ int flag;
    __syncthreads();
    if (threadIdx.x == 0) flag = *((volatile const unsigned *)status) != 0;
    __syncthreads();
    return flag != 0;
}

__device__ unsigned count_le(const unsigned long long *a, unsigned n, unsigned long long v)
{
    unsigned lo = 0, hi = n;
    while (lo < hi) { unsigned m = (lo + hi) >> 1; if (a[m] <= v) lo = m + 1; else hi = m; }
    return lo;
}
__device__ unsigned count_lt(const unsigned long long *a, unsigned n, unsigned long long v)
{
    unsigned lo = 0, hi = n;
    while (lo < hi) { unsigned m = (lo + hi) >> 1; if (a[m] < v) lo = m + 1; else hi = m; }
    return lo;
}

// canonical length tables staged in shared memory
struct LenTabs {
    unsigned long long first[64], lim[64];
    unsigned start[64], count[64];
};

// Canonical tables of every code length from the per-length counts cnt[64]
// (shared memory), by one warp; returns whether the lengths are those of a
// prefix code (the same answer in every lane).  With
// S_L = sum_{j <= L} cnt_j 2^(63 - j), the share of the code space that the
// codewords of at most L bits take (2^63 is all of it):
//   first canonical code of length L     S_{L-1} >> (63 - L)
//   left-justified limit of length <= L  2 S_L  (all ones once the space is full)
// The sums saturate just above 2^63, so an over-full set of lengths is seen
// whatever its counts; a serial recurrence over the 63 lengths took 2.5 us.
constexpr unsigned long long kFullCode = 1ULL << 63;
__device__ __forceinline__ unsigned long long sat_add(unsigned long long a, unsigned long long b)
{
    const unsigned long long c = a + b;
    return (a > kFullCode || b > kFullCode || c > kFullCode || c < a) ? kFullCode + 1 : c;
}
__device__ __forceinline__ bool length_tables(LenTabs &T, const unsigned *cnt)
{
    const unsigned lane = threadIdx.x & 31;
    unsigned long long scarry = 0;
    unsigned ncarry = 0;
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const unsigned L = lane + 32u * h;
        const unsigned c = L ? cnt[L] : 0u;
        // more codewords of L bits than the space holds: over-full
        const unsigned long long share = (unsigned long long)c > (1ULL << L) ? kFullCode + 1
                                                                            : (unsigned long long)c << (63 - L);
        unsigned long long S = share;
        unsigned n = c;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, S, o);
            const unsigned z = __shfl_up_sync(0xffffffffu, n, o);
            if ((int)lane >= o) { S = sat_add(S, y); n += z; }
        }
        S = sat_add(S, scarry);
        n += ncarry;
        unsigned long long before = __shfl_up_sync(0xffffffffu, S, 1);
        if (lane == 0) before = scarry;
        T.count[L] = c;
        T.start[L] = n - c;
        T.first[L] = c ? before >> (63 - L) : 0ULL;
        T.lim[L] = L == 0 ? 0ULL : S >= kFullCode ? ~0ULL : S << 1;
        scarry = __shfl_sync(0xffffffffu, S, 31);
        ncarry = __shfl_sync(0xffffffffu, n, 31);
    }
    return scarry <= kFullCode;
}
// the tables into the scratch that the encoder and the decoder read
__device__ __forceinline__ void store_tables(const HuffScratch &hs, const LenTabs &T, unsigned i)
{
    hs.first[i] = T.first[i];
    hs.lim[i] = T.lim[i];
    hs.start[i] = T.start[i];
    hs.count[i] = T.count[i];
}

// CRC-32 (reflected, polynomial 0xEDB88320, all-ones start and final xor) of
// the first 124 bytes of a 128-byte header, by one warp: lane j < 31 holds word
// j.  The register is linear in the message, so word j adds w_j x^(32 (31 - j))
// mod P (the all-ones start is an xor of the first word): one product of
// polynomials per lane and a reduction, where the bitwise or byte-table
// recurrence over 124 bytes is serial.
struct CrcPowers {
    uint32_t v[32];
    constexpr CrcPowers() : v()
    {
        uint32_t x = 0x80000000u;   // 1: bit 31 is the constant term
        for (int j = 31; j >= 0; j--) {
            v[j] = x;               // x^(32 (31 - j))
            for (int b = 0; b < 32; b++) x = (x >> 1) ^ ((x & 1u) ? 0xEDB88320u : 0u);
        }
    }
};
__constant__ CrcPowers kCrcPowers = CrcPowers();
// (a message of fewer words sits in lanes first..30)
__device__ __forceinline__ uint32_t crc32_words(uint32_t word, unsigned first)
{
    const unsigned lane = threadIdx.x & 31;
    uint32_t a = lane == first ? ~word : word, b = kCrcPowers.v[lane], p = 0;
#pragma unroll
    for (int i = 31; i >= 0; i--) {
        p ^= (a >> i) & 1u ? b : 0u;
        b = (b >> 1) ^ ((b & 1u) ? 0xEDB88320u : 0u);
    }
    return ~__reduce_xor_sync(0xffffffffu, lane >= first && lane < 31 ? p : 0u);
}
__device__ __forceinline__ uint32_t crc32_warp(uint32_t word) { return crc32_words(word, 0); }

// code lengths from the frequency-sorted leaves, one block
__global__ void __launch_bounds__(1024) merge_kernel(HuffScratch hs, unsigned D)
{
    extern __shared__ unsigned long long sm[];
    __shared__ unsigned ia, ib, nb, ka, kb, cnt[kMaxCodeLen + 2];
    __shared__ LenTabs T;
    __shared__ int done;
    const unsigned n = *hs.nsym;
    const unsigned tid = threadIdx.x;
    for (unsigned s = tid; s < D; s += blockDim.x) hs.len[s] = 0;
    for (unsigned L = tid; L < kMaxCodeLen + 2; L += blockDim.x) cnt[L] = 0;
    if (n == 0) return;
    if (n == 1) {
        __syncthreads();
        if (tid == 0) {
            unsigned s = (unsigned)(hs.sorted[0] & 0xFFFFu);
            hs.len[s] = 1;
            hs.keys2[0] = (1ULL << 16) | s;
            cnt[1] = 1;
        }
        __syncthreads();
        if (tid < 32) length_tables(T, cnt);
        __syncthreads();
        if (tid < 64) store_tables(hs, T, tid);
        return;
    }
    const bool insm = n <= (unsigned)kSmemKeys;
    unsigned long long *leafw = insm ? sm : hs.leafw;
    unsigned long long *intw = insm ? sm + n : hs.intw;
    for (unsigned i = tid; i < n; i += blockDim.x) {
        leafw[i] = hs.sorted[i] >> 16;
        intw[i] = 0;
    }
    if (tid == 0) { ia = ib = nb = 0; done = 0; }
    __syncthreads();
    const unsigned long long INF = ~0ULL;
    while (true) {
        if (tid == 0) {
            unsigned remA = n - ia, remB = nb - ib;
            if (remA + remB <= 1) {
                done = 1;
            } else {
                unsigned long long wa = remA ? leafw[ia] : INF, wb = remB ? intw[ib] : INF;
                unsigned long long wmin = wa < wb ? wa : wb;
                unsigned long long thr = wmin > (INF >> 1) ? INF : 2 * wmin;
                unsigned a = count_le(leafw + ia, remA, thr), b = count_le(intw + ib, remB, thr);
                if (a + b < 2) {
                    a = b = 0;
                    for (int t = 0; t < 2; t++) {
                        bool la = (a < remA) && (b >= remB || leafw[ia + a] <= intw[ib + b]);
                        if (la) a++; else b++;
                    }
                } else if ((a + b) & 1) {
                    if (a == 0) b--;
                    else if (b == 0) a--;
                    else if (intw[ib + b - 1] >= leafw[ia + a - 1]) b--;
                    else a--;
                }
                ka = a;
                kb = b;
            }
        }
        __syncthreads();
        if (done) break;
        const unsigned a = ka, b = kb;
        for (unsigned i = tid; i < a + b; i += blockDim.x) {
            unsigned long long w;
            unsigned q, node;
            if (i < a) {
                w = leafw[ia + i];
                q = i + count_lt(intw + ib, b, w);       // equal weights: the leaf first
                node = ia + i;
            } else {
                unsigned j = i - a;
                w = intw[ib + j];
                q = j + count_le(leafw + ia, a, w);
                node = n + ib + j;
            }
            unsigned t = nb + (q >> 1);
            atomicAdd(&intw[t], w);
            hs.parent[node] = n + t;
        }
        __syncthreads();
        if (tid == 0) { ia += a; ib += b; nb += (a + b) >> 1; }
        __syncthreads();
    }
    // depth of every node by pointer jumping (parents have larger indices)
    const unsigned total = 2 * n - 1, root = total - 1;
    unsigned *A0 = hs.anc, *A1 = hs.anc + total, *D0 = hs.dep, *D1 = hs.dep + total;
    for (unsigned i = tid; i < total; i += blockDim.x) {
        A0[i] = (i == root) ? root : hs.parent[i];
        D0[i] = (i == root) ? 0u : 1u;
    }
    __syncthreads();
    for (int step = 0; step < 7; step++) {
        for (unsigned i = tid; i < total; i += blockDim.x) {
            unsigned a = A0[i];
            D1[i] = D0[i] + D0[a];
            A1[i] = A0[a];
        }
        __syncthreads();
        unsigned *t = A0; A0 = A1; A1 = t;
        t = D0; D0 = D1; D1 = t;
    }
    for (unsigned i = tid; i < n; i += blockDim.x) {
        unsigned L = D0[i];
        if (A0[i] != root || L > (unsigned)kMaxCodeLen || L == 0) {
            atomicExch(hs.status, (unsigned)DS_LENGTH);
            L = kMaxCodeLen;
        }
        unsigned s = (unsigned)(hs.sorted[i] & 0xFFFFu);
        hs.len[s] = (uint8_t)L;
        hs.keys2[i] = ((unsigned long long)L << 16) | s;
        atomicAdd(&cnt[L], 1u);
    }
    __syncthreads();
    if (tid < 32 && !length_tables(T, cnt) && tid == 0) atomicExch(hs.status, (unsigned)DS_FORMAT);
    __syncthreads();
    if (tid < 64) store_tables(hs, T, tid);
}

// entry of the encoder's packed codeword table: code << 6 | length for
// codewords of at most 26 bits (0: absent symbol); kPackLong sends the symbol
// to the full tables
constexpr uint32_t kPackLong = 0xFFFFFFFFu;
__device__ __forceinline__ uint32_t pack_code(unsigned long long code, unsigned L)
{
    return L <= 26 ? (uint32_t)((code << 6) | L) : kPackLong;
}

// canonical codeword of every present symbol
__global__ void __launch_bounds__(256) assign_kernel(HuffScratch hs)
{
    const unsigned n = *hs.nsym;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        unsigned long long k = hs.keys2[i];
        unsigned s = (unsigned)(k & 0xFFFFu), L = (unsigned)(k >> 16);
        unsigned r = hs.rank[i];
        hs.code[s] = hs.first[L] + (r - hs.start[L]);
        hs.pack[s] = pack_code(hs.code[s], L);
    }
}

// Decoder table entry of every 13-bit prefix t (P = kLutBits):
//   codeword of at most P bits:     symbol | L << 16                        (1 <= L <= P)
//   longer codewords, Lmax <= P + kSubMax, within the second-level budget:
//                                   kSubFlag | off | (Lmax - P) << 16; the next
//                                   Lmax - P bits r select lut_sub[off + r], an
//                                   entry symbol | L << 16 (0: no codeword)
//   other longer codewords:         kLongFlag | Lmin << 16 | (Lmax - Lmin) << 24
//                                   (canonical codes grow in length with their value)
//   no codeword (incomplete code):  0
constexpr uint32_t kLongFlag = 0x80000000u;
constexpr uint32_t kSubFlag = 0x20000000u;

// length of the canonical codeword at the top of the left-aligned window,
// known to lie in [lo, hi]: the first length l in [lo, hi) whose limit lim[l]
// the window stays below, else hi (the limits do not decrease with l, so a
// binary search finds it)
__device__ __forceinline__ unsigned code_len_in(const LenTabs &t, unsigned long long win, unsigned lo, unsigned hi)
{
    while (lo < hi) {
        const unsigned m = (lo + hi) >> 1;
        if (win >= t.lim[m]) lo = m + 1; else hi = m;
    }
    return lo;
}

// symbol | L << 16 of the codeword of length L at the top of the window (0: none)
__device__ __forceinline__ uint32_t leaf_of(const LenTabs &t, const uint16_t *sorted_sym, unsigned n,
                                            unsigned long long win, unsigned L)
{
    const unsigned long long off = (win >> (64 - L)) - t.first[L];
    if (off >= t.count[L]) return 0u;
    const unsigned idx = t.start[L] + (unsigned)off;
    return idx < n ? ((uint32_t)sorted_sym[idx] | (L << 16)) : 0u;
}

// Canonical codewords (Sec. IV-B): the present symbols ordered by (length,
// symbol) get consecutive codewords within each length, so a symbol's rank is
// start[L] plus the number of smaller symbols of its length L, and its
// codeword first[L] plus that number.  A block of 1024 threads: warp w owns a
// contiguous run of symbols, wc[w][L] counts its symbols of length L (grouped
// by __match_any_sync, 32 at a time), a scan over the warps turns the counts
// into offsets within each length, and a second walk over the run ranks its
// symbols: three block barriers for the whole alphabet.
constexpr int kWcStride = 65;     // 64 lengths, padded against bank conflicts
__device__ __forceinline__ unsigned canonical_run(unsigned D) { return ((D + 1023) / 1024) * 32; }

// wc (zeroed) <- per-warp counts, then offsets within each length; cnt[64] <-
// counts per length.  lens must be complete; ends with a block barrier.
__device__ __forceinline__ void canonical_counts(const uint8_t *lens, unsigned D, unsigned *wc, unsigned *cnt)
{
    const unsigned lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned run = canonical_run(D), r0 = w * run;
    for (unsigned i = 0; i < run; i += 32) {
        const unsigned s = r0 + i + lane;
        const unsigned L = s < D ? lens[s] : 0u;
        const unsigned m = __match_any_sync(0xffffffffu, L);
        if (L && (m & ((1u << lane) - 1)) == 0) wc[w * kWcStride + L] += __popc(m);
        __syncwarp();
    }
    __syncthreads();
    for (unsigned L = w; L < 64; L += 32) {
        const unsigned x = wc[lane * kWcStride + L];
        unsigned y = x;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned z = __shfl_up_sync(0xffffffffu, y, o);
            if ((int)lane >= o) y += z;
        }
        wc[lane * kWcStride + L] = y - x;
        if (lane == 31) cnt[L] = y;
    }
    __syncthreads();
}
// f(s, L, k): symbol s of length L is the k-th of its length (L = 0: absent)
template <typename F>
__device__ __forceinline__ void canonical_ranks(const uint8_t *lens, unsigned D, unsigned *wc, F f)
{
    const unsigned lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned run = canonical_run(D), r0 = w * run;
    for (unsigned i = 0; i < run; i += 32) {
        const unsigned s = r0 + i + lane;
        const unsigned L = s < D ? lens[s] : 0u;
        const unsigned m = __match_any_sync(0xffffffffu, L);
        const unsigned below = __popc(m & ((1u << lane) - 1));
        if (s < D) f(s, L, L ? wc[w * kWcStride + L] + below : 0u);
        __syncwarp();
        if (L && below == 0) wc[w * kWcStride + L] += __popc(m);
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// One-block codebook for alphabets of at most kFusedMaxD symbols, everything
// in shared memory: present symbols, their (frequency, symbol) order, the
// two-queue code lengths in rounds (as merge_kernel), depths, canonical
// codewords.  One block, so latency bounds it: 128 -> 58 us at 8000 present
// symbols (513^3, 1e-3), 80 -> 27 us at 129^2.  What each part does about it (the
// cycles are those of the form it replaced, of 250 thousand at 513^3):
//   sort      radix sort of the frequencies, eight bits a pass and only as many
//             passes as the largest frequency has bytes; stable, so equal
//             frequencies stay in symbol order (merge-path rounds: 125k);
//   rounds    pair t of a round finds its two nodes by one merge-path search
//             and sums them (a rank search and a 64-bit shared atomic per
//             node: 75k); limits by 32-way searches; rounds of at most kWarpRound nodes run on warp 0
//             without block barriers;
//   depths    from the root, round by round: a node's parent is always made in
//             a later round (pointer jumping over all nodes: 28k).
constexpr unsigned kFusedMaxD = 8192;
constexpr unsigned kWarpRound = 64;
// Rounds of one build: no node of weight below 2 w survives the two rounds
// after one whose smallest weight is w, and weights are below 2^64.
constexpr unsigned kMaxRounds = 136;
constexpr unsigned kDigStride = 258;   // 256 digits of 16-bit counts, padded against bank conflicts
constexpr size_t kCodebookSmem = 16ull * kFusedMaxD            // keys + sort buffer / internal weights
                                 + 2ull * 2 * kFusedMaxD         // parents (digit counts while sorting)
                                 + kFusedMaxD                    // depths of the internal nodes
                                 + kFusedMaxD                    // lengths by symbol
                                 + 4ull * 32 * kWcStride;        // per-warp length counts
static_assert(32 * kDigStride * 2 <= 4 * kFusedMaxD, "digit counts fit the parents' space");

// number of the first rem sorted values v(i) that are <= thr (v non-decreasing),
// by one warp: 32 probes a step
template <typename F>
__device__ __forceinline__ unsigned warp_count_le(F v, unsigned rem, unsigned long long thr, unsigned lane)
{
    unsigned lo = 0, len = rem;
    // most counts are small: the first 32 values first
    unsigned c = __popc(__ballot_sync(0xffffffffu, lane < rem && v(lane) <= thr));
    if (c < 32 || rem <= 32) return c;
    lo = 32;
    len = rem - 32;
    while (len > 32) {
        const unsigned step = (len + 31) / 32, e = (lane + 1) * step;   // probe the last value of part `lane`
        c = __popc(__ballot_sync(0xffffffffu, e <= len && v(lo + e - 1) <= thr));
        lo += c * step;
        len = min(step - 1, len - c * step);                             // the part's last value is > thr, or past the end
        if (c == 32) return lo;
    }
    return lo + __popc(__ballot_sync(0xffffffffu, lane < len && v(lo + lane) <= thr));
}

__device__ __forceinline__ void codebook_body(const unsigned long long *hist, unsigned D, const HuffScratch &hs)
{
    extern __shared__ __align__(16) unsigned char csm[];
    unsigned long long *key = reinterpret_cast<unsigned long long *>(csm);   // [kFusedMaxD]
    unsigned long long *aux = key + kFusedMaxD;                              // [kFusedMaxD]
    uint16_t *par = reinterpret_cast<uint16_t *>(aux + kFusedMaxD);          // [2 kFusedMaxD]
    uint8_t *dep = reinterpret_cast<uint8_t *>(par + 2 * kFusedMaxD);        // [kFusedMaxD]
    uint8_t *lens = dep + kFusedMaxD;                                        // [kFusedMaxD]
    unsigned *wc = reinterpret_cast<unsigned *>(lens + kFusedMaxD);          // [32 * kWcStride]
    __shared__ unsigned wcnt[32], wlo[32], whi[32], cnt[64], dbase[256];
    __shared__ unsigned long long wor[32];
    __shared__ LenTabs T;
    __shared__ unsigned s_ia, s_ib, s_nb, s_a, s_b, s_rounds;
    __shared__ int s_done;
    __shared__ uint16_t rstart[kMaxRounds];
    const unsigned tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const unsigned long long INF = ~0ULL;
    constexpr unsigned R = kFusedMaxD / 1024;   // symbols per thread

    // 1. present symbols as keys (frequency << 16) | s, in symbol order: warp w
    //    compacts its run of 32 R symbols
    unsigned n;
    unsigned long long orf;
    {
        unsigned long long f[R];
        unsigned before[R], mycnt = 0;
        const unsigned r0 = w * 32 * R;
#pragma unroll
        for (unsigned i = 0; i < R; i++) f[i] = r0 + 32 * i + lane < D ? hist[r0 + 32 * i + lane] : 0ULL;
        for (unsigned i = tid; i < 32 * kWcStride; i += 1024) wc[i] = 0;
        for (unsigned i = tid; i < (D + 3) / 4; i += 1024) reinterpret_cast<uint32_t *>(lens)[i] = 0;
        unsigned lo = 0xFFFFFFFFu, hi = 0;
        unsigned long long o = 0;
#pragma unroll
        for (unsigned i = 0; i < R; i++) {
            const unsigned ball = __ballot_sync(0xffffffffu, f[i] != 0);
            before[i] = mycnt + __popc(ball & ((1u << lane) - 1));
            mycnt += __popc(ball);
            if (ball) {
                lo = min(lo, r0 + 32 * i + __ffs(ball) - 1);
                hi = r0 + 32 * i + 31 - __clz(ball);
            }
            o |= f[i];
        }
        const unsigned ol = __reduce_or_sync(0xffffffffu, (unsigned)o), oh = __reduce_or_sync(0xffffffffu, (unsigned)(o >> 32));
        if (lane == 0) { wcnt[w] = mycnt; wlo[w] = lo; whi[w] = hi; wor[w] = ((unsigned long long)oh << 32) | ol; }
        __syncthreads();
        // every warp scans the warps' counts
        const unsigned c = wcnt[lane];
        unsigned x = c;
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, x, d);
            if ((int)lane >= d) x += y;
        }
        const unsigned base = __shfl_sync(0xffffffffu, x - c, w);
        n = __shfl_sync(0xffffffffu, x, 31);
        const unsigned long long wo = wor[lane];
        orf = ((unsigned long long)__reduce_or_sync(0xffffffffu, (unsigned)(wo >> 32)) << 32) |
              __reduce_or_sync(0xffffffffu, (unsigned)wo);
        if (w == 0) {
            const unsigned l0 = __reduce_min_sync(0xffffffffu, wlo[lane]), h0 = __reduce_max_sync(0xffffffffu, whi[lane]);
            if (lane == 0) {
                *hs.nsym = n;
                *hs.s_lo = n ? l0 : 0;
                *hs.s_hi = n ? h0 : 0;
            }
        }
#pragma unroll
        for (unsigned i = 0; i < R; i++)
            if (f[i]) key[base + before[i]] = (f[i] << 16) | (r0 + 32 * i + lane);
    }
    __syncthreads();
    if (n == 0) {
        for (unsigned i = tid; i < D; i += 1024) { hs.len[i] = 0; hs.pack[i] = 0; }
        return;
    }

    // 2. radix sort by frequency: warp w ranks its contiguous run of keys
    unsigned long long *src = key, *dst = aux;
    {
        uint16_t *dc = par;   // [32][kDigStride] digit counts of every warp
        const unsigned per = ((n + 1023) / 1024) * 32, p0 = w * per;
        uint16_t *mine = dc + w * kDigStride;
        for (unsigned shift = 16; shift == 16 || (shift < 64 && (orf >> (shift - 16)) != 0); shift += 8) {
            for (unsigned i = lane; i < kDigStride / 2; i += 32) reinterpret_cast<uint32_t *>(mine)[i] = 0;
            __syncwarp();
            unsigned long long k[R];
            unsigned rk[R];
#pragma unroll
            for (unsigned i = 0; i < R; i++) {
                const unsigned p = p0 + 32 * i + lane;
                k[i] = 32 * i < per && p < n ? src[p] : INF;
            }
#pragma unroll
            for (unsigned i = 0; i < R; i++) {
                if (32 * i >= per) break;
                const bool in = p0 + 32 * i + lane < n;
                const unsigned d = in ? (unsigned)(k[i] >> shift) & 0xFFu : 0x100u;
                const unsigned m = __match_any_sync(0xffffffffu, d);
                const unsigned below = __popc(m & ((1u << lane) - 1)), at = in ? mine[d] : 0u;
                __syncwarp();
                if (in && below == 0) mine[d] = (uint16_t)(at + __popc(m));
                __syncwarp();
                rk[i] = at + below;
            }
            __syncthreads();
            // offsets of the warps within each digit, and the digits' totals
#pragma unroll
            for (unsigned j = 0; j < 8; j++) {
                const unsigned d = 8 * w + j, x = dc[lane * kDigStride + d];
                unsigned y = x;
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned z = __shfl_up_sync(0xffffffffu, y, o);
                    if ((int)lane >= o) y += z;
                }
                dc[lane * kDigStride + d] = (uint16_t)(y - x);
                if (lane == 31) dbase[d] = y;
            }
            __syncthreads();
            if (w == 0) {
                unsigned v[8], sum = 0;
#pragma unroll
                for (int j = 0; j < 8; j++) { v[j] = sum; sum += dbase[8 * lane + j]; }
                unsigned x = sum;
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned z = __shfl_up_sync(0xffffffffu, x, o);
                    if ((int)lane >= o) x += z;
                }
#pragma unroll
                for (int j = 0; j < 8; j++) dbase[8 * lane + j] = x - sum + v[j];
            }
            __syncthreads();
#pragma unroll
            for (unsigned i = 0; i < R; i++) {
                const unsigned p = p0 + 32 * i + lane;
                if (32 * i < per && p < n) {
                    const unsigned d = (unsigned)(k[i] >> shift) & 0xFFu;
                    dst[dbase[d] + mine[d] + rk[i]] = k[i];
                }
            }
            __syncthreads();
            unsigned long long *t = src; src = dst; dst = t;
        }
    }
    const unsigned long long *leaf = src;     // [n] sorted keys
    unsigned long long *intw = dst;           // [n - 1] weights of the internal nodes
    auto LW = [&](unsigned i) { return leaf[i] >> 16; };

    // 3. two-queue merging in rounds
    if (tid == 0) { s_ia = s_ib = s_nb = s_rounds = 0; s_done = 0; }
    __syncthreads();
    // pair t of a round: the merged nodes 2t and 2t + 1 of its a leaves and b
    // internal nodes (equal weights: the leaf first) become internal node nb + t
    auto pair = [&](unsigned t, unsigned ia, unsigned ib, unsigned nb, unsigned a, unsigned b) {
        const unsigned d = 2 * t;
        unsigned lo = d > b ? d - b : 0u, hi = min(d, a);
        while (lo < hi) {
            const unsigned m = (lo + hi) >> 1;
            if (LW(ia + m) <= intw[ib + d - 1 - m]) lo = m + 1; else hi = m;
        }
        unsigned i = lo, j = d - lo;
        unsigned long long sum = 0;
#pragma unroll
        for (int e = 0; e < 2; e++) {
            const unsigned long long x = i < a ? LW(ia + i) : INF, y = j < b ? intw[ib + j] : INF;
            const bool l = x <= y;
            sum += l ? x : y;
            par[l ? ia + i : n + ib + j] = (uint16_t)(n + nb + t);
            if (l) i++; else j++;
        }
        intw[nb + t] = sum;
    };
    // s_done is read only between the barrier after warp 0 writes it and the
    // next round's barriers, so every warp leaves the loop at the same barrier
    while (n > 1) {
        if (w == 0) {
            unsigned ia = s_ia, ib = s_ib, nb = s_nb, rounds = s_rounds, a = 0, b = 0;
            int state = 0;
            while (true) {
                const unsigned remA = n - ia, remB = nb - ib;
                if (remA + remB <= 1) { state = 2; break; }
                const unsigned long long wa = remA ? LW(ia) : INF, wb = remB ? intw[ib] : INF;
                const unsigned long long wmin = wa < wb ? wa : wb;
                const unsigned long long thr = wmin > (INF >> 1) ? INF : 2 * wmin;
                a = warp_count_le([&](unsigned i) { return LW(ia + i); }, remA, thr, lane);
                b = warp_count_le([&](unsigned i) { return intw[ib + i]; }, remB, thr, lane);
                if (a + b < 2) {
                    a = b = 0;
                    for (int t = 0; t < 2; t++) {
                        const bool la = (a < remA) && (b >= remB || LW(ia + a) <= intw[ib + b]);
                        if (la) a++; else b++;
                    }
                } else if ((a + b) & 1) {
                    if (a == 0) b--;
                    else if (b == 0) a--;
                    else if (intw[ib + b - 1] >= LW(ia + a - 1)) b--;
                    else a--;
                }
                if (lane == 0 && rounds < kMaxRounds) rstart[rounds] = (uint16_t)nb;
                rounds++;
                if (a + b > kWarpRound) { state = 1; break; }
                if (2 * lane < a + b) pair(lane, ia, ib, nb, a, b);
                __syncwarp();
                ia += a; ib += b; nb += (a + b) >> 1;
            }
            if (lane == 0) {
                s_ia = ia; s_ib = ib; s_nb = nb; s_a = a; s_b = b; s_rounds = rounds;
                s_done = state == 2;
            }
        }
        __syncthreads();
        if (s_done) break;
        const unsigned ia = s_ia, ib = s_ib, nb = s_nb, a = s_a, b = s_b;
        for (unsigned t = tid; 2 * t < a + b; t += 1024) pair(t, ia, ib, nb, a, b);
        __syncthreads();
        if (tid == 0) { s_ia = ia + a; s_ib = ib + b; s_nb = nb + ((a + b) >> 1); }
        __syncthreads();
    }

    // 4. depths of the internal nodes (the root is the last one), the rounds
    //    from the last to the first: warp 0 alone over the small ones at the top
    //    of the tree, then the block.  Depths saturate at 255.
    if (n > 1) {
        const unsigned ni = n - 1;
        int r = (int)s_rounds - 1;
        auto depth = [&](unsigned i) {
            const unsigned d = i + 1 == ni ? 0u : (unsigned)dep[par[n + i] - n] + 1u;
            dep[i] = (uint8_t)min(d, 255u);
        };
        unsigned end = ni;
        for (; r >= 0 && end - rstart[r] <= kWarpRound; end = rstart[r], r--) {
            if (w == 0) {
                for (unsigned i = rstart[r] + lane; i < end; i += 32) depth(i);
                __syncwarp();
            }
        }
        __syncthreads();
        for (; r >= 0; end = rstart[r], r--) {
            for (unsigned i = rstart[r] + tid; i < end; i += 1024) depth(i);
            __syncthreads();
        }
    }

    // 5. code lengths, canonical tables and codewords
    for (unsigned i = tid; i < n; i += 1024) {
        unsigned L = n == 1 ? 1u : (unsigned)dep[par[i] - n] + 1u;
        if (L > (unsigned)kMaxCodeLen) {
            atomicExch(hs.status, (unsigned)DS_LENGTH);
            L = kMaxCodeLen;
        }
        lens[(unsigned)(leaf[i] & 0xFFFFu)] = (uint8_t)L;
    }
    __syncthreads();
    canonical_counts(lens, D, wc, cnt);
    if (w == 0 && !length_tables(T, cnt) && lane == 0) atomicExch(hs.status, (unsigned)DS_FORMAT);
    __syncthreads();
    if (tid < 64) store_tables(hs, T, tid);
    canonical_ranks(lens, D, wc, [&](unsigned s, unsigned L, unsigned k) {
        const unsigned long long code = L ? T.first[L] + k : 0ULL;
        hs.len[s] = (uint8_t)L;
        hs.code[s] = code;
        hs.pack[s] = pack_code(code, L);
    });
}

__global__ void __launch_bounds__(1024, 1) codebook_kernel(const unsigned long long *hist, unsigned D, HuffScratch hs)
{
    next_begin();
    codebook_body(hist, D, hs);
}

// one codebook per block: the codebooks of a batch of fields in one launch
__global__ void __launch_bounds__(1024, 1) codebook_batch_kernel(const CodebookJob *jobs)
{
    const CodebookJob j = jobs[blockIdx.x];
    codebook_body(j.hist, j.D, j.hs);
}

// Decoder tables from the code lengths of symbols s_lo..s_hi (every other
// symbol of the alphabet absent): per-length counts, canonical tables, the
// (length, symbol) order of the symbols, the first-level table and the
// second-level tables, laid out in prefix order by a scan of their sizes
// (prefixes past the budget keep long entries).  With a header on the device
// (a.dh) it is checked and parsed here first.
//
// Single-block latency bounds this (it was three launches of one block: 10 us
// header, 17 us tables, 24-78 us look-up tables at 8192 symbols).  So every
// block of a small grid does the short common part for itself, with no
// exchange between blocks, and the blocks share only what is long: block b
// stores its slice of the first level and its share of the second-level
// entries, one thread per entry.  Block 0 stores everything else.
// One launch of 17 us against 47 at 129^2 (19 against 101 at 130x67x45 and 1e-4,
// 18 against 66 at 513^3).
constexpr int kTabThreads = 1024;
constexpr int kTabBlocks = 16;
constexpr unsigned kTabPer = (1u << kLutBits) / kTabThreads;    // prefixes per thread
constexpr unsigned kTabSyms = 16384;                            // sorted symbols staged in shared memory
constexpr size_t kTabSmem = 4ull * 32 * kWcStride + 2ull * (4u << kLutBits) + 2ull * kTabSyms;   // + D code lengths

// length of the codeword at the top of the left-aligned window: the first L in
// [1, maxL) whose limit it stays below, else maxL
template <int N>
__device__ __forceinline__ void code_lens(const LenTabs &T, const unsigned long long (&win)[N], unsigned maxL,
                                          unsigned (&L)[N])
{
#pragma unroll
    for (int j = 0; j < N; j++) L[j] = 1;
#pragma unroll
    for (unsigned s = 32; s; s >>= 1)
#pragma unroll
        for (int j = 0; j < N; j++)
            if (L[j] + s <= maxL && win[j] >= T.lim[L[j] + s - 1]) L[j] += s;
}

// checks of a container header (the host's parse_header, plus agreement with
// the shape, type and dictionary the caller expects) by one block; the same
// answer in every thread of every block
__device__ __forceinline__ bool parse_header_block(const uint8_t *b, unsigned long long in_bytes, const HdrExpect &ex,
                                                   DevHdr *out)
{
    __shared__ uint32_t hw[32];
    __shared__ DevHdr h;
    __shared__ int good;
    const unsigned tid = threadIdx.x;
    if (in_bytes < 128) return false;
    if (tid < 32) {
        const uint32_t w = reinterpret_cast<const uint32_t *>(b)[tid];
        hw[tid] = w;
        const uint32_t crc = crc32_warp(w);
        if (tid == 31) good = crc == w;
    }
    __syncthreads();
    auto w64 = [&](int at) { return (unsigned long long)hw[at / 4] | ((unsigned long long)hw[at / 4 + 1] << 32); };
    if (tid == 0) {
        bool g = good && hw[0] == 0x52445048u && hw[1] == 3u;    // "HPDR", version 3
        g = g && (int)hw[2] == ex.dtype && (int)hw[3] == ex.ndim && (int)hw[10] == ex.L && hw[12] <= 1u &&
            hw[13] == ex.D && hw[14] == ex.K && w64(96) == ex.N;
        for (int k = 0; k < 3; k++) g = g && w64(16 + 8 * k) == ex.dims[k];
        h.pad = 0;
        h.s_lo = hw[15];
        h.n_esc = w64(104);
        h.total_bits = w64(112);
        const uint32_t w120 = hw[30];
        h.s_hi = w120 & 0xFFFFu;
        h.esc_w = (w120 >> 16) & 0xFFu;
        g = g && (w120 >> 24) == 0u && h.s_hi < ex.D && h.s_lo <= h.s_hi && h.n_esc <= ex.N && h.esc_w <= 63u &&
            ((h.n_esc > 0) == (h.esc_w > 0)) && h.total_bits >= ex.N &&
            h.total_bits <= 63ULL * ex.N + (unsigned long long)h.esc_w * h.n_esc;
        if (g) {
            const unsigned long long nch = (ex.N + ex.K - 1) / ex.K;
            h.nwords = (h.total_bits + 31) / 32;
            h.off_len = a16(128 + 8ULL * (ex.L + 1));
            h.off_chunk = a16(h.off_len + (h.s_hi - h.s_lo + 1));
            h.off_bits = a16(h.off_chunk + 8 * nch);
            g = h.off_bits + 4 * h.nwords <= in_bytes;
        }
        good = g;
    }
    __syncthreads();
    bool g = good != 0;
    if (g && (int)tid <= ex.L) {
        const double q = reinterpret_cast<const double *>(b + 128)[tid];
        g = q > 0.0 && isfinite(q);
    }
    g = __syncthreads_and(g) != 0;
    *out = h;
    return g;
}

__global__ void __launch_bounds__(kTabThreads, 1) dec_tables_kernel(TabArgs a, HuffScratch hs)
{
    extern __shared__ __align__(16) unsigned char tsm[];
    uint32_t *ent = reinterpret_cast<uint32_t *>(tsm);                          // [1 << kLutBits] first level
    unsigned *soff = ent + (1u << kLutBits);                                    // [1 << kLutBits] second-level offsets
    uint16_t *ssym = reinterpret_cast<uint16_t *>(soff + (1u << kLutBits));     // [kTabSyms]
    unsigned *wc = reinterpret_cast<unsigned *>(ssym + kTabSyms);               // [32][kWcStride]
    uint8_t *lens = reinterpret_cast<uint8_t *>(wc + 32 * kWcStride);           // [D]
    __shared__ LenTabs T;
    __shared__ unsigned cnt[64], wsum[32], total_s;
    __shared__ int okc;
    const unsigned tid = threadIdx.x, lane = tid & 31, w = tid >> 5, D = a.D;
    const bool lead = blockIdx.x == 0;
    next_begin();
    // ---- scalars and header
    const uint8_t *lenb = a.lenb;
    unsigned s_lo = a.s_lo, s_hi = a.s_hi;
    if (a.dh || a.set_scalars) {
        if (lead) {
            unsigned char *z = reinterpret_cast<unsigned char *>(a.sc);
            for (unsigned i = tid; i < sizeof(Scalars); i += kTabThreads) z[i] = 0;
            __syncthreads();
        }
        DevHdr h;
        bool ok = true;
        if (a.dh) ok = parse_header_block(a.base, a.in_bytes, a.ex, &h);
        if (!ok) {
            if (lead && tid == 0) a.sc->status = (unsigned)DS_FORMAT;
            return;
        }
        if (a.dh) { lenb = a.base + h.off_len; s_lo = h.s_lo; s_hi = h.s_hi; }
        const int L = a.dh ? a.ex.L : a.si.L;
        if (lead && (int)tid <= L) {
            const double q = a.dh ? reinterpret_cast<const double *>(a.base + 128)[tid] : a.si.q[tid];
            a.sc->q[tid] = q;
            a.sc->q_f[tid] = __double2float_rn(q);
            const double r = 1.0 / q;
            a.sc->rho_d[tid] = r;
            a.sc->rho_f[tid] = __double2float_rn(r);
            a.sc->rho_lo[tid] = __double2float_rn(r - (double)__double2float_rn(r));
        }
        if (lead && tid == 0) {
            a.sc->n_esc = a.dh ? h.n_esc : a.si.n_esc;
            a.sc->esc_w = a.dh ? h.esc_w : a.si.esc_w;
            a.sc->total_bits = a.dh ? h.total_bits : a.si.total_bits;
            if (a.dh) *a.dh = h;
        }
        if (a.deq)
            for (unsigned i = blockIdx.x * kTabThreads + tid; i < (unsigned)(L + 1) * D; i += kTabBlocks * kTabThreads) {
                const unsigned l = i / D;
                const double q = a.dh ? reinterpret_cast<const double *>(a.base + 128)[l] : a.si.q[l];
                a.deq[i] = __dmul_rn((double)((int)(i - l * D) - (int)(D / 2)), q);
            }
    }
    // ---- code lengths; counts per warp and length over the warp's run of symbols
    if (tid == 0) okc = 1;
    for (unsigned i = tid; i < 32 * kWcStride; i += kTabThreads) wc[i] = 0;
    __syncthreads();
    constexpr int U = 8;
    for (unsigned s0 = tid; s0 < D; s0 += U * kTabThreads) {
        unsigned v[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const unsigned s = s0 + u * kTabThreads;
            v[u] = s < D && s >= s_lo && s <= s_hi ? lenb[s - s_lo] : 0u;
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const unsigned s = s0 + u * kTabThreads;
            if (v[u] > (unsigned)kMaxCodeLen) { okc = 0; v[u] = 0; }
            if (s < D) lens[s] = (uint8_t)v[u];
        }
    }
    __syncthreads();
    canonical_counts(lens, D, wc, cnt);
    if (w == 0 && !length_tables(T, cnt) && lane == 0) okc = 0;
    __syncthreads();
    const unsigned n = T.start[63] + T.count[63];
    const bool ok = okc && n > 0;
    // ---- symbols in (length, symbol) order
    uint16_t *sorted = n <= kTabSyms ? ssym : hs.sorted_sym;
    if (ok)
        canonical_ranks(lens, D, wc, [&](unsigned s, unsigned L, unsigned k) {
            if (L) sorted[T.start[L] + k] = (uint16_t)s;
        });
    __syncthreads();
    if (lead) {
        if (tid < 64) store_tables(hs, T, tid);
        if (tid == 0) {
            *hs.nsym = n;
            if (!ok) atomicExch(hs.status, (unsigned)DS_FORMAT);
        }
        if (ok && n <= kTabSyms) for (unsigned i = tid; i < n; i += kTabThreads) hs.sorted_sym[i] = ssym[i];
    }
    // ---- first level: the codeword whose left-justified range holds a prefix's
    // first bit string (at most P bits long, it is a prefix of every extension),
    // else the range of lengths under the prefix
    unsigned maxL = 0;
    for (int l = kMaxCodeLen; l >= 1; l--) if (T.count[l]) { maxL = (unsigned)l; break; }
    const unsigned t0 = tid * kTabPer;
    constexpr unsigned long long kTail = (1ULL << (64 - kLutBits)) - 1;
    unsigned mine = 0;
    unsigned sbs[kTabPer];
    {
        unsigned long long win[kTabPer];
        unsigned lmin[kTabPer], lmax[kTabPer];
#pragma unroll
        for (unsigned j = 0; j < kTabPer; j++) win[j] = (unsigned long long)(t0 + j) << (64 - kLutBits);
        code_lens(T, win, ok ? maxL : 1u, lmin);
#pragma unroll
        for (unsigned j = 0; j < kTabPer; j++) win[j] |= kTail;
        code_lens(T, win, ok ? maxL : 1u, lmax);
#pragma unroll
        for (unsigned j = 0; j < kTabPer; j++) {
            uint32_t e = 0;
            sbs[j] = 0;
            if (ok) {
                if (lmin[j] <= (unsigned)kLutBits) {
                    e = leaf_of(T, sorted, n, win[j] & ~kTail, lmin[j]);
                } else {
                    e = kLongFlag | (lmin[j] << 16) | ((lmax[j] - lmin[j]) << 24);
                    if (lmax[j] <= (unsigned)(kLutBits + kSubMax)) {
                        sbs[j] = lmax[j] - kLutBits;
                        mine += 1u << sbs[j];
                    }
                }
            }
            ent[t0 + j] = e;
        }
    }
    // exclusive scan of the second-level sizes over the block
    unsigned incl = mine;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= (unsigned)o) incl += v;
    }
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    if (w == 0) {
        const unsigned v = wsum[lane];
        unsigned x = v;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= (unsigned)o) x += y;
        }
        wsum[lane] = x - v;
        if (lane == 31) total_s = x < kSubCap ? x : kSubCap;
    }
    __syncthreads();
    unsigned off = wsum[w] + incl - mine;
#pragma unroll
    for (unsigned j = 0; j < kTabPer; j++) {
        soff[t0 + j] = off;
        if (!sbs[j]) continue;
        const unsigned sz = 1u << sbs[j];
        if (off + sz <= kSubCap) ent[t0 + j] = kSubFlag | off | (sbs[j] << 16);
        off += sz;
    }
    __syncthreads();
    // ---- this block's slice of the first level and share of the second
    constexpr unsigned slice = (1u << kLutBits) / kTabBlocks;
    if (tid < slice) hs.lut1[blockIdx.x * slice + tid] = ent[blockIdx.x * slice + tid];
    for (unsigned e = blockIdx.x * kTabThreads + tid; e < total_s; e += kTabBlocks * kTabThreads) {
        // the last prefix whose second-level table starts at or before e
        unsigned t = 0;
#pragma unroll
        for (unsigned s = 1u << (kLutBits - 1); s; s >>= 1)
            if (soff[t + s] <= e) t += s;
        const uint32_t f = ent[t];
        if ((f & (kLongFlag | kSubFlag)) != kSubFlag) continue;   // cut off by the budget
        const unsigned sb = (f >> 16) & 0xFu, r = e - soff[t];
        const unsigned long long win[1] = {((unsigned long long)t << (64 - kLutBits)) |
                                           ((unsigned long long)r << (64 - kLutBits - sb))};
        unsigned L[1];
        code_lens(T, win, kLutBits + sb, L);
        hs.lut_sub[e] = leaf_of(T, sorted, n, win[0], L[0]);
    }
    if (lead && tid == 0) *hs.nsub = total_s;
}

// ---------------------------------------------------------------------------
// Encoder

struct Layout {
    unsigned long long off_len, off_chunk, off_bits, total;
};
__device__ __forceinline__ Layout container_layout(int L, unsigned long long ncoord, unsigned s_lo, unsigned s_hi,
                                                   unsigned long long nch, unsigned long long bits)
{
    Layout y;
    // the node coordinates (ncoord values, when the container carries them) follow q[L+1]
    y.off_len = a16(128 + 8ULL * (L + 1) + 8ULL * ncoord);
    y.off_chunk = a16(y.off_len + (s_hi - s_lo + 1));
    y.off_bits = a16(y.off_chunk + 8 * nch);
    y.total = y.off_bits + 4 * ((bits + 31) / 32);
    return y;
}

constexpr int kEncBlocks = 152 * 4;

// The encoder's unit of work: a warp takes r consecutive chunks (r K symbols,
// 32 per lane) when K < 1024 divides 1024, else one chunk.  The bitstream is
// continuous across chunks, so the grouping changes no output bit.
__host__ __device__ inline unsigned enc_group(unsigned K) { return (K < 1024 && 1024 % K == 0) ? 1024 / K : 1; }

// bits of every chunk (codewords + escape payloads); block b owns the
// contiguous chunk range [b*cpb, (b+1)*cpb) and leaves its sum in bsum
template <typename S>
__global__ void __launch_bounds__(256) enc_count_kernel(EncodeArgs a)
{
    constexpr int V = 16 / sizeof(S);   // symbols per 16-byte load
    const S *__restrict__ sym = reinterpret_cast<const S *>(a.sym);
    extern __shared__ __align__(16) uint8_t slen[];
    __shared__ unsigned long long wb[8];
    next_begin();
    if (block_skip(&a.sc->status)) return;
    // the length table's space in the scratch is a multiple of 256 bytes
    for (unsigned i = threadIdx.x; i < (a.D + 15) / 16; i += blockDim.x)
        reinterpret_cast<uint4 *>(slen)[i] = reinterpret_cast<const uint4 *>(a.len)[i];
    __syncthreads();
    // an escape adds its payload width to its codeword
    if (a.esc && threadIdx.x == 0) slen[0] = (uint8_t)(slen[0] + a.sc->esc_w);
    __syncthreads();
    const unsigned long long nch = (a.N + a.K - 1) / a.K;
    const unsigned long long cpb = (nch + gridDim.x - 1) / gridDim.x;
    const unsigned long long c0 = blockIdx.x * cpb, c1 = c0 + cpb < nch ? c0 + cpb : nch;
    const unsigned lane = threadIdx.x & 31, warp = (unsigned)warp_index();
    unsigned long long tb = 0;
    const unsigned r = enc_group(a.K);
    if (r > 1) {
        // r chunks per warp, 32 / r lanes per chunk, 32 symbols per lane
        const unsigned lpc = 32 / r;
        for (unsigned long long g = c0 + (unsigned long long)warp * r; g < c1; g += (blockDim.x >> 5) * r) {
            const unsigned long long c = g + lane / lpc;
            unsigned long long bits = 0;
            if (c < c1) {
                const unsigned long long beg = c * a.K + (unsigned long long)(lane % lpc) * 32;
                const unsigned long long cend = (c + 1) * a.K < a.N ? (c + 1) * a.K : a.N;
                if (beg + 32 <= cend) {
                    const uint4 *v = reinterpret_cast<const uint4 *>(sym + beg);
                    uint4 x[32 / V];
#pragma unroll
                    for (int u = 0; u < 32 / V; u++) x[u] = v[u];
#pragma unroll
                    for (int u = 0; u < 32 / V; u++) {
                        const S *e = reinterpret_cast<const S *>(&x[u]);
#pragma unroll
                        for (int k = 0; k < V; k++) bits += slen[e[k]];
                    }
                } else {
                    for (unsigned long long i = beg; i < cend; i++) bits += slen[sym[i]];
                }
            }
            // sum over the lpc lanes of each chunk
            for (unsigned o = 1; o < lpc; o <<= 1) bits += __shfl_xor_sync(0xffffffffu, bits, o);
            if (lane % lpc == 0 && c < c1) { a.chunk_bits[c] = bits; tb += bits; }
        }
        tb = warp_sum64(tb);
    } else
    for (unsigned long long c = c0 + warp; c < c1; c += blockDim.x >> 5) {
        const unsigned long long beg = c * a.K;
        const unsigned long long end = beg + a.K < a.N ? beg + a.K : a.N;
        unsigned long long bits = 0;
        if (end - beg == a.K) {
            // four 16-byte loads per lane in flight (K is a multiple of 128)
            const uint4 *v = reinterpret_cast<const uint4 *>(sym + beg);
            const unsigned nq = a.K / V;
            for (unsigned i0 = lane; i0 < nq; i0 += 128) {
                uint4 x[4];
                bool ok[4];
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    ok[u] = i0 + 32 * u < nq;
                    if (ok[u]) x[u] = v[i0 + 32 * u];
                }
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    if (!ok[u]) continue;
                    const S *e = reinterpret_cast<const S *>(&x[u]);
#pragma unroll
                    for (int k = 0; k < V; k++) bits += slen[e[k]];
                }
            }
        } else {
            for (unsigned long long i = beg + lane; i < end; i += 32) bits += slen[sym[i]];
        }
        bits = warp_sum64(bits);
        if (lane == 0) { a.chunk_bits[c] = bits; tb += bits; }
    }
    if (lane == 0) wb[warp] = tb;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long x = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) x += wb[w];
        a.bsum[blockIdx.x] = x;
    }
}

__device__ __forceinline__ uint32_t *enc_words(const EncodeArgs &a, unsigned long long nch, unsigned long long bits)
{
    if (!a.container) return a.words_out;
    Layout lay = container_layout(a.L, a.ncoord, a.sc->s_lo, a.sc->s_hi, nch, bits);
    return reinterpret_cast<uint32_t *>(a.container + lay.off_bits);
}

// chunk offsets and chunk table, container layout and capacity, and zeroed
// words where more than one writer will meet.  Block b continues from the sums
// of the blocks before it, which every block adds up for itself (a scan in a
// launch of its own cost 5 us and a gap on every call).
__global__ void __launch_bounds__(256) enc_scan_kernel(EncodeArgs a)
{
    __shared__ unsigned long long spre[8], stot[8];
    next_begin();
    if (block_skip(&a.sc->status)) return;
    const unsigned long long nch = (a.N + a.K - 1) / a.K;
    const unsigned long long cpb = (nch + gridDim.x - 1) / gridDim.x;
    const unsigned long long c0 = blockIdx.x * cpb, c1 = c0 + cpb < nch ? c0 + cpb : nch;
    const unsigned t = threadIdx.x, lane = t & 31, w = t >> 5;
    unsigned long long pre = 0, total = 0;
    for (unsigned i = t; i < gridDim.x; i += 256) {
        const unsigned long long x = a.bsum[i];
        total += x;
        if (i < blockIdx.x) pre += x;
    }
    pre = warp_sum64(pre);
    total = warp_sum64(total);
    if (lane == 0) { spre[w] = pre; stot[w] = total; }
    __syncthreads();
    pre = total = 0;
#pragma unroll
    for (int i = 0; i < 8; i++) { pre += spre[i]; total += stot[i]; }
    // the same decision in every block: nothing is written past the capacity
    uint32_t *words = a.words_out;
    unsigned long long *ctab = a.chunk_out;
    bool fits;
    if (a.container) {
        const Layout lay = container_layout(a.L, a.ncoord, a.sc->s_lo, a.sc->s_hi, nch, total);
        words = reinterpret_cast<uint32_t *>(a.container + lay.off_bits);
        ctab = reinterpret_cast<unsigned long long *>(a.container + lay.off_chunk);
        fits = lay.total <= a.capacity;
        if (blockIdx.x == 0 && t == 0) a.sc->out_bytes = lay.total;
    } else {
        fits = (total + 31) / 32 <= a.words_cap;
    }
    if (blockIdx.x == 0 && t == 0) {
        a.sc->total_bits = total;
        a.chunk_bits[nch] = total;
        if (!fits) atomicExch(&a.sc->status, (unsigned)DS_CAPACITY);
    }
    if (!fits) return;
    unsigned long long carry = pre;
    for (unsigned long long base = c0; base < c1; base += 256) {
        const unsigned long long c = base + t;
        const unsigned long long v = c < c1 ? a.chunk_bits[c] : 0;
        unsigned long long x = v;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
            if ((int)lane >= o) x += y;
        }
        __syncthreads();
        if (lane == 31) spre[w] = x;
        __syncthreads();
        unsigned long long before = 0, sum = 0;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            if (i < (int)w) before += spre[i];
            sum += spre[i];
        }
        if (c < c1) {
            const unsigned long long off = carry + before + x - v;
            a.chunk_bits[c] = off;
            ctab[c] = off;
            const unsigned long long cend = off + v;
            // a complete group of at least 1024 symbols (one warp, 32 or more per lane)
            // shares only its first word with the previous group and stores every
            // other word whole; other chunks are written word by word with atomics:
            // zero them
            const unsigned r = enc_group(a.K);
            const unsigned long long G = (unsigned long long)a.K * r;
            const bool full = (c / r + 1) * G <= a.N && G >= 1024;
            if (full) {
                if (c % r == 0) words[off >> 5] = 0u;
            } else {
                for (unsigned long long i = off >> 5; i <= ((cend ? cend - 1 : 0) >> 5); i++) words[i] = 0u;
            }
            if (c + 1 == nch && (total & 31)) words[total >> 5] = 0u;
        }
        carry += sum;
    }
}

// A complete group of 1024 symbols by one warp, 32 consecutive symbols per
// lane; what bounds it is the issue rate and the shared-memory look-ups, so a
// symbol is looked up once (its entry stays in a register for the emission),
// the bits move through two 32-bit registers by funnel shifts, and finished
// words go to shared memory, from where the group's words leave in whole
// rows: stored by each lane as they finish, every word was a sector of its own
// in L2.  An escape is a codeword of its total length whose payload is OR-ed in
// from a prefetched load.  513^3: 405 -> 207 us (300x431x517 at 1e-4, where most
// symbols are escapes: 396 -> 257 us); a 129^2 field, whose last group ran symbol
// by symbol from global memory, 24 -> 9 us.
constexpr unsigned kEncOutWords = 832;     // words a group may take in shared memory (26 bits per symbol)
constexpr int kEncWarps = 8;
// returns its bits, or 0 (nothing done) where the group needs the general path: a
// codeword above 26 bits, an escape above 32 bits in all, more than kEncOutWords
// words.  PART: the stream's last group, cnt < 1024 symbols; its lanes may hold
// few bits or none, so its words are merged in cleared shared memory.  more: the
// warp's next group goes on in the last word, which is stored, not merged.
// look(s): the entry of symbol s.
template <bool PART, typename S, typename Look>
__device__ __forceinline__ unsigned enc_fast_group(Look look, uint32_t *buf, const S *sym, unsigned cnt,
                                                   const long long *esc, uint32_t e0, uint32_t code0, unsigned ew,
                                                   unsigned long long start, uint32_t *words, bool more)
{
    const unsigned lane = threadIdx.x & 31;
    uint32_t e[32];
    unsigned mb = 0, worst = 0;
    if (PART) {
        S x[32];
#pragma unroll
        for (unsigned q = 0; q < 32; q++) x[q] = 32 * lane + q < cnt ? sym[32 * lane + q] : (S)0;
#pragma unroll
        for (unsigned q = 0; q < 32; q++) e[q] = 32 * lane + q < cnt ? look(x[q]) : 0u;
    } else {
        const uint4 *v = reinterpret_cast<const uint4 *>(sym + 32 * lane);
        constexpr int per = 4 / sizeof(S), nv = 2 * sizeof(S);   // symbols per word, 16-byte loads
        uint4 x[nv];
#pragma unroll
        for (int u = 0; u < nv; u++) x[u] = __ldcs(v + u);
#pragma unroll
        for (int u = 0; u < nv; u++) {
            const uint32_t y[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
#pragma unroll
            for (int k = 0; k < 4; k++)
#pragma unroll
                for (int h = 0; h < per; h++)
                    e[per * (4 * u + k) + h] = look((y[k] >> (8 * sizeof(S) * h)) & (sizeof(S) == 1 ? 0xFFu : 0xFFFFu));
        }
    }
#pragma unroll
    for (int q = 0; q < 32; q++) { mb += e[q] & 63u; worst = max(worst, e[q]); }
    unsigned xb = mb;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, xb, o);
        if (lane >= (unsigned)o) xb += y;
    }
    const unsigned s0 = (unsigned)(start & 31), endb = s0 + __shfl_sync(0xffffffffu, xb, 31);
    const unsigned W = (endb + 31) >> 5;
    if (__any_sync(0xffffffffu, worst == kPackLong) || W > kEncOutWords) return 0u;
    if (PART) {
        for (unsigned i = lane; i < W; i += 32) buf[i] = 0u;
        __syncwarp();
    }
    const unsigned at = s0 + xb - mb;
    unsigned n = at & 31u;
    uint32_t hi = 0, lo = 0;
    uint32_t *o = buf + (at >> 5);
    // low words of the escaped codes, eight symbols ahead of their use
    const int *el = reinterpret_cast<const int *>(esc + 32 * lane);
    int zn[8], zc[8];
    auto fetch = [&](int b) {
#pragma unroll
        for (int q = 0; q < 8; q++) {
            zn[q] = 0;
            if (e[8 * b + q] == e0) zn[q] = __ldcs(el + 2 * (8 * b + q));
        }
    };
    fetch(0);
#pragma unroll
    for (int b = 0; b < 4; b++) {
#pragma unroll
        for (int q = 0; q < 8; q++) zc[q] = zn[q];
        if (b < 3) fetch(b + 1);
#pragma unroll
        for (int q = 0; q < 8; q++) {
            const uint32_t f = e[8 * b + q];
            const unsigned L = f & 63u;
            uint32_t c = f >> 6;
            // zigzag(k) of an escape fits its payload width (below 32 bits)
            if (f == e0) c = (code0 << ew) | (((uint32_t)zc[q] << 1) ^ (uint32_t)(zc[q] >> 31));
            hi = __funnelshift_lc(lo, hi, L);
            lo = __funnelshift_lc(0u, lo, L) | c;
            n += L;
            if (n >= 32u) {
                n -= 32u;
                const uint32_t v = __funnelshift_r(lo, hi, n);
                if (PART) atomicOr(o++, v);
                else *o++ = v;
            }
        }
    }
    // the word a lane ends in is the next lane's first one (every lane of a
    // complete group holds at least 32 bits); the last lane's is stored alone
    __syncwarp();
    if (n) {
        const uint32_t last = lo << (32u - n);
        if (!PART && lane == 31) *o = last;
        else if (last) atomicOr(o, last);
    }
    __syncwarp();
    uint32_t *g = words + (start >> 5);
    for (unsigned i = lane; i < W; i += 32) {
        const uint32_t v = buf[i];
        // the group's first and last words are shared with its neighbours (zeroed before)
        if ((i == 0 && s0) || (i + 1 == W && (endb & 31u) && !more)) atomicOr(g + i, v);
        else g[i] = v;
    }
    __syncwarp();
    return endb - s0;
}

// S: type of the symbols; SM: the packed codeword table (pack_code) fits shared
// memory, else it is read through the caches; PIECES: groups above 1024 symbols, which
// a warp takes in pieces of 1024 (chunks of 32768 as runs of 1024 symbols a lane: 5000
// symbols 294 us, in pieces 15; with the loop over pieces for every chunk size 513^3
// compression took 1415 us instead of 1396)
template <typename S, bool SM, bool PIECES>
__global__ void __launch_bounds__(32 * kEncWarps, 3) enc_write_kernel(EncodeArgs a)
{
    extern __shared__ __align__(16) uint32_t esm32[];
    next_begin();
    if (block_skip(&a.sc->status)) return;
    const S *__restrict__ sym = reinterpret_cast<const S *>(a.sym);
    uint32_t *spk = esm32;
    // per warp: a group's finished words
    const unsigned Dv = (a.D + 3) / 4;   // the table's space in the scratch is a multiple of 256 bytes
    const unsigned warp = (unsigned)warp_index();
    uint32_t *sw = esm32 + (SM ? 4 * Dv : 0) + warp * kEncOutWords;
    const long long *__restrict__ esc = a.esc;
    const int ew = esc ? (int)a.sc->esc_w : 0;       // escape payload width
    const unsigned L0 = a.len[0];
    const uint32_t code0 = (uint32_t)a.code[0];
    // entry of an escape: its total length, the payload comes from its code
    const uint32_t e0 = !ew ? 0xFFFFFFFEu : L0 + ew <= 32 ? L0 + ew : kPackLong;
    if (SM) {
        const uint4 *src = reinterpret_cast<const uint4 *>(a.pack);
        constexpr int U = 8;
        for (unsigned i0 = threadIdx.x; i0 < Dv; i0 += U * blockDim.x) {
            uint4 v[U];
#pragma unroll
            for (int u = 0; u < U; u++) v[u] = src[min(i0 + u * blockDim.x, Dv - 1)];
#pragma unroll
            for (int u = 0; u < U; u++)
                if (i0 + u * blockDim.x < Dv) reinterpret_cast<uint4 *>(spk)[i0 + u * blockDim.x] = v[u];
        }
        __syncthreads();
        if (threadIdx.x == 0 && ew && L0) spk[0] = e0;
    }
    __syncthreads();
    auto look = [&](unsigned sv) -> uint32_t {
        if (SM) return spk[sv];
        return ew && sv == 0 ? e0 : __ldg(a.pack + sv);
    };
    // (codeword, length) of symbol s
    auto cw_of = [&](unsigned sv, unsigned long long &cw, int &L) {
        const uint32_t e = ew && sv == 0 ? kPackLong : look(sv);
        if (e != kPackLong) { cw = e >> 6; L = (int)(e & 63u); }
        else { cw = a.code[sv]; L = a.len[sv]; }
    };
    const unsigned long long nch = (a.N + a.K - 1) / a.K;
    uint32_t *__restrict__ words = enc_words(a, nch, a.sc->total_bits);
    const unsigned lane = threadIdx.x & 31;
    const unsigned r = enc_group(a.K);
    const unsigned long long G = (unsigned long long)a.K * r;   // symbols per warp group
    const unsigned long long ngr = (a.N + G - 1) / G;
    const unsigned P = PIECES ? 1024u : (unsigned)G;
    const unsigned long long wg = blockIdx.x * (unsigned long long)(blockDim.x >> 5) + warp;
    const unsigned long long nw = (unsigned long long)gridDim.x * (blockDim.x >> 5);
    for (unsigned long long c = wg; c < ngr; c += nw) {
        const unsigned long long gend = c * G + G < a.N ? c * G + G : a.N;
        const bool complete = gend - c * G == G;
        unsigned long long beg = c * G, at = a.chunk_bits[c * r];
    do {
        const unsigned long long end = beg + P < gend ? beg + P : gend;
        const unsigned cnt = (unsigned)(end - beg);
        const bool more = PIECES && end < gend;
        if (PIECES || G == 1024) {
            const long long *ge = esc ? esc + beg : nullptr;
            const unsigned bits =
                cnt == 1024 ? enc_fast_group<false>(look, sw, sym + beg, cnt, ge, e0, code0, (unsigned)ew, at, words, more)
                            : enc_fast_group<true>(look, sw, sym + beg, cnt, ge, e0, code0, (unsigned)ew, at, words, more);
            if (PIECES) at += bits;
            if (bits) continue;
        }
        // the words inside a complete group above 1024 symbols are not zeroed before, so
        // every lane that takes part in a piece of it has 32 symbols
        const unsigned spl = PIECES ? (complete ? 32u : (cnt + 31) >> 5) : (unsigned)(G >> 5);
        const unsigned last = PIECES && complete ? cnt / 32 - 1 : 31u;   // the last lane that takes part
        unsigned long long m0 = beg + (unsigned long long)lane * spl, m1 = m0 + spl;
        if (m0 > end) m0 = end;
        if (m1 > end) m1 = end;
        unsigned long long mb = 0;
        // the general path: symbol by symbol, four in flight
#pragma unroll 4
        for (unsigned long long i = m0; i < m1; i++) {
            const unsigned sv = sym[i];
            unsigned long long cw;
            int L;
            cw_of(sv, cw, L);
            mb += L + (sv == 0 ? ew : 0);
        }
        unsigned long long xb = mb;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long yb = __shfl_up_sync(0xffffffffu, xb, o);
            if ((int)lane >= o) xb += yb;
        }
        const unsigned long long start = at + xb - mb;
        if (PIECES) at += __shfl_sync(0xffffffffu, xb, 31);
        unsigned long long acc = 0;
        unsigned nacc = (unsigned)(start & 31);
        unsigned long long widx = start >> 5;
        const unsigned long long fidx = widx;
        uint32_t firstw = 0;
        bool have_first = false;
        // append the low L bits of cw (L <= 64), most significant first
        auto emit = [&](unsigned long long cw, int L) {
            if (L <= 32) {
                // nacc < 32 here, so the codeword fits the 64-bit accumulator whole
                acc |= cw << (64 - nacc - L);
                nacc += L;
                if (nacc >= 32) {
                    const uint32_t wv = (uint32_t)(acc >> 32);
                    if (!have_first) { firstw = wv; have_first = true; }
                    else words[widx] = wv;
                    widx++;
                    acc <<= 32;
                    nacc -= 32;
                }
                return;
            }
            while (L > 0) {
                const int take = L > 32 ? 32 : L;
                const unsigned long long part = (cw >> (L - take)) & ((1ULL << take) - 1);
                L -= take;
                acc |= part << (64 - nacc - take);
                nacc += take;
                if (nacc >= 32) {
                    const uint32_t wv = (uint32_t)(acc >> 32);
                    if (!have_first) { firstw = wv; have_first = true; }
                    else words[widx] = wv;
                    widx++;
                    acc <<= 32;
                    nacc -= 32;
                }
            }
        };
        // codeword (cw, L) of symbol s at stream index i, with its escape payload
        auto put_cw = [&](unsigned long long cw, int L, unsigned s, unsigned long long i) {
            if (ew && s == 0) {
                // codeword and zigzag(k) in ew bits, in one emission when they fit 64 bits
                const unsigned long long z = zigzag(esc[i]);
                if (L + ew <= 64) {
                    cw = (cw << ew) | z;
                    L += ew;
                } else {
                    emit(cw, L);
                    cw = z;
                    L = ew;
                }
            }
            emit(cw, L);
        };
        for (unsigned long long i = m0; i < m1; i += 4) {
            // the loads of four symbols first, then their emissions
            unsigned sv[4];
            unsigned long long cv[4];
            int lv[4];
            const int nu = (int)(m1 - i < 4 ? m1 - i : 4);
#pragma unroll
            for (int u = 0; u < 4; u++) sv[u] = u < nu ? sym[i + u] : 0u;
#pragma unroll
            for (int u = 0; u < 4; u++) if (u < nu) cw_of(sv[u], cv[u], lv[u]);
#pragma unroll
            for (int u = 0; u < 4; u++) if (u < nu) put_cw(cv[u], lv[u], sv[u], i + u);
        }
        const uint32_t lastw = (uint32_t)(acc >> 32);
        const bool has_last = nacc > 0;
        // a complete group whose every lane holds >= 32 bits (always true with 32
        // symbols per lane): lane i's last partial word is lane i+1's first word
        const bool full = __all_sync(0xffffffffu, complete && (mb >= 32 || lane > last));
        if (full) {
            const uint32_t prev = __shfl_up_sync(0xffffffffu, lastw, 1);
            const bool sh = (start & 31) != 0;
            if (lane > 0 && sh) firstw |= prev;
            if (have_first) {
                if (lane == 0 && sh) atomicOr(&words[fidx], firstw);
                else words[fidx] = firstw;
            }
            if (lane == last && has_last) {
                if (more) words[widx] = lastw;
                else atomicOr(&words[widx], lastw);
            }
        } else {
            if (have_first) {
                if (start & 31) atomicOr(&words[fidx], firstw);
                else words[fidx] = firstw;
            }
            if (has_last) atomicOr(&words[widx], lastw);
        }
        if (PIECES) __syncwarp();
    } while (PIECES && (beg += P) < gend);
    }
}


// Container header, bins, coordinates, code lengths and the zero gaps before
// the chunk table and the bitstream.  One block: what bounds it is latency, so
// the scalars are loaded together and put into words, one warp forms the CRC,
// and the code lengths move a word per thread with eight words' loads in
// flight (byte by byte, each load waiting for the store before it, they took
// most of the 19-23 us; now 5-7 us).
constexpr int kHeaderThreads = 512;
__device__ __forceinline__ void header_body(const HeaderArgs &h, const uint8_t *__restrict__ len, Scalars *sc,
                                            uint8_t *__restrict__ out)
{
    if (block_skip(&sc->status)) return;
    const unsigned tid = threadIdx.x, nt = blockDim.x;
    const unsigned s_lo = sc->s_lo, s_hi = sc->s_hi;
    const unsigned long long bits = sc->total_bits;
    const unsigned long long nch = (h.N + h.K - 1) / h.K;
    const Layout lay = container_layout(h.L, h.ncoord, s_lo, s_hi, nch, bits);
    if (tid < 32) {
        __shared__ uint32_t hw[32];
        if (tid == 0) {
            const unsigned long long n_esc = h.hist ? h.hist[0] : 0ULL;
            const unsigned esc_w = sc->esc_w;
            const double tau = sc->tau_abs, mx = sc->maxabs, rms = sqrt(sc->sumsq / (double)h.N);
            auto w64 = [&](int at, unsigned long long v) { hw[at / 4] = (uint32_t)v; hw[at / 4 + 1] = (uint32_t)(v >> 32); };
            auto wd = [&](int at, double v) { w64(at, (unsigned long long)__double_as_longlong(v)); };
            hw[0] = 0x52445048u;   // "HPDR"
            hw[1] = 3;
            hw[2] = (uint32_t)h.dtype;
            hw[3] = (uint32_t)h.ndim;
            for (int k = 0; k < 3; k++) w64(16 + 8 * k, h.dims[k]);
            hw[10] = (uint32_t)h.L;
            hw[11] = (uint32_t)h.mode;
            hw[12] = (uint32_t)h.tol_kind | (h.ncoord ? 0x100u : 0u);
            hw[13] = h.D;
            hw[14] = h.K;
            hw[15] = s_lo;
            wd(64, h.tol);
            wd(72, tau);
            wd(80, mx);
            wd(88, rms);
            w64(96, h.N);
            w64(104, n_esc);
            w64(112, bits);
            hw[30] = s_hi | ((n_esc ? esc_w : 0u) << 16);
            hw[31] = 0;
            sc->n_esc = n_esc;
        }
        __syncwarp();
        const uint32_t w = hw[tid], crc = crc32_warp(w);
        reinterpret_cast<uint32_t *>(out)[tid] = tid == 31 ? crc : w;
    }
    const unsigned long long qend = 128 + 8ULL * (h.L + 1);
    for (int l = tid; l <= h.L; l += nt) reinterpret_cast<double *>(out + 128)[l] = sc->q[l];
    for (unsigned long long i = tid; i < h.ncoord; i += nt) reinterpret_cast<double *>(out + qend)[i] = h.coords[i];
    for (unsigned long long i = qend + 8 * h.ncoord + tid; i < lay.off_len; i += nt) out[i] = 0;
    const unsigned nlen = s_hi - s_lo + 1, nw = nlen / 4;
    const uint8_t *lsrc = len + s_lo;
    uint32_t *lw = reinterpret_cast<uint32_t *>(out + lay.off_len);
    constexpr int U = 4;
    for (unsigned i0 = tid; i0 < nw; i0 += U * nt) {
        uint32_t v[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const unsigned i = min(i0 + u * nt, nw - 1);
            v[u] = (uint32_t)lsrc[4 * i] | ((uint32_t)lsrc[4 * i + 1] << 8) | ((uint32_t)lsrc[4 * i + 2] << 16) |
                   ((uint32_t)lsrc[4 * i + 3] << 24);
        }
#pragma unroll
        for (int u = 0; u < U; u++) if (i0 + u * nt < nw) lw[i0 + u * nt] = v[u];
    }
    for (unsigned i = 4 * nw + tid; i < nlen; i += nt) out[lay.off_len + i] = lsrc[i];
    for (unsigned long long i = lay.off_len + nlen + tid; i < lay.off_chunk; i += nt) out[i] = 0;
    for (unsigned long long i = lay.off_chunk + 8 * nch + tid; i < lay.off_bits; i += nt) out[i] = 0;
}

// one container header per block, then the field's {bytes, status} pair
__device__ __forceinline__ void header_job(const HeaderJob &j)
{
    header_body(j.h, j.len, j.sc, j.out);
    __syncthreads();
    if (threadIdx.x == 0 && j.size_status) {
        j.size_status[0] = j.sc->out_bytes;
        j.size_status[1] = j.sc->status;
    }
}
__global__ void __launch_bounds__(kHeaderThreads) header_kernel(HeaderJob j)
{
    next_begin();
    header_job(j);
}
__global__ void __launch_bounds__(kHeaderThreads) header_batch_kernel(const HeaderJob *jobs)
{
    header_job(jobs[blockIdx.x]);
}

// ---------------------------------------------------------------------------
// Decoder: one thread per chunk, canonical decode with a two-level table and
// a per-length fallback for the longest codewords.
//
// A thread decodes its chunk of K symbols.  It keeps the next bits of the
// chunk MSB-aligned in two 32-bit registers hi:lo (nb valid bits, at least 32
// before every look-up) and the next word of the stream in a third.  A codeword
// of at most 13 bits is one load from the first-level table of every 13-bit
// prefix; one of up to 23 bits is a second load from the table its prefix
// names, indexed by the bits after the prefix; either gives symbol and length,
// with no search.  Every other case (longer codewords, prefixes past the
// second-level budget, escape payloads that do not fit the 32-bit window,
// invalid codes) leaves the loop for an out-of-line routine that reads its
// window from global memory.
//
// What bounds the kernel is the latency of a step (two dependent shared loads
// under load) against the at most 32 warps that 64 registers a thread allow, and
// the instructions of a step, so a step is short and has no divergent branch:
//   - table entries hold their fields where the step uses them: the length in
//     the low bits, the symbol in the high half, flag bits for the unusual cases,
//     and in a second-level pointer the byte offset of its table and the shift
//     that isolates its index;
//   - the stream passes through a ring of 32 words per thread in shared memory
//     ([word][thread], conflict-free), filled once every eight symbols by the
//     32-byte sector prefetched in registers: a step's refill is one predicated
//     shared load, where selecting the word from a register block and reloading
//     the block took most of the 88 instructions a step, and every sector is
//     fetched once (the threads' lines do not fit what is left of L1);
//   - the second-level load, the refill and the store of a sparse escape are
//     predicated (as branches they cost the warp both sides at nearly every
//     step); only the out-of-line cases branch.
// 513^3 at 1e-3: 515 -> 335 us; 300x431x517 at 1e-4, where most symbols are
// escapes: 434 -> 295 us; 64 Mi byte keys: 222 -> 114 us.
//
// An escape whose codeword and payload do not fit 32 bits is three such steps where
// escapes are dense (decode_chunk<3>; out of line, with its code stored alone, as
// sparse ones still are, the 45 million codes of 15x1500x2000 binary64 at 1e-8 took
// 2099 us; in line 303).
//
// Escaped codes: where they are dense (more than one symbol in sixteen) a
// thread keeps the payloads of eight symbols in registers and writes each half
// with an escape as one 32-byte sector: single 8-byte stores scattered over the
// escape array cost a read-modify-write of their sector in DRAM.  The other
// slots of a stored sector carry zeros or stale values; nothing reads the escape
// array where no escape is.  Sparse escapes are stored one by one.
constexpr int kDecThreads = 1024;
constexpr unsigned kRingWords = 32;
constexpr size_t kDecSmem = (4u << kLutBits) + 4 * kSubCap + sizeof(LenTabs) + 4ull * kRingWords * kDecThreads;

// Decoder entries (the staged copy of the look-up tables):
//   leaf                  symbol << 16 | L
//   folded escape         kDecEsc | L          (L = codeword + payload, at most 32)
//   second-level pointer  byte offset << 16 | kDecSub | (32 - index bits)
//   long codeword         kDecSlow | Lmin << 16 | (Lmax - Lmin) << 24
//   unfolded escape       kDecSlow | kDecOpen | L << 16
//   no codeword           kDecSlow
constexpr uint32_t kDecEsc = 0x40u, kDecSlow = 0x80u, kDecSub = 0x100u, kDecOpen = 0x200u;

__device__ __forceinline__ uint32_t ldw(const uint32_t *w, unsigned long long i, unsigned long long n)
{
    return i < n ? __ldg(w + i) : 0u;
}

// one 32-byte sector: a load that does not stay in L1, a store
struct Words8 {
    uint32_t v[8];
};
__device__ __forceinline__ Words8 ldg32(const uint32_t *p)
{
    Words8 r;
    asm volatile("ld.global.nc.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r.v[0]), "=r"(r.v[1]), "=r"(r.v[2]), "=r"(r.v[3]), "=r"(r.v[4]), "=r"(r.v[5]), "=r"(r.v[6]),
                   "=r"(r.v[7])
                 : "l"(p));
    return r;
}
__device__ __forceinline__ void stg32(long long *p, long long a, long long b, long long c, long long d)
{
    asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" :: "l"(p), "l"(a), "l"(b), "l"(c), "l"(d) : "memory");
}
__device__ __forceinline__ uint32_t lds32(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts32(uint32_t addr, uint32_t v)
{
    asm volatile("st.shared.u32 [%0], %1;" :: "r"(addr), "r"(v) : "memory");
}
// predicated shared load and global store (no branch around them)
__device__ __forceinline__ void lds_if(uint32_t &v, uint32_t cond, uint32_t addr)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t@p ld.shared.u32 %0, [%2];\n\t}"
                 : "+r"(v) : "r"(cond), "r"(addr) : "memory");
}
__device__ __forceinline__ void stg_if(long long *dst, uint32_t cond, long long v)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t@p st.global.u64 [%0], %2;\n\t}"
                 :: "l"(dst), "r"(cond), "l"(v) : "memory");
}

// A thread's view of its chunk's words, counted in 32 bits from `base`, the
// 32-byte sector of memory in which the chunk starts (a chunk has at most 32768
// symbols of 126 bits); no word outside the stream is loaded.  rc: ring index of the prefetched word `next`, wr: end
// of the words in the ring, pa: the sector after it.  left: words of the stream
// from base on (words past it read as zero), lvec: the same as far as whole
// sectors can be loaded (0 for a stream that does not start on 16 bytes).
struct BitQueue {
    const uint32_t *base;
    unsigned left, lvec;
    uint32_t ring;            // shared address of this thread's column, kDecThreads words between rows
    unsigned rc, wr;
    Words8 pa;
    uint32_t next;
    __device__ __forceinline__ Words8 sector(unsigned i) const
    {
        if (i + 8 <= lvec) return ldg32(base + i);
        Words8 r;
#pragma unroll
        for (unsigned k = 0; k < 8; k++) r.v[k] = ldw(base, i + k, left);
        return r;
    }
    __device__ __forceinline__ uint32_t addr(unsigned i) const { return ring + (i % kRingWords) * (4 * kDecThreads); }
    __device__ __forceinline__ uint32_t at(unsigned i) const { return lds32(addr(i)); }
    __device__ __forceinline__ void append()
    {
        const uint32_t r = addr(wr);   // wr is a multiple of 8: no wrap inside
#pragma unroll
        for (unsigned k = 0; k < 8; k++) sts32(r + 4 * kDecThreads * k, pa.v[k]);
        wr += 8;
        pa = sector(wr);
    }
    // Eight symbols take at most eight words (32 bits each; longer steps move the
    // queue themselves), so one sector keeps up: with ten words from `next` on
    // before eight symbols, ten are left after this before the next eight.  The
    // two words of the window stay in the ring, for a seek may start in them.
    __device__ __forceinline__ void top_up()
    {
        if (wr - rc + 2 <= kRingWords - 8) append();
    }
    // the first 64 bits from bit pos of base on (at or after the current words)
    __device__ __forceinline__ void seek(unsigned pos, uint32_t &hi, uint32_t &lo, int &nb)
    {
        rc = pos >> 5;
        while ((int)(wr - rc) < 12) append();
        const uint32_t w0 = at(rc), w1 = at(rc + 1);
        const unsigned sh = pos & 31u;
        hi = __funnelshift_l(w1, w0, sh);
        lo = w1 << sh;
        nb = 64 - (int)sh;
        rc += 2;
        next = at(rc);
    }
    __device__ __forceinline__ void start(const uint32_t *w, unsigned long long n, unsigned long long pos, uint32_t &hi,
                                          uint32_t &lo, int &nb)
    {
        // a stream on 16 bytes may start in the middle of a sector: the words before
        // it are not its own and are not loaded
        const bool vec = (reinterpret_cast<uintptr_t>(w) & 15) == 0;
        const long long lead = vec ? (long long)((reinterpret_cast<uintptr_t>(w) & 31) / 4) : 0;
        const long long wb = (((long long)(pos >> 5) + lead) & ~7LL) - lead, l = (long long)n - wb;
        base = w + wb;
        left = l < 0x7FFFFFFFll ? (unsigned)l : 0x7FFFFFFFu;
        lvec = vec ? left : 0u;
        wr = 0;
        if (wb < 0) {
#pragma unroll
            for (int k = 0; k < 8; k++) pa.v[k] = k + wb >= 0 ? ldw(w, (unsigned long long)(k + wb), n) : 0u;
        } else {
            pa = sector(0);
        }
        seek((unsigned)((long long)pos - 32 * wb), hi, lo, nb);
    }
    // bit position of the window, from base
    __device__ __forceinline__ unsigned pos(int nb) const { return (rc << 5) - (unsigned)nb; }
};

// 64 bits of the stream from bit pos (words past the end read as zero)
__device__ __forceinline__ unsigned long long window64(const uint32_t *w, unsigned long long n,
                                                       unsigned long long pos)
{
    const unsigned long long i = pos >> 5;
    const unsigned sh = (unsigned)(pos & 31);
    const unsigned long long hi = (((unsigned long long)ldw(w, i, n)) << 32) | ldw(w, i + 1, n);
    return sh ? (hi << sh) | (ldw(w, i + 2, n) >> (32 - sh)) : hi;
}

struct SlowOut {
    unsigned long long pos;
    uint32_t sv, bad;
};

// A step the table loop does not take: the entry e at pos is a long entry,
// invalid, or an escape whose payload does not fit the 32-bit window.
__device__ __noinline__ SlowOut decode_slow(uint32_t e, unsigned long long pos, const uint32_t *words,
                                            unsigned long long nwords, const LenTabs *T, const uint16_t *symtab,
                                            unsigned nsym, int ew, long long *esc_i)
{
    SlowOut o;
    o.bad = 0;
    const unsigned long long win = window64(words, nwords, pos);
    uint32_t sv = 0;
    unsigned L = (e >> 16) & 0x3Fu;
    if (e & kDecOpen) {
        // the escape's codeword
    } else if (L) {
        const unsigned lmin = L, lmax = L + ((e >> 24) & 0x3Fu);
        L = code_len_in(*T, win, lmin, lmax);
        const unsigned long long off = (win >> (64 - L)) - T->first[L];
        if (off >= T->count[L]) o.bad = 1;
        const unsigned idx = T->start[L] + (unsigned)(off < T->count[L] ? off : 0);
        sv = symtab[idx < nsym ? idx : 0];
    } else {
        o.bad = 1;               // no codeword starts here
        sv = 0;
        L = 1;
    }
    pos += L;
    if (ew && sv == 0) {
        // escape payload: zigzag(k) in ew bits
        const unsigned long long z = window64(words, nwords, pos) >> (64 - ew);
        pos += (unsigned)ew;
        *esc_i = unzigzag(z);
    }
    o.pos = pos;
    o.sv = sv;
    return o;
}

// One chunk: cnt symbols from symbol beg on, from bit pos0 to bit expect.  EW: 0 no escapes,
// 1 sparse ones, 2 dense ones, 3 dense ones of which codewords and payloads do not fit
// 32 bits.  Returns whether the stream was sound.
template <typename S, int EW>
__device__ __forceinline__ bool decode_chunk(const DecodeArgs &a, const HuffScratch &hs, const LenTabs *T, unsigned nsym,
                                             uint32_t lut, uint32_t sub, uint32_t ring, unsigned long long pos0,
                                             unsigned long long expect, unsigned long long beg, unsigned cnt)
{
    const unsigned ew = EW ? a.esc_w : 0u;     // escape payload width (1..63)
    BitQueue q;
    q.ring = ring;
    uint32_t hi, lo;
    int nb;
    q.start(a.words, a.nwords, pos0, hi, lo, nb);
    const unsigned expos = q.pos(nb) + (unsigned)(expect - pos0);
    bool bad = false;
    S *sym = reinterpret_cast<S *>(a.sym) + beg;
    long long *e8 = EW ? a.esc + beg : nullptr;   // escape slots of the current group of eight symbols
    // EW 2: payloads of the group, bit j of emask where there is one; EW 3: of half a
    // group, the high words in z[4..7]
    uint32_t z[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    unsigned emask = 0;
    // drops L <= 32 bits, then refills to at least 32 valid bits (the valid bits are
    // all in hi then)
    auto drop = [&](unsigned L) {
        hi = __funnelshift_lc(lo, hi, L);
        lo = __funnelshift_lc(0u, lo, L);
        nb -= (int)L;
        const bool need = nb < 32;
        const uint32_t ih = q.next >> (nb & 31), il = __funnelshift_r(0u, q.next, nb);
        hi |= need ? ih : 0u;
        lo = need ? il : lo;
        nb += need ? 32 : 0;
        q.rc += need ? 1u : 0u;
        lds_if(q.next, need, q.addr(q.rc));
    };
    // symbol in the high half
    auto step = [&](unsigned j, uint32_t &zj, uint32_t &zh) -> uint32_t {
        uint32_t e = lds32(lut + 4 * (hi >> (32 - kLutBits)));
        // a codeword of up to 23 bits: its second-level entry, indexed by the
        // bits after the prefix (all within hi, nb >= 32)
        lds_if(e, e & kDecSub, sub + (e >> 16) + 4 * ((hi << kLutBits) >> (e & 31u)));
        if (EW == 3 && (e & kDecOpen)) {
            // the escape's codeword, then up to 63 bits of payload: three words at most,
            // and the ring is topped up behind them
            drop((e >> 16) & 0x3Fu);
            const unsigned w0 = min(ew, 32u), w1 = ew - w0;
            const uint32_t p0 = hi >> (32u - w0);
            drop(w0);
            const uint32_t p1 = w1 ? hi >> (32u - w1) : 0u;
            drop(w1);
            zh = w1 ? p0 >> (32u - w1) : 0u;
            zj = w1 ? p0 << w1 | p1 : p0;
            emask |= 1u << j;
            q.top_up();
            return 0u;
        }
        if (e & kDecSlow) {
            long long kv = 0;
            const SlowOut o = decode_slow(e, q.pos(nb), q.base, q.left, T, hs.sorted_sym, nsym, (int)ew, &kv);
            if (EW && o.sv == 0) {
                // at once: its payload may not fit the group's registers
                e8[j] = kv;
                if (EW >= 2) emask |= 0x100u << j;
            }
            bad |= o.bad != 0;
            q.seek((unsigned)o.pos, hi, lo, nb);
            return o.sv << 16;
        }
        const unsigned L = e & 63u;
        if (EW) {
            // folded escape: codeword of L - ew bits, then zigzag(k) in ew < 32 bits
            const uint32_t y = (hi << ((L - ew) & 31u)) >> ((32u - ew) & 31u);
            if (EW >= 2) {
                zj = y;
                if (EW == 3) zh = 0u;
                emask |= ((e / kDecEsc) & 1u) << j;
            } else {
                stg_if(e8 + j, e & kDecEsc, (long long)((int)(y >> 1) ^ -(int)(y & 1u)));
            }
        }
        drop(L);
        return e;
    };
    // the escaped codes of a group: each half with an escape as one 32-byte
    // store; a code stored by its own step (upper mask) keeps its half from being
    // overwritten: the others of that half go one by one
    auto code = [&](unsigned j) -> long long {
        if (EW == 3) return unzigzag((unsigned long long)z[4 + (j & 3u)] << 32 | z[j & 3u]);
        return (long long)((int)(z[j] >> 1) ^ -(int)(z[j] & 1u));
    };
    // (symbols h0..h1 of it)
    auto flush = [&](unsigned h0, unsigned h1) {
#pragma unroll
        for (unsigned h = h0; h < h1; h += 4) {
            const unsigned m = (emask >> h) & 0xFu;
            if (!m) continue;
            if ((emask >> (8 + h)) & 0xFu) {
#pragma unroll
                for (unsigned j = 0; j < 4; j++) stg_if(e8 + h + j, (m >> j) & 1u, code(h + j));
            } else {
                stg32(e8 + h, code(h), code(h + 1), code(h + 2), code(h + 3));
            }
        }
        emask = 0;
    };
    // eight symbols per store (K is a multiple of 128)
    for (unsigned g = cnt / 8; g; g--) {
        uint32_t o[4];   // pairs: two 16-bit symbols, or two bytes in the low half
        q.top_up();
#pragma unroll
        for (unsigned j = 0; j < 8; j += 2) {
            if (EW == 3 && j == 4) {
                if (emask) flush(0, 4);
                q.top_up();
            }
            const unsigned i = EW == 3 ? j & 3u : j;
            const uint32_t v0 = step(j, z[i], z[EW == 3 ? 4 + i : 0]), v1 = step(j + 1, z[i + 1], z[EW == 3 ? 5 + i : 0]);
            o[j / 2] = __byte_perm(v0, v1, sizeof(S) == 2 ? 0x7632 : 0x0062);
        }
        // streaming store: the symbols are written once and read by the next
        // kernel, so they should not push the bitstream out of L2
        if (sizeof(S) == 2) __stcs(reinterpret_cast<uint4 *>(sym), make_uint4(o[0], o[1], o[2], o[3]));
        else __stcs(reinterpret_cast<uint2 *>(sym),
                    make_uint2(__byte_perm(o[0], o[1], 0x5410), __byte_perm(o[2], o[3], 0x5410)));
        sym += 8;
        if (EW == 2 && emask) flush(0, 8);
        if (EW == 3 && emask) flush(4, 8);
        if (EW) e8 += 8;
    }
    // a last group of fewer than eight: its escapes one by one
    q.top_up();
    for (unsigned j = 0; j < cnt % 8; j++) {
        uint32_t y = 0, yh = 0;
        sym[j] = (S)(step(j, y, yh) >> 16);
        if (EW >= 2 && ((emask >> j) & 1u))
            e8[j] = EW == 3 ? unzigzag((unsigned long long)yh << 32 | y) : (long long)((int)(y >> 1) ^ -(int)(y & 1u));
    }
    return !bad && q.pos(nb) == expos;
}

// S: type of the symbols; bytes carry no escapes (the lossless stage)
template <typename S>
__global__ void __launch_bounds__(kDecThreads, 1) decode_kernel(DecodeArgs a_in, HuffScratch hs)
{
    DecodeArgs a = a_in;
    const unsigned long long nch = (a.N + a.K - 1) / a.K;
    next_begin();
    if (blockIdx.x >= nch) return;
    if (block_skip(hs.status)) return;
    if (a.dh) {
        const DevHdr h = *a.dh;
        a.words = reinterpret_cast<const uint32_t *>(a.base + h.off_bits);
        a.nwords = h.nwords;
        a.chunk = reinterpret_cast<const unsigned long long *>(a.base + h.off_chunk);
        a.total_bits = h.total_bits;
        a.esc_w = h.esc_w;
        a.n_esc = h.n_esc;
        if (h.esc_w == 0) a.esc = nullptr;
    }
    extern __shared__ __align__(16) unsigned char dsm[];
    uint32_t *lut = reinterpret_cast<uint32_t *>(dsm);                       // [1 << kLutBits]
    uint32_t *sub = lut + (1u << kLutBits);                                   // [kSubCap]
    LenTabs *T = reinterpret_cast<LenTabs *>(sub + kSubCap);
    uint32_t *ring = reinterpret_cast<uint32_t *>(T + 1);                      // [kRingWords][kDecThreads]
    const unsigned nsym = *hs.nsym;
    const unsigned nsub = *hs.nsub < kSubCap ? *hs.nsub : kSubCap;
    int open = 0;   // whether an escape's codeword and payload do not fit 32 bits
    {
        // escape entries take their payload width into their length when both fit 32 bits
        const unsigned ewc = a.esc ? a.esc_w : 0u;
        auto entry = [&](uint32_t e) -> uint32_t {
            if (e == 0) return kDecSlow;
            const unsigned L = (e >> 16) & 0x3Fu;
            if (e & kLongFlag) return kDecSlow | (L << 16) | (((e >> 24) & 0x3Fu) << 24);
            if (e & kSubFlag) return ((e & 0x3FFFu) << 18) | kDecSub | (32u - ((e >> 16) & 0xFu));
            if (ewc && (e & 0xFFFFu) == 0) {
                if (L + ewc <= 32) return kDecEsc | (L + ewc);
                open = 1;
                return kDecSlow | kDecOpen | (L << 16);
            }
            return (e << 16) | L;
        };
        auto four = [&](uint4 v) { return make_uint4(entry(v.x), entry(v.y), entry(v.z), entry(v.w)); };
        const uint4 *g1 = reinterpret_cast<const uint4 *>(hs.lut1), *g2 = reinterpret_cast<const uint4 *>(hs.lut_sub);
        uint4 *d1 = reinterpret_cast<uint4 *>(lut), *d2 = reinterpret_cast<uint4 *>(sub);
        constexpr unsigned N1 = (1u << kLutBits) / 4 / kDecThreads, N2 = kSubCap / 4 / kDecThreads;
        uint4 v1[N1], v2[N2];
#pragma unroll
        for (unsigned u = 0; u < N1; u++) v1[u] = g1[threadIdx.x + u * kDecThreads];
#pragma unroll
        for (unsigned u = 0; u < N2; u++)
            if (4 * (threadIdx.x + u * kDecThreads) < nsub) v2[u] = g2[threadIdx.x + u * kDecThreads];
#pragma unroll
        for (unsigned u = 0; u < N1; u++) d1[threadIdx.x + u * kDecThreads] = four(v1[u]);
#pragma unroll
        for (unsigned u = 0; u < N2; u++)
            if (4 * (threadIdx.x + u * kDecThreads) < nsub) d2[threadIdx.x + u * kDecThreads] = four(v2[u]);
    }
    if (threadIdx.x < 64) {
        T->first[threadIdx.x] = hs.first[threadIdx.x];
        T->lim[threadIdx.x] = hs.lim[threadIdx.x];
        T->start[threadIdx.x] = hs.start[threadIdx.x];
        T->count[threadIdx.x] = hs.count[threadIdx.x];
    }
    open = __syncthreads_or(open);
    const int mode = !a.esc || !a.esc_w ? 0 : a.n_esc * 16 > a.N ? (open ? 3 : 2) : 1;
    const uint32_t lut_a = smem_u32(lut), sub_a = smem_u32(sub), ring_a = smem_u32(ring + threadIdx.x);
    // chunks interleave over the blocks so that every SM gets a share
    for (unsigned long long c = blockIdx.x + (unsigned long long)gridDim.x * threadIdx.x; c < nch;
         c += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned long long pos0 = a.chunk[c];
        const unsigned long long expect = (c + 1 < nch) ? a.chunk[c + 1] : a.total_bits;
        bool ok = pos0 <= a.total_bits && expect <= a.total_bits && pos0 <= expect;
        const unsigned long long beg = c * a.K;
        const unsigned cnt = (unsigned)(beg + a.K < a.N ? a.K : a.N - beg);
        // a chunk of more bits than its symbols can have is not sound either
        ok = ok && expect - pos0 <= 126ull * a.K;
        if (ok) {
            if (sizeof(S) == 1 || mode == 0) ok = decode_chunk<S, 0>(a, hs, T, nsym, lut_a, sub_a, ring_a, pos0, expect, beg, cnt);
            else if (mode == 1) ok = decode_chunk<S, 1>(a, hs, T, nsym, lut_a, sub_a, ring_a, pos0, expect, beg, cnt);
            else if (mode == 3) ok = decode_chunk<S, 3>(a, hs, T, nsym, lut_a, sub_a, ring_a, pos0, expect, beg, cnt);
            else ok = decode_chunk<S, 2>(a, hs, T, nsym, lut_a, sub_a, ring_a, pos0, expect, beg, cnt);
        }
        if (!ok) atomicExch(hs.status, (unsigned)DS_FORMAT);
    }
}

__global__ void __launch_bounds__(256)
hist_kernel(const uint16_t *sym, unsigned long long N, unsigned D, unsigned long long *hist,
            unsigned *status)
{
    extern __shared__ unsigned hsm[];
    const bool sm = D <= 16384;
    if (sm) for (unsigned i = threadIdx.x; i < D; i += blockDim.x) hsm[i] = 0;
    __syncthreads();
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < N;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        unsigned s = sym[i];
        if (s >= D) { atomicExch(status, (unsigned)DS_ARG); continue; }
        if (sm) atomicAdd(&hsm[s], 1u); else atomicAdd(&hist[s], 1ULL);
    }
    __syncthreads();
    if (sm)
        for (unsigned i = threadIdx.x; i < D; i += blockDim.x)
            if (hsm[i]) atomicAdd(&hist[i], (unsigned long long)hsm[i]);
}

// Histogram of bytes.  Lane l of every warp counts in its own column of
// [256][32] shared counters, so the frequent bytes of a warp neither collide nor
// serialize (one counter per byte had the lanes of a warp queue on a few hot
// ones: 198 us for 64 Mi bytes); a thread takes 64 bytes a turn in four 16-byte
// loads.  n: bytes; in is 16-byte aligned.  64 Mi bytes: 198 -> 18 us.
constexpr int kHistByteThreads = 512;
__global__ void __launch_bounds__(kHistByteThreads)
hist_bytes_kernel(const uint8_t *__restrict__ in, unsigned long long n, unsigned long long *hist)
{
    __shared__ unsigned c[256 * 32];
    const unsigned tid = threadIdx.x, lane = tid & 31;
    for (unsigned i = tid; i < 256 * 32; i += kHistByteThreads) c[i] = 0;
    __syncthreads();
    unsigned *mine = c + lane;
    const uint4 *v = reinterpret_cast<const uint4 *>(in);
    const unsigned long long nv = n / 16, step = (unsigned long long)gridDim.x * kHistByteThreads;
    constexpr int U = 4;
    for (unsigned long long i0 = blockIdx.x * (unsigned long long)kHistByteThreads + tid; i0 < nv; i0 += U * step) {
        uint4 x[U];
#pragma unroll
        for (int u = 0; u < U; u++) if (i0 + u * step < nv) x[u] = __ldcs(v + i0 + u * step);
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (i0 + u * step >= nv) continue;
            const unsigned y[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
#pragma unroll
            for (int q = 0; q < 16; q++) atomicAdd(&mine[((y[q >> 2] >> (8 * (q & 3))) & 0xFFu) * 32], 1u);
        }
    }
    if (blockIdx.x == 0 && tid < n % 16) atomicAdd(&mine[(unsigned)in[nv * 16 + tid] * 32], 1u);
    __syncthreads();
    for (unsigned b = tid; b < 256; b += kHistByteThreads) {
        unsigned long long s = 0;
        for (unsigned k = 0; k < 32; k++) s += c[b * 32 + ((k + b) & 31)];
        if (s) atomicAdd(&hist[b], s);
    }
}

// Header of a lossless container, the code lengths and the zero gaps around the
// chunk table, by one block; nothing where the status is set.
__global__ void __launch_bounds__(256) lossless_header_kernel(LosslessHeader h, const uint8_t *__restrict__ len,
                                                              const Scalars *sc, uint8_t *__restrict__ out)
{
    if (sc->status) return;
    const unsigned tid = threadIdx.x;
    if (tid < 32) {
        const unsigned long long f[4] = {h.n, sc->total_bits, h.off_chunk, h.off_bits};
        uint32_t w = 0;
        if (tid == 0) w = 0x4C445048u;   // "HPDL"
        else if (tid == 1) w = 1;
        else if (tid == 2) w = h.key_bytes;
        else if (tid == 3) w = h.D;
        else if (tid == 4) w = h.K;
        else if (tid >= 6 && tid < 14) w = (uint32_t)(f[(tid - 6) / 2] >> (32 * (tid & 1)));
        // the 15 words before the CRC take the last 15 powers of a 31-word message
        const uint32_t x = __shfl_sync(0xffffffffu, w, (int)tid - 16), crc = crc32_words(x, 16);
        if (tid < 15) reinterpret_cast<uint32_t *>(out)[tid] = w;
        if (tid == 15) reinterpret_cast<uint32_t *>(out)[15] = crc;
    }
    for (unsigned i = tid; i < h.D; i += 256) out[64 + i] = len[i];
    for (unsigned long long i = 64 + h.D + tid; i < h.off_chunk; i += 256) out[i] = 0;
    for (unsigned long long i = h.off_chunk + 8 * h.nch + tid; i < h.off_bits; i += 256) out[i] = 0;
}

// Histogram of an alphabet above 16384 symbols (up to 65536): two 16-bit
// counters per 32-bit shared word, 128 KB.  A block counts at most 32768 keys
// per round, so no counter carries into its neighbour, then adds the nonzero
// counts to the global histogram and clears its words.
constexpr int kHistWideThreads = 1024;
constexpr unsigned kHistWideRound = 32u * kHistWideThreads;
__global__ void __launch_bounds__(kHistWideThreads, 1)
hist_wide_kernel(const uint16_t *sym, unsigned long long N, unsigned D, unsigned long long *hist, unsigned *status)
{
    extern __shared__ unsigned hw[];
    const unsigned nw = (D + 1) / 2;
    for (unsigned i = threadIdx.x; i < nw; i += blockDim.x) hw[i] = 0;
    __syncthreads();
    for (unsigned long long r0 = blockIdx.x * (unsigned long long)kHistWideRound; r0 < N;
         r0 += (unsigned long long)gridDim.x * kHistWideRound) {
        const unsigned long long r1 = r0 + kHistWideRound < N ? r0 + kHistWideRound : N;
        if (r1 - r0 == kHistWideRound && ((uintptr_t)(sym + r0) & 15) == 0) {
            // a full round: four 16-byte loads (32 keys) per thread
            const uint4 *v = reinterpret_cast<const uint4 *>(sym + r0);
            uint4 x[4];
#pragma unroll
            for (int u = 0; u < 4; u++) x[u] = v[threadIdx.x + u * kHistWideThreads];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const unsigned w4[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
#pragma unroll
                for (int q = 0; q < 8; q++) {
                    const unsigned s = (w4[q >> 1] >> (16 * (q & 1))) & 0xFFFFu;
                    if (s >= D) { atomicExch(status, (unsigned)DS_ARG); continue; }
                    atomicAdd(&hw[s >> 1], (s & 1) ? 0x10000u : 1u);
                }
            }
        } else {
            for (unsigned long long i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
                const unsigned s = sym[i];
                if (s >= D) { atomicExch(status, (unsigned)DS_ARG); continue; }
                atomicAdd(&hw[s >> 1], (s & 1) ? 0x10000u : 1u);
            }
        }
        __syncthreads();
        for (unsigned i = threadIdx.x; i < nw; i += blockDim.x) {
            const unsigned w = hw[i];
            if (w) {
                if (w & 0xFFFFu) atomicAdd(&hist[2 * i], (unsigned long long)(w & 0xFFFFu));
                if (w >> 16) atomicAdd(&hist[2 * i + 1], (unsigned long long)(w >> 16));
                hw[i] = 0;
            }
        }
        __syncthreads();
    }
}

PerDeviceOnce g_attr_done;
cudaError_t set_attrs_now()
{
    cudaError_t e = cudaFuncSetAttribute(rank_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kSmemKeys * 8);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(merge_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemKeys * 16);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(codebook_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCodebookSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(codebook_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kCodebookSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(dec_tables_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kTabSmem + 65536);
    const auto smem = [&](auto kern, int bytes) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    };
    smem(enc_write_kernel<uint16_t, true, false>, 200 * 1024);
    smem(enc_write_kernel<uint16_t, true, true>, 200 * 1024);
    smem(enc_count_kernel<uint16_t>, 65536);
    smem(decode_kernel<uint16_t>, (int)kDecSmem);
    smem(decode_kernel<uint8_t>, (int)kDecSmem);
    return e;
}
cudaError_t set_attrs() { return once_per_device(g_attr_done, set_attrs_now); }

}  // namespace

size_t huff_scratch_bytes(unsigned int D)
{
    size_t d = D;
    size_t b = 0;
    auto add = [&](size_t x) { b += (x + 255) & ~size_t(255); };
    add(8 * d); add(8 * d); add(8 * d); add(4 * d);    // keys, keys2, sorted, rank
    add(4 * 2 * d); add(4 * 4 * d); add(4 * 4 * d);    // parent, anc, dep
    add(8 * d); add(8 * d);                            // leafw, intw
    add(4); add(8 * 64); add(4 * 64); add(4 * 64);     // nsym, first, count, start
    add(d); add(8 * d); add(2 * d); add(4u << kLutBits);
    add(8 * 64);
    add(4 * kSubCap); add(4); add(4 * d);
    return b;
}

void huff_scratch_carve(void *base, unsigned int D, Scalars *sc, HuffScratch *hs)
{
    char *p = (char *)base;
    size_t d = D;
    auto take = [&](size_t x) { char *r = p; p += (x + 255) & ~size_t(255); return (void *)r; };
    hs->keys = (unsigned long long *)take(8 * d);
    hs->keys2 = (unsigned long long *)take(8 * d);
    hs->sorted = (unsigned long long *)take(8 * d);
    hs->rank = (unsigned *)take(4 * d);
    hs->parent = (unsigned *)take(4 * 2 * d);
    hs->anc = (unsigned *)take(4 * 4 * d);
    hs->dep = (unsigned *)take(4 * 4 * d);
    hs->leafw = (unsigned long long *)take(8 * d);
    hs->intw = (unsigned long long *)take(8 * d);
    hs->nsym = (unsigned *)take(4);
    hs->first = (unsigned long long *)take(8 * 64);
    hs->count = (unsigned *)take(4 * 64);
    hs->start = (unsigned *)take(4 * 64);
    hs->len = (uint8_t *)take(d);
    hs->code = (unsigned long long *)take(8 * d);
    hs->sorted_sym = (uint16_t *)take(2 * d);
    hs->lut1 = (uint32_t *)take(4u << kLutBits);
    hs->lim = (unsigned long long *)take(8 * 64);
    hs->lut_sub = (uint32_t *)take(4 * kSubCap);
    hs->nsub = (unsigned *)take(4);
    hs->pack = (uint32_t *)take(4 * d);
    hs->status = &sc->status;
    hs->s_lo = &sc->s_lo;
    hs->s_hi = &sc->s_hi;
}

cudaError_t launch_codebook(const unsigned long long *hist, unsigned int D, const HuffScratch &hs,
                            cudaStream_t s)
{
    cudaError_t e = set_attrs();
    if (e != cudaSuccess) return e;
    if (D <= kFusedMaxD) {
        count_launch();
        return launch_next(codebook_kernel, 1, 1024, kCodebookSmem, s, hist, D, hs);
    }
    compact_kernel<<<1, 1024, 0, s>>>(hist, D, hs.keys, hs.nsym, hs.s_lo, hs.s_hi);
    rank_kernel<<<kRankBlocks, 256, kSmemKeys * 8, s>>>(hs.keys, hs.nsym, hs.sorted, nullptr);
    merge_kernel<<<1, 1024, kSmemKeys * 16, s>>>(hs, D);
    rank_kernel<<<kRankBlocks, 256, kSmemKeys * 8, s>>>(hs.keys2, hs.nsym, nullptr, hs.rank);
    assign_kernel<<<64, 256, 0, s>>>(hs);
    count_launch(5);
    return cudaGetLastError();
}

cudaError_t launch_decode_tables(const TabArgs &a, const HuffScratch &hs, cudaStream_t s)
{
    cudaError_t e = set_attrs();
    if (e != cudaSuccess) return e;
    count_launch();
    return launch_next(dec_tables_kernel, kTabBlocks, kTabThreads, kTabSmem + a.D, s, a, hs);
}

cudaError_t launch_encode(const EncodeArgs &a, cudaStream_t s)
{
    cudaError_t e = set_attrs();
    if (e != cudaSuccess) return e;
    // eight warps a block, a group each: no more blocks than the stream has groups
    const unsigned long long groups = ((a.N + a.K - 1) / a.K + enc_group(a.K) - 1) / enc_group(a.K);
    const unsigned nb = (unsigned)std::min<unsigned long long>(kEncBlocks, (groups + 7) / 8);
    const bool code_sm = a.D <= (unsigned)kSmemCodes;
    const size_t smc = (a.D + 15) / 16 * 16, smw = ((code_sm ? (size_t)(a.D + 3) / 4 * 4 : 0) + kEncWarps * kEncOutWords) * 4;
    e = launch_next(a.bytes ? enc_count_kernel<uint8_t> : enc_count_kernel<uint16_t>, nb, 256, smc, s, a);
    if (e == cudaSuccess) e = launch_next(enc_scan_kernel, nb, 256, 0, s, a);
    if (e != cudaSuccess) return e;
    const auto write = [&](auto kern) -> cudaError_t {
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * kEncWarps, smw) != cudaSuccess) {
            cudaGetLastError();
            per_sm = 3;
        }
        const unsigned long long full = (unsigned long long)sm_count() * std::max(1, per_sm);
        return launch_next(kern, (unsigned)std::min(full, (groups + kEncWarps - 1) / kEncWarps), 32 * kEncWarps, smw, s, a);
    };
    count_launch(3);
    if (a.K > 1024) {
        if (a.bytes) return write(enc_write_kernel<uint8_t, true, true>);
        return code_sm ? write(enc_write_kernel<uint16_t, true, true>) : write(enc_write_kernel<uint16_t, false, true>);
    }
    if (a.bytes) return write(enc_write_kernel<uint8_t, true, false>);
    return code_sm ? write(enc_write_kernel<uint16_t, true, false>) : write(enc_write_kernel<uint16_t, false, false>);
}

cudaError_t launch_header(const HeaderJob &j, cudaStream_t s)
{
    count_launch();
    return launch_next(header_kernel, 1, kHeaderThreads, 0, s, j);
}

bool codebook_fused(unsigned int D) { return D <= kFusedMaxD; }

cudaError_t launch_codebook_batch(const CodebookJob *jobs, int n, cudaStream_t s)
{
    cudaError_t e = set_attrs();
    if (e != cudaSuccess) return e;
    if (n < 1) return cudaSuccess;
    codebook_batch_kernel<<<n, 1024, kCodebookSmem, s>>>(jobs);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_header_batch(const HeaderJob *jobs, int n, cudaStream_t s)
{
    if (n < 1) return cudaSuccess;
    header_batch_kernel<<<n, kHeaderThreads, 0, s>>>(jobs);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_histogram(const uint16_t *sym, unsigned long long N, unsigned D,
                             unsigned long long *hist, unsigned *status, cudaStream_t s)
{
    static PerDeviceOnce attr;
    cudaError_t ea = once_per_device(attr, [] {
        cudaError_t e = cudaFuncSetAttribute(hist_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 65536);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(hist_wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 65536 * 2);
        return e;
    });
    if (ea != cudaSuccess) return ea;
    if (D <= 16384) {
        hist_kernel<<<152 * 4, 256, D * 4, s>>>(sym, N, D, hist, status);
    } else {
        int dev = 0, nsm = 152;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            nsm = 152;
        }
        const unsigned long long rounds = (N + kHistWideRound - 1) / kHistWideRound;
        const unsigned grid = (unsigned)(rounds < (unsigned long long)nsm ? rounds : (unsigned long long)nsm);
        hist_wide_kernel<<<grid, kHistWideThreads, ((D + 1) / 2) * 4, s>>>(sym, N, D, hist, status);
    }
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_histogram_bytes(const uint8_t *in, unsigned long long n, unsigned long long *hist, cudaStream_t s)
{
    // 32 KB of counters a block; a block per 512 threads' turn of 64 bytes
    const unsigned long long need = (n + 64ull * kHistByteThreads - 1) / (64ull * kHistByteThreads);
    hist_bytes_kernel<<<(unsigned)std::min<unsigned long long>(need, 4ull * sm_count()), kHistByteThreads, 0, s>>>(in, n, hist);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_lossless_header(const LosslessHeader &h, const uint8_t *len, const Scalars *sc, uint8_t *out,
                                   cudaStream_t s)
{
    lossless_header_kernel<<<1, 256, 0, s>>>(h, len, sc, out);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_decode(const DecodeArgs &a, const HuffScratch &hs, cudaStream_t s)
{
    cudaError_t e = set_attrs();
    if (e != cudaSuccess) return e;
    count_launch();
    return launch_next(a.bytes ? decode_kernel<uint8_t> : decode_kernel<uint16_t>, sm_count(), kDecThreads, kDecSmem, s, a, hs);
}

}  // namespace hpdr
