// Popcount counting path of the exhaustive search.
//
// Section 2.4 / Algorithm 1: combinations are visited prefix by prefix; the
// genotype table of the (k-1)-prefix (Section 2.1, Listing A.1 semantics:
// row-wise AND) is built once into shared memory and reused for every last
// SNP j; the last level is never stored but fused with the population count
// (Section 2.2, Listing A.2 semantics).  The score is the single-precision MI
// of Eq. 1-3 (Section 2.3) and only the best candidates are kept
// (Section 2.4).
//
// GPU mapping:
//   * persistent grid; CTA b owns the contiguous lexicographic rank range
//     [R_b, R_{b+1}) (every combination costs the same, so a static split
//     balances); it unranks R_b once and then steps prefixes in lex order;
//   * a sub-tile is up to T consecutive ranks spanning at most `slots`
//     prefixes; their tables are staged in shared memory as uint4 rows;
//   * one thread per combination: 128-bit loads of the last SNP's rows for
//     genotypes 0 and 1, AND + POPC against every prefix row; genotype 2 is
//     the prefix row's total minus the other two (exact, saves a third of
//     the work);
//   * the counts never leave registers: MI is evaluated in the same thread
//     and compared against the CTA's current threshold; survivors go to a
//     shared-memory buffer that is merged into the CTA's sorted list;
//   * orders 6-8 (batched launches, and samples beyond the histogram
//     kernel's): the same kernel with one warp per combination; at orders
//     7-8 the prefix table (729 or 2187 rows) is materialised in a per-CTA
//     global buffer (the paper's stored `combine` table, Section 2.1), read
//     through L1/L2 by the CTA's threads, which walk the same prefix rows
//     (batched launches keep it in shared memory where it fits).
#include "epi_internal.cuh"
#include "epi_host.h"

namespace epi {

__host__ __device__ constexpr int ipow3(int k) { return k <= 0 ? 1 : 3 * ipow3(k - 1); }

// Words between consecutive rows of a staged prefix table (orders 1-5).
// Orders 6-8 read the table with one lane per row (a warp per combination)
// and store it transposed by 16-byte words instead: uint4 u of row r at
// [u][r], so the 32 lanes' loads of one word position are 512 contiguous
// bytes (coalesced from global memory, conflict-free in shared memory).
__host__ __device__ inline int popc_row_stride(int k, int32_t Wt) { (void)k; return Wt; }

// One dataset of a launch.  A launch may cover several datasets of the same
// order (batched search): CTAs [cta_begin, cta_begin + cta_count) of the grid
// search this dataset's rank range, sized in proportion to its work.
struct PopcDs {
    DevData d;
    uint64_t rank_begin, rank_end;  // lexicographic range searched
    int32_t cta_begin, cta_count;
    uint32_t *global_thr;           // float bits of max over its CTAs of their pool-th score
};

struct PopcParams {
    PopcDs one;                     // the dataset when the launch has one
    const PopcDs *many;             // else [n_ds] in device memory
    const int32_t *cta_ds;          // and the dataset of each CTA
    int32_t tile;                   // combinations per sub-tile (T)
    int32_t pool;                   // list entries kept per CTA
    int32_t slots;                  // prefixes staged per sub-tile
    int32_t cand_p2;                // shared candidate arrays (power of two)
    int32_t max_wt;                 // largest Wt of the launch (shared-memory layout)
    float *list_score;              // [grid][pool]
    uint64_t *list_rank;            // [grid][pool]
    int32_t *list_count;            // [grid]
    float *all_scores;              // optional: every score, [rank - rank_begin] (single dataset)
    uint32_t *pre_global;           // global prefix tables: [grid][pre_cta_words] (global-prefix kernels)
    int64_t pre_cta_words;
};

struct SlotInfo {
    int64_t base;     // rank of the prefix's first combination (j = s_last + 1)
    int32_t s_last;   // last prefix SNP (-1 for order 1)
    int32_t N;        // number of last SNPs: n - 1 - s_last
    int32_t snp[kMaxOrderGpu];
};

struct SubtileState {
    int64_t F, F_end;              // current sub-tile [F, F_end)
    int64_t cur_base;
    int32_t cur_prefix[kMaxOrderGpu];
    int32_t nslots;
    int32_t list_len, nbuf;
    float thr;
    int32_t done;
};

// next (k-1)-subset of [0, n-1) in lex order; false after the last
__device__ inline bool next_prefix(int32_t *p, int km1, int64_t n)
{
    const int64_t u = n - 1;           // the last SNP needs room after the prefix
    int t = km1 - 1;
    while (t >= 0 && p[t] == u - km1 + t) t--;
    if (t < 0) return false;
    p[t]++;
    for (int v = t + 1; v < km1; v++) p[v] = p[v - 1] + 1;
    return true;
}

__device__ __forceinline__ uint32_t popc4(uint4 p, uint4 a)
{
    return __popc(p.x & a.x) + __popc(p.y & a.y) + __popc(p.z & a.z) + __popc(p.w & a.w);
}

// Counts of one combination against R staged prefix rows, over words [wb, we).
template <int R>
__device__ __forceinline__ void count_rows(const uint32_t *__restrict__ pre, int Wt, const uint32_t *__restrict__ mj,
                                           int wb, int we, uint32_t (&c0)[R], uint32_t (&c1)[R])
{
#pragma unroll
    for (int r = 0; r < R; r++) { c0[r] = 0; c1[r] = 0; }
#pragma unroll 2
    for (int w = wb; w < we; w += 4) {
        const uint4 a = __ldg(reinterpret_cast<const uint4 *>(mj + w));
        const uint4 b = __ldg(reinterpret_cast<const uint4 *>(mj + Wt + w));
#pragma unroll
        for (int r = 0; r < R; r++) {
            const uint4 p = *reinterpret_cast<const uint4 *>(pre + r * Wt + w);
            c0[r] += popc4(p, a);
            c1[r] += popc4(p, b);
        }
    }
}

// Single-precision MI of one combination: the prefix rows are taken R at a
// time (R counters per genotype and class stay in registers); genotype 2 of
// the last SNP is the prefix row's total minus genotypes 0 and 1.
template <int K, int R>
__device__ __forceinline__ float score_popc(const uint32_t *__restrict__ pre, const uint32_t *__restrict__ tot,
                                            const uint32_t *__restrict__ mj, const DevData &d, const MiConstF32 &mc)
{
    constexpr int PR = ipow3(K - 1);
    constexpr int G = PR / R;
    static_assert(PR % R == 0, "row group must divide the prefix rows");
    SumF32 acc;
#pragma unroll 1
    for (int grp = 0; grp < G; grp++) {
        const uint32_t *pg = pre + grp * R * d.Wt;
        uint32_t a0[R], a1[R], b0[R], b1[R];
        count_rows<R>(pg, d.Wt, mj, 0, d.W1, a0, a1);
        count_rows<R>(pg, d.Wt, mj, d.W1, d.Wt, b0, b1);
#pragma unroll
        for (int r = 0; r < R; r++) {
            const uint32_t t1 = tot[(grp * R + r) * 2 + 0];
            const uint32_t t0 = tot[(grp * R + r) * 2 + 1];
            acc.add(cell_terms_f32(a0[r], b0[r], mc));
            acc.add(cell_terms_f32(a1[r], b1[r], mc));
            acc.add(cell_terms_f32(t1 - a0[r] - a1[r], t0 - b0[r] - b1[r], mc));
        }
    }
    return __fdiv_rn(acc.value(), mc.fm);
}

// Sort the live list + buffer, keep the best `pool`, refresh the threshold.
__device__ inline void flush_list(SubtileState &S, float *sc, uint64_t *rk, int pool, int cand_p2,
                                  uint32_t *global_thr)
{
    __syncthreads();
    const int live = S.list_len + S.nbuf;
    const int p2 = next_pow2(live < 2 ? 2 : live);
    for (int i = live + threadIdx.x; i < p2 && i < cand_p2; i += blockDim.x) { sc[i] = -1.0f; rk[i] = ~0ull; }
    __syncthreads();
    block_sort_cands(sc, rk, p2);
    if (threadIdx.x == 0) {
        S.list_len = live < pool ? live : pool;
        S.nbuf = 0;
        if (S.list_len == pool) {
            const float t = sc[pool - 1];
            S.thr = t;
            atomicMax(global_thr, __float_as_uint(t));
        }
    }
    __syncthreads();
}

// Exact FP32 MI of one combination by one warp (orders 6-8): lane l takes
// the prefix rows l, l + 32, ... four at a time, counts them against the last
// SNP's genotype-0/1 rows (the same words for every lane: broadcast loads),
// derives genotype 2 from the row totals, sums its cell terms, and the warp
// adds the lanes' sums.
template <int K>
__device__ __forceinline__ float score_popc_warp(const uint32_t *__restrict__ pre,
                                                 const uint32_t *__restrict__ tot, const uint32_t *__restrict__ mj,
                                                 const DevData &d, const MiConstF32 &mc, int lane)
{
    constexpr int PR = ipow3(K - 1);
    SumF32 acc;
    // the table is transposed by uint4: word group u of row r at uint4 u PR + r
    const uint4 *T = reinterpret_cast<const uint4 *>(pre);
#pragma unroll 1
    for (int r0 = lane; r0 < PR; r0 += 4 * 32) {
        const uint4 *rp[4];
#pragma unroll
        for (int i = 0; i < 4; i++) rp[i] = T + min(r0 + 32 * i, PR - 1);
        uint32_t a0[4] = {0, 0, 0, 0}, a1[4] = {0, 0, 0, 0}, b0[4] = {0, 0, 0, 0}, b1[4] = {0, 0, 0, 0};
#pragma unroll 2
        for (int w = 0; w < d.W1; w += 4) {
            const uint4 x = __ldg(reinterpret_cast<const uint4 *>(mj + w));
            const uint4 y = __ldg(reinterpret_cast<const uint4 *>(mj + d.Wt + w));
            const size_t off = (size_t)(w >> 2) * PR;
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const uint4 p = rp[i][off];
                a0[i] += popc4(p, x);
                a1[i] += popc4(p, y);
            }
        }
#pragma unroll 2
        for (int w = d.W1; w < d.Wt; w += 4) {
            const uint4 x = __ldg(reinterpret_cast<const uint4 *>(mj + w));
            const uint4 y = __ldg(reinterpret_cast<const uint4 *>(mj + d.Wt + w));
            const size_t off = (size_t)(w >> 2) * PR;
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const uint4 p = rp[i][off];
                b0[i] += popc4(p, x);
                b1[i] += popc4(p, y);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int r = r0 + 32 * i;
            if (r < PR) {
                const uint32_t t1 = tot[r * 2 + 0], t0 = tot[r * 2 + 1];
                acc.add(cell_terms_f32(a0[i], b0[i], mc));
                acc.add(cell_terms_f32(a1[i], b1[i], mc));
                acc.add(cell_terms_f32(t1 - a0[i] - a1[i], t0 - b0[i] - b1[i], mc));
            }
        }
    }
    float v = acc.value();
#pragma unroll
    for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return __fdiv_rn(v, mc.fm);
}

template <int K, int R, bool GP>
__global__ void __launch_bounds__(128) popc_search_kernel(PopcParams P)
{
    constexpr int PR = ipow3(K - 1);
    constexpr bool kWarpPerComb = K >= 6;
    const PopcDs &D = P.many ? P.many[P.cta_ds[blockIdx.x]] : P.one;
    const DevData d = D.d;
    const int rstride = popc_row_stride(K, d.Wt);
    const int slot_words = PR * rstride + 4;   // 16-byte skew: slots start on different banks
    extern __shared__ __align__(16) unsigned char smem[];
    // layout: prefix rows (unless global) | totals | candidate scores | candidate ranks
    const size_t pre_words = GP ? 0 : (size_t)P.slots * (PR * popc_row_stride(K, P.max_wt) + 4);
    uint32_t *pre = GP ? P.pre_global + (size_t)blockIdx.x * (size_t)P.pre_cta_words
                       : reinterpret_cast<uint32_t *>(smem);
    uint32_t *tot = reinterpret_cast<uint32_t *>(smem) + pre_words;
    uint64_t *rk = reinterpret_cast<uint64_t *>(smem + (((pre_words + (size_t)P.slots * PR * 2) * 4 + 15) & ~(size_t)15));
    float *sc = reinterpret_cast<float *>(rk + P.cand_p2);
    __shared__ SlotInfo slot[8];
    __shared__ SubtileState S;

    const int km1 = K - 1;
    const MiConstF32 mc = make_mi_const(d.m, d.m1, d.m0);
    const uint64_t span = D.rank_end - D.rank_begin;
    const uint64_t cb = blockIdx.x - (uint64_t)D.cta_begin, cn = (uint64_t)D.cta_count;
    const int64_t R_b = (int64_t)(D.rank_begin + (uint64_t)(((unsigned __int128)span * cb) / cn));
    const int64_t R_e = (int64_t)(D.rank_begin + (uint64_t)(((unsigned __int128)span * (cb + 1)) / cn));

    if (threadIdx.x == 0) {
        S.list_len = 0; S.nbuf = 0; S.thr = -1.0f; S.done = R_b >= R_e;
        S.F = R_b;
        if (!S.done) {
            int32_t c[kMaxOrderGpu];
            unrank_lex(d.binom, d.n, K, (uint64_t)R_b, c);
            const int32_t s_last = K > 1 ? c[K - 2] : -1;
            for (int t = 0; t < km1; t++) S.cur_prefix[t] = c[t];
            S.cur_base = R_b - (c[K - 1] - (s_last + 1));
        }
    }
    __syncthreads();

    while (!S.done) {
        // ---- assemble the sub-tile's prefixes ----------------------------
        if (threadIdx.x == 0) {
            const int64_t lim = min((int64_t)S.F + P.tile, R_e);
            int32_t p[kMaxOrderGpu];
            for (int t = 0; t < km1; t++) p[t] = S.cur_prefix[t];
            int64_t base = S.cur_base;
            int ns = 0;
            bool more = true;
            while (true) {
                SlotInfo &sl = slot[ns];
                sl.base = base;
                sl.s_last = km1 > 0 ? p[km1 - 1] : -1;
                sl.N = (int32_t)(d.n - 1 - sl.s_last);
                for (int t = 0; t < km1; t++) sl.snp[t] = p[t];
                ns++;
                base += sl.N;
                if (base >= lim || ns == P.slots) break;
                if (km1 == 0 || !next_prefix(p, km1, d.n)) { more = false; break; }
            }
            const SlotInfo &last = slot[ns - 1];
            const int64_t last_end = last.base + last.N;
            S.F_end = min(lim, last_end);
            S.nslots = ns;
            // prefix containing the next sub-tile's first rank
            if (S.F_end == last_end && S.F_end < R_e) {
                for (int t = 0; t < km1; t++) p[t] = last.snp[t];
                if (km1 > 0) more = next_prefix(p, km1, d.n);
                for (int t = 0; t < km1; t++) S.cur_prefix[t] = p[t];
                S.cur_base = last_end;
                (void)more;
            } else {
                for (int t = 0; t < km1; t++) S.cur_prefix[t] = last.snp[t];
                S.cur_base = last.base;
            }
            // stricter of the CTA threshold and the best known global one
            const float g = __uint_as_float(*(volatile uint32_t *)D.global_thr);
            if (S.list_len == P.pool || g > 0.0f) S.thr = fmaxf(S.thr, g);
        }
        __syncthreads();

        // ---- stage prefix tables: row x' = sum_t g_t 3^(k-2-t) -------------
        const int ns = S.nslots;
        const int W4 = d.Wt >> 2;
        if constexpr (K >= 6) {
            // blocks of 9 rows that share the genotypes of the first k-3
            // prefix SNPs: their AND is formed once, then the last two SNPs'
            // rows (k + 3 loads per 9 rows instead of 9 (k - 1))
            constexpr int PB = PR / 9;
            // block index fastest: consecutive threads write consecutive rows
            // of one word group of the transposed table
            for (int idx = threadIdx.x; idx < ns * PB * W4; idx += blockDim.x) {
                const int blk = idx % PB;
                const int w4 = (idx / PB) % W4;
                const int s = idx / (W4 * PB);
                uint4 base = make_uint4(~0u, ~0u, ~0u, ~0u);
                int rem = blk;
                int div = PB / 3;
#pragma unroll
                for (int t = 0; t < km1 - 2; t++) {
                    const int g = rem / div;
                    rem -= g * div;
                    div = div > 1 ? div / 3 : 1;
                    const uint4 v = __ldg(reinterpret_cast<const uint4 *>(
                        d.masks + ((int64_t)slot[s].snp[t] * 3 + g) * d.Wt) + w4);
                    base.x &= v.x; base.y &= v.y; base.z &= v.z; base.w &= v.w;
                }
                const uint4 *ma = reinterpret_cast<const uint4 *>(d.masks + (int64_t)slot[s].snp[km1 - 2] * 3 * d.Wt);
                const uint4 *mb = reinterpret_cast<const uint4 *>(d.masks + (int64_t)slot[s].snp[km1 - 1] * 3 * d.Wt);
                uint4 lb[3];
#pragma unroll
                for (int h = 0; h < 3; h++) lb[h] = __ldg(mb + h * W4 + w4);
                uint4 *ps = reinterpret_cast<uint4 *>(pre + (size_t)s * slot_words) + (size_t)w4 * PR + blk * 9;
#pragma unroll
                for (int g = 0; g < 3; g++) {
                    const uint4 a = __ldg(ma + g * W4 + w4);
                    const uint4 b1 = make_uint4(base.x & a.x, base.y & a.y, base.z & a.z, base.w & a.w);
#pragma unroll
                    for (int h = 0; h < 3; h++)
                        ps[g * 3 + h] = make_uint4(b1.x & lb[h].x, b1.y & lb[h].y, b1.z & lb[h].z, b1.w & lb[h].w);
                }
            }
        } else
        for (int idx = threadIdx.x; idx < ns * PR * W4; idx += blockDim.x) {
            const int w4 = idx % W4;
            const int row = (idx / W4) % PR;
            const int s = idx / (W4 * PR);
            uint4 acc;
            if (K == 1) {
                // the empty prefix: every real individual of each subtable
                const int w = w4 * 4;
                uint32_t v[4];
                for (int q = 0; q < 4; q++) {
                    const int ww = w + q;
                    const int64_t first = ww < d.W1 ? (int64_t)ww * 32 : (int64_t)(ww - d.W1) * 32;
                    const int64_t size = ww < d.W1 ? d.m1 : d.m0;
                    const int64_t left = size - first;
                    v[q] = left >= 32 ? 0xffffffffu : (left <= 0 ? 0u : ((1u << left) - 1u));
                }
                acc = make_uint4(v[0], v[1], v[2], v[3]);
            } else {
                acc = make_uint4(~0u, ~0u, ~0u, ~0u);
                int rem = row;
                int div = PR / 3;
#pragma unroll
                for (int t = 0; t < km1; t++) {
                    const int g = rem / div;
                    rem -= g * div;
                    div = div > 1 ? div / 3 : 1;
                    const uint4 v = __ldg(reinterpret_cast<const uint4 *>(
                        d.masks + ((int64_t)slot[s].snp[t] * 3 + g) * d.Wt) + w4);
                    acc.x &= v.x; acc.y &= v.y; acc.z &= v.z; acc.w &= v.w;
                }
            }
            reinterpret_cast<uint4 *>(pre + (size_t)s * slot_words + (size_t)row * rstride)[w4] = acc;
        }
        __syncthreads();
        // per-row totals of each subtable (the third genotype by subtraction);
        // orders 6-8: one thread per (row, subtable) of the transposed table,
        // consecutive threads on consecutive rows
        if constexpr (K >= 6) {
            for (int idx = threadIdx.x; idx < ns * PR * 2; idx += blockDim.x) {
                const int row = idx % PR;
                const int half = (idx / PR) & 1;
                const int s = idx / (PR * 2);
                const uint4 *T = reinterpret_cast<const uint4 *>(pre + (size_t)s * slot_words) + row;
                const int ub = half ? d.W1 / 4 : 0, ue = half ? d.Wt / 4 : d.W1 / 4;
                uint32_t c = 0;
                for (int u = ub; u < ue; u++) {
                    const uint4 v = T[(size_t)u * PR];
                    c += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
                }
                tot[((size_t)s * PR + row) * 2 + half] = c;
            }
        } else
        for (int idx = threadIdx.x; idx < ns * PR * 2; idx += blockDim.x) {
            const int half = idx & 1;
            const int sr = idx >> 1;
            const uint32_t *row = pre + (size_t)(sr / PR) * slot_words + (size_t)(sr % PR) * rstride;
            uint32_t c = 0;
            const int wb = half ? d.W1 : 0, we = half ? d.Wt : d.W1;
            for (int w = wb; w < we; w++) c += __popc(row[w]);
            tot[sr * 2 + half] = c;
        }
        __syncthreads();

        // ---- count and score: one thread per combination -------------------
        const int64_t F = S.F, F_end = S.F_end;
        const int list_len = S.list_len;
        const float thr = S.thr;
        if constexpr (kWarpPerComb) {
            // one warp per combination
            const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
            for (int64_t f = F + warp; f < F_end; f += blockDim.x >> 5) {
                int s = 0;
                while (s + 1 < ns && f >= slot[s + 1].base) s++;
                const int32_t j = slot[s].s_last + 1 + (int32_t)(f - slot[s].base);
                const float score = score_popc_warp<K>(pre + (size_t)s * slot_words, tot + s * PR * 2,
                                                       d.masks + (int64_t)j * 3 * d.Wt, d, mc, lane);
                if (lane == 0) {
                    if (P.all_scores) P.all_scores[f - (int64_t)D.rank_begin] = score;
                    if (score >= thr) {
                        const int pos = list_len + atomicAdd(&S.nbuf, 1);
                        sc[pos] = score;
                        rk[pos] = (uint64_t)f;
                    }
                }
            }
        } else
        for (int64_t f = F + threadIdx.x; f < F_end; f += blockDim.x) {
            int s = 0;
            while (s + 1 < ns && f >= slot[s + 1].base) s++;
            const int32_t j = slot[s].s_last + 1 + (int32_t)(f - slot[s].base);
            const float score = score_popc<K, R>(pre + (size_t)s * slot_words, tot + s * PR * 2,
                                                 d.masks + (int64_t)j * 3 * d.Wt, d, mc);
            if (P.all_scores) P.all_scores[f - (int64_t)D.rank_begin] = score;
            if (score >= thr) {
                const int pos = list_len + atomicAdd(&S.nbuf, 1);
                sc[pos] = score;
                rk[pos] = (uint64_t)f;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            S.F = F_end;
            S.done = F_end >= R_e;
        }
        __syncthreads();
        if (S.nbuf > P.tile || (S.done && S.nbuf > 0)) flush_list(S, sc, rk, P.pool, P.cand_p2, D.global_thr);
    }
    __syncthreads();
    const int L = S.list_len;
    for (int i = threadIdx.x; i < L; i += blockDim.x) {
        P.list_score[(size_t)blockIdx.x * P.pool + i] = sc[i];
        P.list_rank[(size_t)blockIdx.x * P.pool + i] = rk[i];
    }
    if (threadIdx.x == 0) P.list_count[blockIdx.x] = L;
}

template <int K, int R, bool GP>
static cudaError_t launch_kr(const PopcParams &p, int grid, size_t smem, cudaStream_t st)
{
    auto kern = popc_search_kernel<K, R, GP>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<grid, 128, smem, st>>>(p);
    return cudaGetLastError();
}

template <int K, int R, bool GP>
static int occupancy_kr(size_t smem)
{
    auto kern = popc_search_kernel<K, R, GP>;
    int n = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, 128, smem) != cudaSuccess) return 0;
    return n;
}

// Row-group sizes compiled per order: every R divides 3^(k-1).
bool popc_row_group_ok(int k, int R)
{
    switch (k) {
    case 1: return R == 1;
    case 2: return R == 3;
    case 3: return R == 9;
    case 4: return R == 9 || R == 27;
    case 5: return R == 9 || R == 27;
    case 6: return R == 9;
    case 7: return R == 9;
    case 8: return R == 9;
    default: return false;
    }
}

// orders whose prefix tables may also live in global memory
bool popc_global_prefix_ok(int k, int R) { return (k == 7 || k == 8) && R == 9; }

int popc_default_row_group(int k)
{
    return k == 1 ? 1 : (k == 2 ? 3 : 9);
}

int popc_slot_words(int k, int32_t Wt)
{
    return ipow3(k - 1) * popc_row_stride(k, Wt) + 4;   // 16-byte skew: slots start on different banks
}

size_t popc_smem_bytes(int k, int32_t Wt, int slots, int cand_p2, bool global_prefix)
{
    const size_t PR = (size_t)ipow3(k - 1);
    const size_t pre = global_prefix ? 0 : (size_t)slots * popc_slot_words(k, Wt);
    size_t b = ((pre + (size_t)slots * PR * 2) * 4 + 15) & ~(size_t)15;
    return b + (size_t)cand_p2 * 12;
}

int popc_max_active(int k, int R, size_t smem, bool global_prefix)
{
    if (global_prefix) {
        switch (k * 100 + R) {
        case 709: return occupancy_kr<7, 9, true>(smem);
        case 809: return occupancy_kr<8, 9, true>(smem);
        default: return 0;
        }
    }
    switch (k * 100 + R) {
    case 101: return occupancy_kr<1, 1, false>(smem);
    case 203: return occupancy_kr<2, 3, false>(smem);
    case 309: return occupancy_kr<3, 9, false>(smem);
    case 409: return occupancy_kr<4, 9, false>(smem);
    case 427: return occupancy_kr<4, 27, false>(smem);
    case 509: return occupancy_kr<5, 9, false>(smem);
    case 527: return occupancy_kr<5, 27, false>(smem);
    case 609: return occupancy_kr<6, 9, false>(smem);
    case 709: return occupancy_kr<7, 9, false>(smem);
    case 809: return occupancy_kr<8, 9, false>(smem);
    default: return 0;
    }
}

static cudaError_t launch_dispatch(const PopcParams &p, int k, int R, int grid, size_t smem, cudaStream_t st)
{
    if (p.pre_global) {
        switch (k * 100 + R) {
        case 709: return launch_kr<7, 9, true>(p, grid, smem, st);
        case 809: return launch_kr<8, 9, true>(p, grid, smem, st);
        default: return cudaErrorInvalidValue;
        }
    }
    switch (k * 100 + R) {
    case 101: return launch_kr<1, 1, false>(p, grid, smem, st);
    case 203: return launch_kr<2, 3, false>(p, grid, smem, st);
    case 309: return launch_kr<3, 9, false>(p, grid, smem, st);
    case 409: return launch_kr<4, 9, false>(p, grid, smem, st);
    case 427: return launch_kr<4, 27, false>(p, grid, smem, st);
    case 509: return launch_kr<5, 9, false>(p, grid, smem, st);
    case 527: return launch_kr<5, 27, false>(p, grid, smem, st);
    case 609: return launch_kr<6, 9, false>(p, grid, smem, st);
    case 709: return launch_kr<7, 9, false>(p, grid, smem, st);
    case 809: return launch_kr<8, 9, false>(p, grid, smem, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_popc_search(const DevData &d, int k, int R, uint64_t rank_begin, uint64_t rank_end, int tile,
                               int pool, int slots, int cand_p2, uint32_t *global_thr, float *list_score,
                               uint64_t *list_rank, int32_t *list_count, int grid, size_t smem, cudaStream_t st,
                               float *all_scores, uint32_t *pre_global)
{
    PopcParams p;
    p.all_scores = all_scores;
    p.pre_global = pre_global;
    p.pre_cta_words = (int64_t)slots * popc_slot_words(k, d.Wt);
    p.one.d = d;
    p.one.rank_begin = rank_begin;
    p.one.rank_end = rank_end;
    p.one.cta_begin = 0;
    p.one.cta_count = grid;
    p.one.global_thr = global_thr;
    p.many = nullptr;
    p.cta_ds = nullptr;
    p.tile = tile;
    p.pool = pool;
    p.slots = slots;
    p.cand_p2 = cand_p2;
    p.max_wt = d.Wt;
    p.list_score = list_score;
    p.list_rank = list_rank;
    p.list_count = list_count;
    return launch_dispatch(p, k, R, grid, smem, st);
}

size_t popc_ds_bytes() { return sizeof(PopcDs); }

void popc_fill_ds(void *dst, const DevData &d, uint64_t rank_begin, uint64_t rank_end, int cta_begin, int cta_count,
                  uint32_t *global_thr)
{
    PopcDs *o = static_cast<PopcDs *>(dst);
    o->d = d;
    o->rank_begin = rank_begin;
    o->rank_end = rank_end;
    o->cta_begin = cta_begin;
    o->cta_count = cta_count;
    o->global_thr = global_thr;
}

cudaError_t launch_popc_batch(const void *ds_dev, const int32_t *cta_ds_dev, int k, int R, int max_wt, int tile,
                              int pool, int slots, int cand_p2, float *list_score, uint64_t *list_rank,
                              int32_t *list_count, int grid, size_t smem, cudaStream_t st)
{
    PopcParams p;
    p.all_scores = nullptr;
    p.pre_global = nullptr;
    p.pre_cta_words = 0;
    p.one = PopcDs();
    p.many = static_cast<const PopcDs *>(ds_dev);
    p.cta_ds = cta_ds_dev;
    p.tile = tile;
    p.pool = pool;
    p.slots = slots;
    p.cand_p2 = cand_p2;
    p.max_wt = max_wt;
    p.list_score = list_score;
    p.list_rank = list_rank;
    p.list_count = list_count;
    return launch_dispatch(p, k, R, grid, smem, st);
}

}  // namespace epi
