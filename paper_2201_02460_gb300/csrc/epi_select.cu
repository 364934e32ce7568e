// Top-N retention (Section 2.4: only the combinations with the highest MI
// are kept) made exact on the GPU:
//   1. merge_level: the per-CTA candidate lists of the search kernel are
//      merged, level by level, into one pool ordered by (single-precision score desc, rank asc);
//   2. rescore: every pooled combination is recounted exactly (AND + POPC of
//      its k genotype rows, Section 2.2) and scored in double precision;
//   3. finalize: the pool is sorted by (double MI desc, lexicographic rank
//      asc), the best N are written out, and the margin check proves that no
//      combination outside the pool could have entered the top N (otherwise
//      the host retries with a larger pool).
// Also the table kernels behind epi_tables / epi_score_tables.
#include "epi_internal.cuh"
#include "epi_host.h"

namespace epi {

// Shared memory of a merge block: its entries, and the pool's best of them.
__host__ __device__ inline int merge_entries(int group, int cap, int pool)
{
    const int e = group * cap < 2 ? 2 : group * cap;
    return next_pow2(e) + (pool < 2 ? 2 : pool);
}

// Entries up to which the last level of a merge sorts by counting, with work
// that grows with their square (the k best of 2^20 floats in order, by counting
// and by the bitonic sort: k = 600 171 and 170 us, 1000 198 and 175, 4096 943
// and 243).
constexpr int kCountSort = 512;

// float bits in an order-preserving unsigned form
__device__ __forceinline__ uint32_t order_bits(float f)
{
    const uint32_t u = __float_as_uint(f);
    return u & 0x80000000u ? ~u : u | 0x80000000u;
}

// One level of the merge: block b takes lists [b group, (b + 1) group) -- list
// i at ls + i pitch with lc[i lstep] entries -- and keeps the best `pool` of
// their entries: in place as list b group of the next level, or sorted in
// out_* when this is the last level (one block).  The cut is found by a radix
// select over the scores (four 8-bit passes), and the last level sorts few
// entries by counting, for each, the better ones, and more of them by a bitonic
// sort; entries below the search's
// threshold are dropped on loading.  (One block that sorted 1024 entries at a
// time took 124 us for 155 lists of 128, two levels of 4096-entry bitonic
// sorts 2 x 45.)
__global__ void __launch_bounds__(1024) merge_level_kernel(float *__restrict__ ls, uint64_t *__restrict__ lr,
                                                           int32_t *__restrict__ lc, int nlists, int64_t pitch,
                                                           int lstep, int group, int cap, int pool,
                                                           float *__restrict__ out_s, uint64_t *__restrict__ out_r,
                                                           int32_t *__restrict__ out_n,
                                                           const uint32_t *__restrict__ thr, float floor)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int entries = merge_entries(group, cap, pool);
    uint64_t *rk = reinterpret_cast<uint64_t *>(smem);
    float *sc = reinterpret_cast<float *>(rk + entries);
    __shared__ int32_t live_sh, kept_sh, need_sh;
    __shared__ uint32_t hist[256], digit_sh;
    const int first = blockIdx.x * group;
    const int lists = min(group, nlists - first);
    if (threadIdx.x == 0) { live_sh = 0; kept_sh = 0; need_sh = pool; }
    __syncthreads();
    const float cut = thr ? fmaxf(floor, __uint_as_float(*thr)) : floor;
    for (int e = threadIdx.x; e < lists * cap; e += blockDim.x) {
        const int l = e / cap, i = e - l * cap;
        if (i < lc[(int64_t)(first + l) * lstep]) {
            const int64_t at = (int64_t)(first + l) * pitch + i;
            const float v = ls[at];
            if (v >= cut) {
                const int pos = atomicAdd(&live_sh, 1);
                sc[pos] = v;
                rk[pos] = lr[at];
            }
        }
    }
    __syncthreads();
    const int live = live_sh;
    float *ks = sc;                                  // the kept entries
    uint64_t *kr = rk;
    int L = live;
    if (live > pool) {
        // the pool-th largest score, digit by digit
        uint32_t prefix = 0, mask = 0;
        for (int shift = 24; shift >= 0; shift -= 8) {
            if (threadIdx.x < 256) hist[threadIdx.x] = 0;
            __syncthreads();
            for (int i = threadIdx.x; i < live; i += blockDim.x) {
                const uint32_t u = order_bits(sc[i]);
                if ((u & mask) == prefix) atomicAdd(&hist[(u >> shift) & 255u], 1u);
            }
            __syncthreads();
            if (threadIdx.x < 32) {
                // 8 bins a lane, from the top
                const int lane = threadIdx.x, hi = 255 - 8 * lane;
                int sum = 0;
                for (int q = 0; q < 8; q++) sum += (int)hist[hi - q];
                int inc = sum;
                for (int off = 1; off < 32; off <<= 1) {
                    const int o = __shfl_up_sync(0xffffffffu, inc, off);
                    if (lane >= off) inc += o;
                }
                const int need = need_sh;
                __syncwarp();
                int before = inc - sum;
                if (before < need && inc >= need) {
                    int q = 0;
                    while (before + (int)hist[hi - q] < need) before += (int)hist[hi - q++];
                    digit_sh = (uint32_t)(hi - q);
                    need_sh = need - before;
                }
            }
            __syncthreads();
            prefix |= digit_sh << shift;
            mask |= 255u << shift;
            __syncthreads();
        }
        // every entry above the cut, and of those at it the need_sh best by
        // rank (usually all of them)
        ks = sc + entries - pool;
        kr = rk + entries - pool;
        const int need = need_sh;
        for (int i = threadIdx.x; i < live; i += blockDim.x) {
            const uint32_t u = order_bits(sc[i]);
            bool keep = u > prefix;
            if (u == prefix) {
                int better = 0;
                const uint64_t r = rk[i];
                for (int q = 0; q < live; q++) better += order_bits(sc[q]) == prefix && rk[q] < r;
                keep = better < need;
            }
            if (keep) {
                const int pos = atomicAdd(&kept_sh, 1);
                ks[pos] = sc[i];
                kr[pos] = rk[i];
            }
        }
        __syncthreads();
        L = pool;
    }
    if (out_s && L > kCountSort) {
        // (entries past the front are free: the kept ones lie behind them all)
        if (ks != sc)
            for (int i = threadIdx.x; i < L; i += blockDim.x) { sc[i] = ks[i]; rk[i] = kr[i]; }
        const int p2 = next_pow2(L);
        for (int i = L + threadIdx.x; i < p2; i += blockDim.x) { sc[i] = -INFINITY; rk[i] = ~0ull; }
        __syncthreads();
        block_sort_cands(sc, rk, p2);
        for (int i = threadIdx.x; i < L; i += blockDim.x) { out_s[i] = sc[i]; out_r[i] = rk[i]; }
        if (threadIdx.x == 0) *out_n = L;
    } else if (out_s) {
        for (int i = threadIdx.x; i < L; i += blockDim.x) {
            const float v = ks[i];
            const uint64_t r = kr[i];
            int pos = 0;
            for (int q = 0; q < L; q++) pos += cand_better(ks[q], kr[q], v, r);
            out_s[pos] = v;
            out_r[pos] = r;
        }
        if (threadIdx.x == 0) *out_n = L;
    } else {
        for (int i = threadIdx.x; i < L; i += blockDim.x) {
            ls[(int64_t)first * pitch + i] = ks[i];
            lr[(int64_t)first * pitch + i] = kr[i];
        }
        if (threadIdx.x == 0) lc[(int64_t)first * lstep] = L;
    }
}

// Exact counts of one combination, cell x = sum_t g_t 3^(k-1-t): one thread
// per (class, cell) pair, or, where those are fewer than the block's threads,
// one warp per pair with the lanes along the words (an order-2 table has 18
// pairs: one thread each walked its words alone).  From order 6 the table has
// about as many cells as individuals or more, and the individuals are visited
// instead, a warp per mask word adding into the zeroed table (order 8 x 2048,
// 164 candidates: 0.5 ms less of 1.07).
__device__ inline void count_cells(const DevData &d, int k, const int32_t *comb, uint32_t *out)
{
    int cells = 1;
    for (int t = 0; t < k; t++) cells *= 3;
    if (k >= 6) {
        for (int x = threadIdx.x; x < 2 * cells; x += blockDim.x) out[x] = 0;
        __syncthreads();
        const int lane = threadIdx.x & 31;
        for (int w = threadIdx.x >> 5; w < d.Wt; w += blockDim.x >> 5) {
            uint32_t any = 0;
            int x = 0;
#pragma unroll 4
            for (int t = 0; t < k; t++) {
                const uint32_t *r = d.masks + (int64_t)comb[t] * 3 * d.Wt + w;
                const uint32_t g0 = r[0], g1 = r[d.Wt], g2 = r[2 * (int64_t)d.Wt];
                any = g0 | g1 | g2;
                x = 3 * x + (int)(g1 >> lane & 1u) + 2 * (int)(g2 >> lane & 1u);
            }
            if (any >> lane & 1u) atomicAdd(out + (w < d.W1 ? 0 : cells) + x, 1u);
        }
        return;
    }
    const bool by_warp = 2 * cells < (int)blockDim.x;
    const int lane = by_warp ? threadIdx.x & 31 : 0, width = by_warp ? 32 : 1;
    for (int idx = by_warp ? threadIdx.x >> 5 : threadIdx.x; idx < 2 * cells; idx += blockDim.x / width) {
        const int half = idx / cells;
        const int x = idx - half * cells;
        const uint32_t *rows[EPI_MAX_ORDER];
        int rem = x, div = cells / 3;
        for (int t = 0; t < k; t++) {
            const int g = rem / div;
            rem -= g * div;
            div = div > 1 ? div / 3 : 1;
            rows[t] = d.masks + ((int64_t)comb[t] * 3 + g) * d.Wt;
        }
        const int wb = half ? d.W1 : 0, we = half ? d.Wt : d.W1;
        uint32_t c = 0;
        for (int w = wb + lane; w < we; w += width) {
            uint32_t v = rows[0][w];
            for (int t = 1; t < k; t++) v &= rows[t][w];
            c += __popc(v);
        }
        if (by_warp) c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0) out[half * cells + x] = c;
    }
}

// unrank_lex by one warp: each element's search probes 32 places at a time
// (the binomials come from L2: a binary search waits for log2 n of them).
__device__ inline void unrank_lex_warp(const uint64_t *tab, int64_t n, int k, uint64_t r, int32_t *out)
{
    const int lane = threadIdx.x & 31;
    int64_t start = 0;
    for (int t = 0; t < k; t++) {
        const int rem = k - t;
        const uint64_t total = binom_at(tab, n, n - start, rem);
        const uint64_t x = total - r;
        // smallest c in [start, n - rem] with C(n - 1 - c, rem) < x (true at n - rem)
        int64_t lo = start, hi = n - rem;
        while (lo < hi) {
            const int64_t step = (hi - lo + 31) / 32;
            const int64_t c = lo + lane * step < hi ? lo + lane * step : hi;
            const uint32_t ok = __ballot_sync(0xffffffffu, binom_at(tab, n, n - 1 - c, rem) < x);
            const int f = ok ? __ffs(ok) - 1 : 32;   // first probe that holds
            const int64_t at = lo + f * step;
            if (f > 0) lo += (f - 1) * step + 1;
            hi = f < 32 && at < hi ? at : hi;
        }
        r -= total - binom_at(tab, n, n - lo, rem);
        if (lane == 0) out[t] = (int32_t)lo;
        start = lo + 1;
    }
}

// double-precision MI of a counted table, cells in ascending order
__device__ inline double table_mi_f64(const DevData &d, const uint32_t *ct, int cells)
{
    double acc = 0.0;
    for (int x = 0; x < cells; x++) {
        const uint32_t a = ct[x], b = ct[cells + x];
        acc += mi_term_f64(a, a + b, d.m1, d.m);
        acc += mi_term_f64(b, a + b, d.m0, d.m);
    }
    return acc / (double)d.m;
}

__device__ inline float table_mi_f32(const DevData &d, const uint32_t *ct, int cells)
{
    const MiConstF32 mc = make_mi_const(d.m, d.m1, d.m0);
    SumF32 acc;
    for (int x = 0; x < cells; x++) acc.add(cell_terms_f32(ct[x], ct[cells + x], mc));
    return __fdiv_rn(acc.value(), mc.fm);
}

constexpr int kRescoreThreads = 256;

// One pooled combination per block: its table, then its double-precision MI
// with the cells shared out over the block (thread t takes cells t, t + 256,
// ...) and the threads' sums added as a tree in a fixed order, so the value
// is the same on every run (the 13,122 terms of an order-8 table took one
// thread 4.8 ms of double-precision divisions and logarithms).  Orders 6 and
// up: 164 order-8 tables of 2048 individuals took 1.07 ms; 0.58 with the
// counts by individuals, 0.22 with the empty cells left out as well.
__global__ void __launch_bounds__(kRescoreThreads) rescore_kernel(DevData d, int k,
                                                                  const uint64_t *__restrict__ cand_rank,
                                                                  const int32_t *__restrict__ cand_n,
                                                                  uint32_t *__restrict__ counts,
                                                                  double *__restrict__ mi64, int32_t *__restrict__ combs)
{
    __shared__ int32_t comb[EPI_MAX_ORDER];
    __shared__ double part[kRescoreThreads];
    const int c = blockIdx.x;
    if (c >= *cand_n) return;
    int cells = 1;
    for (int t = 0; t < k; t++) cells *= 3;
    if (threadIdx.x < 32) {
        unrank_lex_warp(d.binom, d.n, k, cand_rank[c], comb);
        __syncwarp();
        if (threadIdx.x < k) combs[(int64_t)c * k + threadIdx.x] = comb[threadIdx.x];
    }
    __syncthreads();
    uint32_t *ct = counts + (int64_t)c * 2 * cells;
    count_cells(d, k, comb, ct);
    __syncthreads();
    double acc = 0.0;
    if (k < 6) {
        for (int x = threadIdx.x; x < cells; x += kRescoreThreads) {
            const uint32_t a = ct[x], b = ct[cells + x];
            acc += mi_term_f64(a, a + b, d.m1, d.m);
            acc += mi_term_f64(b, a + b, d.m0, d.m);
        }
    } else {
        // most cells are empty: each warp gathers 32 others before it takes
        // them to double precision, and every lane then adds the terms of its
        // own cells in their order (an empty cell would have added zero)
        __shared__ uint16_t queue[kRescoreThreads / 32][64];
        __shared__ double term[kRescoreThreads / 32][64];
        uint16_t *q = queue[threadIdx.x >> 5];
        double *te = term[threadIdx.x >> 5];
        const int lane = threadIdx.x & 31;
        int held = 0;
        uint64_t mine = 0;   // places of the lane's own cells in the queue
        auto take32 = [&]() {
            if (lane < held) {
                const int x = q[lane];
                const uint32_t a = ct[x], b = ct[cells + x];
                te[lane] = mi_term_f64(a, a + b, d.m1, d.m);
                te[32 + lane] = mi_term_f64(b, a + b, d.m0, d.m);
            }
            const uint16_t next = q[32 + lane];
            __syncwarp();
            for (uint32_t own = (uint32_t)mine; own; own &= own - 1) {
                const int e = __ffs(own) - 1;
                acc += te[e];
                acc += te[32 + e];
            }
            q[lane] = next;
            mine >>= 32;
            held -= 32;
            __syncwarp();
        };
        q[32 + lane] = 0;
        for (int x0 = threadIdx.x & ~31; x0 < cells; x0 += kRescoreThreads) {
            const int x = x0 + lane;
            const bool some = x < cells && (ct[x] | ct[cells + x]) != 0;
            const uint32_t mask = __ballot_sync(0xffffffffu, some);
            const int at = held + __popc(mask & ((1u << lane) - 1u));
            if (some) {
                q[at] = (uint16_t)x;
                mine |= 1ull << at;
            }
            held += __popc(mask);
            __syncwarp();
            if (held >= 32) take32();
        }
        if (held > 0) take32();
    }
    part[threadIdx.x] = acc;
    __syncthreads();
    for (int w = kRescoreThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) mi64[c] = part[0] / (double)d.m;
}

__device__ __forceinline__ bool final_better(double ma, uint64_t ra, double mb, uint64_t rb)
{
    return ma > mb || (ma == mb && ra < rb);
}

__global__ void __launch_bounds__(1024) finalize_kernel(DevData d, int k, int top_n, int pool,
                                                        const float *__restrict__ cand_s, const uint64_t *__restrict__ cand_r,
                                                        const int32_t *__restrict__ cand_n,
                                                        const double *__restrict__ mi64, const int32_t *__restrict__ combs,
                                                        const uint32_t *__restrict__ counts, const uint32_t *__restrict__ global_thr,
                                                        uint64_t total, epi_result *__restrict__ out,
                                                        uint32_t *__restrict__ out_counts, int32_t *__restrict__ n_out,
                                                        int32_t *__restrict__ status)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int L = *cand_n;
    const int p2 = next_pow2(L < 2 ? 2 : L);
    double *key = reinterpret_cast<double *>(smem);
    uint64_t *rk = reinterpret_cast<uint64_t *>(key + p2);
    int32_t *idx = reinterpret_cast<int32_t *>(rk + p2);
    for (int i = threadIdx.x; i < p2; i += blockDim.x) {
        if (i < L) { key[i] = mi64[i]; rk[i] = cand_r[i]; idx[i] = i; }
        else { key[i] = -1.0; rk[i] = ~0ull; idx[i] = -1; }
    }
    __syncthreads();
    for (int kk = 2; kk <= p2; kk <<= 1) {
        for (int jj = kk >> 1; jj > 0; jj >>= 1) {
            for (int i = threadIdx.x; i < p2; i += blockDim.x) {
                const int ixj = i ^ jj;
                if (ixj > i) {
                    const bool up = (i & kk) == 0;
                    const bool sw = up ? final_better(key[ixj], rk[ixj], key[i], rk[i])
                                       : final_better(key[i], rk[i], key[ixj], rk[ixj]);
                    if (sw) {
                        double tk = key[i]; key[i] = key[ixj]; key[ixj] = tk;
                        uint64_t tr = rk[i]; rk[i] = rk[ixj]; rk[ixj] = tr;
                        int32_t ti = idx[i]; idx[i] = idx[ixj]; idx[ixj] = ti;
                    }
                }
            }
            __syncthreads();
        }
    }
    const int N = L < top_n ? L : top_n;
    int cells = 1;
    for (int t = 0; t < k; t++) cells *= 3;
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const int c = idx[i];
        epi_result r;
        for (int t = 0; t < EPI_MAX_ORDER; t++) r.snp[t] = t < k ? (uint32_t)combs[(int64_t)c * k + t] : 0u;
        r.mi = mi64[c];
        r.mi_f32 = cand_s[c];
        r.order = (uint32_t)k;
        r.rank = cand_r[c];
        out[i] = r;
    }
    if (out_counts) {
        for (int64_t e = threadIdx.x; e < (int64_t)N * 2 * cells; e += blockDim.x) {
            const int i = (int)(e / (2 * cells));
            const int q = (int)(e - (int64_t)i * 2 * cells);
            out_counts[e] = counts[(int64_t)idx[i] * 2 * cells + q];
        }
    }
    if (threadIdx.x == 0) {
        *n_out = N;
        // margin check: every combination outside the pool scored at most
        // tau in single precision, hence at most tau / (1 - eps) exactly
        float tau = __uint_as_float(*global_thr);
        if (L == pool && (uint64_t)L < total) tau = fmaxf(tau, cand_s[L - 1]);
        if (tau > 0.0f && N > 0 && (uint64_t)L < total) {
            const double eps = f32_rel_bound(k, d.m);
            const double sigma = key[N - 1];
            if (!((double)tau / (1.0 - eps) < sigma * (1.0 - 1e-12))) atomicOr(status, ST_POOL_OVERFLOW);
        }
    }
}

__global__ void tables_kernel(DevData d, int k, const uint32_t *__restrict__ combs, int64_t count,
                              uint32_t *__restrict__ out)
{
    __shared__ int32_t comb[EPI_MAX_ORDER];
    int cells = 1;
    for (int t = 0; t < k; t++) cells *= 3;
    for (int64_t c = blockIdx.x; c < count; c += gridDim.x) {
        __syncthreads();
        if (threadIdx.x < k) comb[threadIdx.x] = (int32_t)combs[c * k + threadIdx.x];
        __syncthreads();
        count_cells(d, k, comb, out + c * 2 * cells);
    }
}

__global__ void score_tables_kernel(DevData d, int k, const uint32_t *__restrict__ tabs, int64_t count,
                                    float *__restrict__ f32, double *__restrict__ f64)
{
    int cells = 1;
    for (int t = 0; t < k; t++) cells *= 3;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < count; c += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t *ct = tabs + c * 2 * cells;
        if (f32) f32[c] = table_mi_f32(d, ct, cells);
        if (f64) f64[c] = table_mi_f64(d, ct, cells);
    }
}

__global__ void publish_status_kernel(const int32_t *__restrict__ bits, int32_t *__restrict__ code)
{
    const int32_t b = *bits;
    int32_t c = EPI_OK;
    if (b & ST_TIMEOUT) c = EPI_ETIMEOUT;
    else if (b & ST_POOL_OVERFLOW) c = EPI_EOVERFLOW;
    else if (b & (ST_BAD_GENO | ST_BAD_PHENO)) c = EPI_EINVAL;
    else if (b) c = EPI_ECUDA;
    *code = c;
}

cudaError_t launch_publish_status(const int32_t *bits, int32_t *code, cudaStream_t st)
{
    publish_status_kernel<<<1, 1, 0, st>>>(bits, code);
    return cudaGetLastError();
}

__global__ void unrank_kernel(DevData d, int k, const uint64_t *__restrict__ ranks, int64_t count,
                              uint32_t *__restrict__ combs)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        int32_t c[EPI_MAX_ORDER];
        unrank_lex(d.binom, d.n, k, ranks[i], c);
        for (int t = 0; t < k; t++) combs[i * k + t] = (uint32_t)c[t];
    }
}

cudaError_t launch_unrank(const DevData &d, int k, const uint64_t *ranks, int64_t count, uint32_t *combs,
                          cudaStream_t st)
{
    int64_t g = (count + 255) / 256;
    if (g > 4096) g = 4096;
    unrank_kernel<<<(unsigned)(g < 1 ? 1 : g), 256, 0, st>>>(d, k, ranks, count, combs);
    return cudaGetLastError();
}

size_t finalize_smem_bytes(int pool) { return (size_t)next_pow2(pool < 2 ? 2 : pool) * 20; }

cudaError_t launch_merge(float *ls, uint64_t *lr, int32_t *lc, int nlists, int stride, int pool, float *out_s,
                         uint64_t *out_r, int32_t *out_n, cudaStream_t st, const uint32_t *thr, float floor)
{
    // entries one block takes: 4096, or twice the longest list
    int cap = stride;
    int64_t pitch = stride;
    int lstep = 1;
    for (int n = nlists;;) {
        const int room = 2 * cap > 4096 ? 2 * cap : 4096;
        const int group = n < room / cap ? n : room / cap;
        const int blocks = (n + group - 1) / group;
        const size_t smem = (size_t)merge_entries(group, cap, pool) * 12;
        cudaError_t e = cudaFuncSetAttribute(merge_level_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        const bool last = blocks == 1;
        merge_level_kernel<<<blocks, 1024, smem, st>>>(ls, lr, lc, n, pitch, lstep, group, cap, pool,
                                                       last ? out_s : nullptr, out_r, out_n, thr, floor);
        e = cudaGetLastError();
        if (e != cudaSuccess || last) return e;
        n = blocks;
        pitch *= group;
        lstep *= group;
        cap = pool;
    }
}

cudaError_t launch_rescore(const DevData &d, int k, int pool, const uint64_t *cand_r, const int32_t *cand_n,
                           uint32_t *counts, double *mi64, int32_t *combs, cudaStream_t st)
{
    rescore_kernel<<<pool, kRescoreThreads, 0, st>>>(d, k, cand_r, cand_n, counts, mi64, combs);
    return cudaGetLastError();
}

cudaError_t launch_finalize(const DevData &d, int k, int top_n, int pool, const float *cand_s, const uint64_t *cand_r,
                            const int32_t *cand_n, const double *mi64, const int32_t *combs, const uint32_t *counts,
                            const uint32_t *global_thr, uint64_t total, epi_result *out, uint32_t *out_counts,
                            int32_t *n_out, int32_t *status, cudaStream_t st)
{
    const size_t smem = finalize_smem_bytes(pool);
    cudaError_t e = cudaFuncSetAttribute(finalize_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    finalize_kernel<<<1, 1024, smem, st>>>(d, k, top_n, pool, cand_s, cand_r, cand_n, mi64, combs, counts, global_thr,
                                           total, out, out_counts, n_out, status);
    return cudaGetLastError();
}

cudaError_t launch_tables(const DevData &d, int k, const uint32_t *combs, int64_t count, uint32_t *out, int num_sms,
                          cudaStream_t st)
{
    int64_t g = count < (int64_t)num_sms * 8 ? count : (int64_t)num_sms * 8;
    if (g < 1) g = 1;
    tables_kernel<<<(unsigned)g, 256, 0, st>>>(d, k, combs, count, out);
    return cudaGetLastError();
}

cudaError_t launch_score_tables(const DevData &d, int k, const uint32_t *tabs, int64_t count, float *f32, double *f64,
                                int num_sms, cudaStream_t st)
{
    int64_t g = (count + 255) / 256;
    if (g > num_sms * 4) g = num_sms * 4;
    if (g < 1) g = 1;
    score_tables_kernel<<<(unsigned)g, 256, 0, st>>>(d, k, tabs, count, f32, f64);
    return cudaGetLastError();
}

// Exact single-precision MI of order-5 sets without materialising their
// tables (Section 2.2 counts, Eq. 1-3 in the cancellation-free form): one
// warp per set.  The set's 15 genotype rows are staged in shared memory in
// chunks of kS5Ch words (rows padded to an odd stride, so lanes reading the
// three genotype rows of one SNP hit distinct banks); lane l owns the
// four-SNP prefixes p = l, l + 32, l + 64 (p < 81; the lanes past 81 repeat
// prefix 0 and discard it) and, per word, counts popc(prefix & last-SNP
// genotype g) into case or control counters (the class of a word is uniform
// across the warp).  Cell x = 3 p + g; each lane sums the terms of its cells,
// the warp sums the lanes.  The summation order differs from the serial
// table sum, inside the same FP32 error bound.
constexpr int kS5Warps = 8, kS5Ch = 64, kS5Pad = kS5Ch + 1;

__global__ void __launch_bounds__(kS5Warps * 32) score5_f32_kernel(DevData d, const uint32_t *__restrict__ combs,
                                                                  int64_t count, float *__restrict__ out)
{
    __shared__ uint32_t rows[kS5Warps][15][kS5Pad];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t(*R)[kS5Pad] = rows[warp];
    const MiConstF32 mc = make_mi_const(d.m, d.m1, d.m0);
    const int Wt = d.Wt, W1 = d.W1;
    // the lane's prefixes: row index t * 3 + g_t of the four prefix SNPs
    int off[3][4];
    bool valid[3];
#pragma unroll
    for (int j = 0; j < 3; j++) {
        const int p0 = lane + 32 * j;
        valid[j] = p0 < 81;
        const int p = valid[j] ? p0 : 0;
        off[j][0] = p / 27;
        off[j][1] = 3 + (p / 9) % 3;
        off[j][2] = 6 + (p / 3) % 3;
        off[j][3] = 9 + p % 3;
    }
    for (int64_t s = (int64_t)blockIdx.x * kS5Warps + warp; s < count; s += (int64_t)gridDim.x * kS5Warps) {
        const uint32_t *src[5];
#pragma unroll
        for (int t = 0; t < 5; t++) src[t] = d.masks + (int64_t)combs[s * 5 + t] * 3 * Wt;
        uint32_t cc[3][3] = {}, ck[3][3] = {};
        for (int c0 = 0; c0 < Wt; c0 += kS5Ch) {
            const int cw = min(kS5Ch, Wt - c0);
            __syncwarp();
#pragma unroll
            for (int r = 0; r < 15; r++)
                for (int w = lane; w < cw; w += 32) R[r][w] = src[r / 3][(r % 3) * Wt + c0 + w];
            __syncwarp();
            const int split = min(max(W1 - c0, 0), cw);   // words [0, split) are cases
            auto word = [&](int w, uint32_t (&acc)[3][3]) {
                const uint32_t l0 = R[12][w], l1 = R[13][w], l2 = R[14][w];
#pragma unroll
                for (int j = 0; j < 3; j++) {
                    const uint32_t pw = R[off[j][0]][w] & R[off[j][1]][w] & R[off[j][2]][w] & R[off[j][3]][w];
                    acc[j][0] += __popc(pw & l0);
                    acc[j][1] += __popc(pw & l1);
                    acc[j][2] += __popc(pw & l2);
                }
            };
            for (int w = 0; w < split; w++) word(w, cc);
            for (int w = split; w < cw; w++) word(w, ck);
        }
        SumF32 acc;
#pragma unroll
        for (int j = 0; j < 3; j++)
            if (valid[j]) {
#pragma unroll
                for (int g = 0; g < 3; g++) acc.add(cell_terms_f32(cc[j][g], ck[j][g], mc));
            }
        float v = acc.value();
#pragma unroll
        for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) out[s] = __fdiv_rn(v, mc.fm);
    }
}

cudaError_t launch_score5_f32(const DevData &d, const uint32_t *combs, int64_t count, float *out, int num_sms,
                              cudaStream_t st)
{
    if (count <= 0) return cudaSuccess;
    int64_t g = (count + kS5Warps - 1) / kS5Warps;
    if (g > (int64_t)num_sms * 6) g = (int64_t)num_sms * 6;
    score5_f32_kernel<<<(unsigned)g, kS5Warps * 32, 0, st>>>(d, combs, count, out);
    return cudaGetLastError();
}

// Ranks rank_base + i of the scores at or above thr (any order), appended
// while they fit in `cap`; *n counts all of them.
__global__ void select_ge_kernel(const float *__restrict__ scores, int64_t count, float thr, uint64_t rank_base,
                                 uint64_t *__restrict__ out, uint64_t cap, unsigned long long *__restrict__ n)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        const float v = scores[i];
        if (v >= thr) {
            const unsigned long long at = atomicAdd(n, 1ull);
            if (at < cap) out[at] = rank_base + (uint64_t)i;
        }
    }
}

cudaError_t launch_select_ge(const float *scores, int64_t count, float thr, uint64_t rank_base, uint64_t *out,
                             uint64_t cap, unsigned long long *n, int num_sms, cudaStream_t st)
{
    if (count <= 0) return cudaSuccess;
    int64_t g = (count + 255) / 256;
    if (g > (int64_t)num_sms * 8) g = (int64_t)num_sms * 8;
    select_ge_kernel<<<(unsigned)g, 256, 0, st>>>(scores, count, thr, rank_base, out, cap, n);
    return cudaGetLastError();
}

}  // namespace epi
