// High orders by histogram.
//
// A table of order 6-8 has 729 to 6561 cells a class, more than most studies
// have individuals, and a bitwise AND and population count visits every cell
// for every word of the sample.  Here the individuals are visited instead
// (Section 2.1's table, filled one individual at a time): each adds one to its
// cell of a shared-memory table, reads the finished cell back, adds its share
// of the score, and clears the cell.  The empty cells are never touched, and
// the work per combination is three shared accesses an individual whatever
// the order.
//
// Eq. 1-3 as a sum over individuals i with cell counts own_i (of i's class)
// and n_i (of both classes):
//     m MI = sum_i [ln own_i - ln n_i] + m ln m - m1 ln m1 - m0 ln m0,
// with ln from a table in fixed point (2^-44), so the sum is exact in any
// order and the score is rounded once, to FP32: its error is at most
// 2^-24 MI + 2^-43 (the logarithms' roundings, at most two units an
// individual).  Below an MI of 2^-19, where the second part would be the larger
// (balanced or nearly constant genotypes; the margin of the exact top N needs
// a relative bound, and an MI of zero has to score zero), the combination is
// counted again and its cells scored in the cancellation-free form, in double
// precision.
//
// What bounds it is shared memory: per individual one atomic add, a read and a
// clear at scattered cells (about 3.5 wavefronts a warp) and two reads of the
// logarithms.  23 x 2048 at order 8, 490314 combinations: 2.38 ms (shared-memory
// data pipe 80 % of its peak; 2.35 without the recount of small scores), where the
// bitwise kernel on prefix tables took 35 ms; 3.8 ms with 98 registers a
// thread instead of 64 (two CTAs an SM instead of four) and a predicate per
// item for the places without an individual.
//
// Rare variants put most individuals into one cell, and an atomic add takes the
// lanes of one cell in turn: order 6, 40 x 2048, 18.7 ms at allele frequencies
// of 0.05-0.5, 29.7 at 0.01-0.05 and 34.6 at 0.001-0.01 (the bitwise kernel 30
// at all of them).  Studies whose commonest cell is expected to hold
// kCrowdShare of the individuals run a kernel whose warps look, prefix by
// prefix, for a cell that half of their lanes share, and add that crowd once:
// 18.6 and 15.9 ms.  The look costs the others 1 to 3 %, hence the two
// kernels; they meet at a share of 0.3 to 0.4 (frequencies 0.02-0.15: order 6
// 23.7 plain and 22.5, order 7, 26 x 2048, 4.38 and 4.48, order 8, 23 x 2048,
// 3.78 and 3.89; 0.01-0.1: 26.6 and 21.1, 4.83 and 4.52, 4.12 and 4.08).
//
// GPU mapping: persistent CTAs with contiguous rank ranges, one table (4-byte
// cells, cases in the upper half) a CTA and as many CTAs as fit.  A thread
// keeps its kItems individuals' cell of the first K-1 and K-2 SNPs in
// registers; genotypes are 4-bit fields (4 x genotype, a byte offset) of one
// word per eight individuals.  A warp's individuals are all cases or all
// controls, 32 of a mask word per item; places without an individual count in
// a cell of their lane and class past the table, where they add ln c - ln c.
#include <algorithm>

#include "epi_host.h"
#include "epi_internal.cuh"

namespace epi {
namespace hist {

constexpr int kLogShared = 1024;    // ln table entries in shared memory
constexpr int kBuffer = 192;        // candidates between sorts
constexpr double kCrowdShare = 0.33;
constexpr int kCrowd = 16;          // individuals of a warp that make a crowd
constexpr double kLnScale = 17592186044416.0;   // 2^44

__host__ __device__ constexpr int cells_of(int k) { return k <= 0 ? 1 : 3 * cells_of(k - 1); }
__host__ __device__ constexpr int ln_offset(int k) { return ((cells_of(k) + 64) * 4 + 15) & ~15; }

struct Params {
    DevData d;
    uint64_t rank_begin, rank_end;
    const uint32_t *geno;           // [n][words][threads]: 4-bit fields of 4 x genotype
    const long long *ln;            // ln c 2^44 for c = 0 .. m (0 at 0)
    int32_t pool, cand_p2, top_n;
    int32_t case_warps;             // the first warps of a CTA hold the cases
    uint32_t *global_thr;
    float *list_score;              // [grid][pool]
    uint64_t *list_rank;
    int32_t *list_count;
    float *all_scores;              // optional: [rank - rank_begin]
};

// next (k-1)-subset of [0, n-1) in lex order: the first place that changed,
// or -1 after the last
__device__ inline int next_prefix(int32_t *p, int km1, int64_t n)
{
    int t = km1 - 1;
    while (t >= 0 && p[t] == n - 1 - km1 + t) t--;
    if (t < 0) return -1;
    p[t]++;
    for (int v = t + 1; v < km1; v++) p[v] = p[v - 1] + 1;
    return t;
}

// The mask word of item i of a warp, -1 past its class's words.
__device__ __forceinline__ int word_of(const DevData &d, int i, int warp, int warps, int case_warps)
{
    const bool ca = warp < case_warps;
    const int w = ca ? i * case_warps + warp : d.W1 + i * (warps - case_warps) + warp - case_warps;
    return w < (ca ? d.W1 : d.Wt) ? w : -1;
}

__global__ void __launch_bounds__(256) build_kernel(DevData d, int threads, int case_warps, int words,
                                                    uint32_t *__restrict__ geno, long long *__restrict__ ln)
{
    const int64_t total = d.n * words * threads;
    const int warps = threads / 32;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int t = (int)(e % threads);
        const int64_t s = e / threads / words;
        const int q = (int)(e / threads % words);
        uint32_t out = 0;
        for (int i = 0; i < 8; i++) {
            const int w = word_of(d, 8 * q + i, t / 32, warps, case_warps);
            if (w < 0) break;
            const uint32_t g1 = d.masks[(s * 3 + 1) * d.Wt + w] >> (t & 31) & 1u;
            const uint32_t g2 = d.masks[(s * 3 + 2) * d.Wt + w] >> (t & 31) & 1u;
            out |= (4u * g1 + 8u * g2) << (4 * i);
        }
        geno[e] = out;
    }
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c <= d.m; c += (int64_t)gridDim.x * blockDim.x)
        ln[c] = c > 0 ? llrint(log((double)c) * kLnScale) : 0;
}

struct State {
    int64_t rank;                    // of the combination (prefix, last)
    int32_t pre[kMaxOrderGpu];
    int32_t last, from;              // the prefix's first last SNP here; first changed place
    int32_t list_len, nbuf, done, published, small;
    float thr;
};

__device__ inline void flush(State &S, float *sc, uint64_t *rk, const Params &P)
{
    __syncthreads();
    const int live = S.list_len + S.nbuf;
    const int p2 = next_pow2(live < 2 ? 2 : live);
    for (int i = live + threadIdx.x; i < p2 && i < P.cand_p2; i += blockDim.x) { sc[i] = -1.0f; rk[i] = ~0ull; }
    __syncthreads();
    block_sort_cands(sc, rk, p2);
    if (threadIdx.x == 0) {
        S.list_len = live < P.pool ? live : P.pool;
        S.nbuf = 0;
        float t = S.thr;
        if (S.list_len == P.pool) t = fmaxf(t, sc[P.pool - 1]);
        // top_n combinations score at least the top_n-th here: nothing below
        // it, less the final margin check's bound (four times over), is asked
        if (P.top_n > 0 && S.list_len >= P.top_n)
            t = fmaxf(t, sc[P.top_n - 1] * (float)(1.0 - 4.0 * f32_rel_bound(kMaxOrderGpu, P.d.m)));
        if (t > 0.0f) {
            atomicMax(P.global_thr, __float_as_uint(t));
            S.thr = t;
        }
    }
    __syncthreads();
}

// MI of the block's table in double precision, without cancellation: the cells
// shared out over the threads, the sums added in a fixed order.  Out of line,
// so that its registers are not the counting loop's.
__device__ __noinline__ double precise_mi(const uint32_t *tab, int cells, int64_t m1, int64_t m0, int64_t m,
                                          long long *part)
{
    double x = 0.0;
    for (int c = threadIdx.x; c < cells; c += blockDim.x) {
        const uint32_t a = tab[c] >> 16, n = a + (tab[c] & 0xffffu);
        x += mi_term_f64(a, n, m1, m);
        x += mi_term_f64(n - a, n, m0, m);
    }
    for (int off = 16; off; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = __double_as_longlong(x);
    __syncthreads();
    x = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) x += __longlong_as_double(part[w]);
    return x / (double)m;
}

template <int K, int kItems, bool CROWDS>
__global__ void __launch_bounds__(kItems == 8 ? 512 : 1024, kItems == 8 ? 2 : 1) hist_kernel(Params P)
{
    constexpr int kWords = kItems / 8;
    const DevData d = P.d;
    extern __shared__ __align__(16) unsigned char smem[];
    // cells, 64 spare ones | ln table | candidate ranks | candidate scores
    constexpr int kCells = cells_of(K);
    unsigned char *tab = smem;
    long long *ln = reinterpret_cast<long long *>(smem + ln_offset(K));
    uint64_t *rk = reinterpret_cast<uint64_t *>(ln + kLogShared);
    float *sc = reinterpret_cast<float *>(rk + P.cand_p2);
    __shared__ State S;
    __shared__ long long part[32];

    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, warps = blockDim.x >> 5;
    const uint64_t span = P.rank_end - P.rank_begin;
    const int64_t R_b = (int64_t)(P.rank_begin + (uint64_t)(((unsigned __int128)span * blockIdx.x) / gridDim.x));
    const int64_t R_e = (int64_t)(P.rank_begin + (uint64_t)(((unsigned __int128)span * (blockIdx.x + 1)) / gridDim.x));
    for (int c = t; c < kLogShared && c <= d.m; c += blockDim.x) ln[c] = P.ln[c];
    for (int c = t; c < kCells + 64; c += blockDim.x) reinterpret_cast<uint32_t *>(tab)[c] = 0;
    if (t == 0) {
        S.list_len = 0; S.nbuf = 0; S.thr = -1.0f; S.published = 0;
        S.done = R_b >= R_e;
        S.rank = R_b;
        S.from = 0;
        if (!S.done) {
            int32_t c[kMaxOrderGpu];
            unrank_lex(d.binom, d.n, K, (uint64_t)R_b, c);
            for (int q = 0; q < K - 1; q++) S.pre[q] = c[q];
            S.last = c[K - 1];
        }
    }
    const bool is_case = warp < P.case_warps;
    const uint32_t sh = is_case ? 16u : 0u, inc = is_case ? 0x10000u : 1u;
    const uint32_t spare = 4u * (kCells + (is_case ? 32 : 0) + lane);
    uint32_t valid = 0;
#pragma unroll
    for (int i = 0; i < kItems; i++) {
        const int w = word_of(d, i, warp, warps, P.case_warps);
        if (w >= 0) valid |= ((d.masks[w] | d.masks[d.Wt + w] | d.masks[2 * d.Wt + w]) >> lane & 1u) << i;
    }
    const long long base = d.m * P.ln[d.m] - d.m1 * P.ln[d.m1] - d.m0 * P.ln[d.m0];
    const double scale = 1.0 / ((double)d.m * kLnScale);
    const long long small = (long long)d.m << 25;   // an MI of 2^-19
    uint32_t c6[kItems], c7[kItems];   // byte offsets of the first K-2 and K-1 SNPs' cells, times 3
#pragma unroll
    for (int i = 0; i < kItems; i++) c6[i] = c7[i] = 0;
    __syncthreads();

    auto geno = [&](int snp, uint32_t (&g)[kWords]) {
#pragma unroll
        for (int q = 0; q < kWords; q++) g[q] = __ldg(P.geno + ((int64_t)snp * kWords + q) * blockDim.x + t);
    };
    while (!S.done) {
        // ---- the prefix's cells
        uint32_t g[kWords];
        if (S.from < K - 2) {
#pragma unroll
            for (int i = 0; i < kItems; i++) c6[i] = 0;
#pragma unroll
            for (int q = 0; q < K - 2; q++) {
                geno(S.pre[q], g);
#pragma unroll
                for (int i = 0; i < kItems; i++) c6[i] = 3 * (c6[i] + (g[i / 8] >> (4 * (i % 8)) & 12u));
            }
        }
        geno(S.pre[K - 2], g);
#pragma unroll
        for (int i = 0; i < kItems; i++)
            c7[i] = valid >> i & 1u ? 3 * (c6[i] + (g[i / 8] >> (4 * (i % 8)) & 12u)) : spare;
        // a cell of the prefix that kCrowd of the warp's first items share: lane
        // 0's or (low bit set) lane 13's
        uint32_t crowd = ~0u;
        if constexpr (CROWDS) {
            const uint32_t a = __shfl_sync(0xffffffffu, c7[0], 0), b = __shfl_sync(0xffffffffu, c7[0], 13);
            const int na = __popc(__ballot_sync(0xffffffffu, c7[0] == a));
            const int nb = __popc(__ballot_sync(0xffffffffu, c7[0] == b));
            if (max(na, nb) >= kCrowd) crowd = na >= nb ? a : b | 1u;
        }
        const int64_t r0 = S.rank;
        const int j0 = S.last;
        const int nj = (int)min((int64_t)(d.n - j0), R_e - r0);
        geno(j0, g);
        auto record = [&](float score, int jj) {
            if (P.all_scores) P.all_scores[r0 + jj - (int64_t)P.rank_begin] = score;
            if (score >= S.thr) {
                const int pos = S.list_len + S.nbuf++;
                sc[pos] = score;
                rk[pos] = (uint64_t)(r0 + jj);
            }
        };
#pragma unroll 1
        for (int jj = 0; jj < nj; jj++) {
            uint32_t at[kItems];
#pragma unroll
            for (int i = 0; i < kItems; i++) at[i] = c7[i] + (g[i / 8] >> (4 * (i % 8)) & 12u);
            if (!CROWDS || crowd == ~0u) {
#pragma unroll
                for (int i = 0; i < kItems; i++) atomicAdd(reinterpret_cast<uint32_t *>(tab + at[i]), inc);
            } else {
                // the crowd's cell once for the warp
                const uint32_t its = (crowd & ~1u) + (__shfl_sync(0xffffffffu, g[0], crowd & 1u ? 13 : 0) & 12u);
                uint32_t many = 0;
#pragma unroll
                for (int i = 0; i < kItems; i++) {
                    many += __popc(__ballot_sync(0xffffffffu, at[i] == its));
                    if (at[i] != its) atomicAdd(reinterpret_cast<uint32_t *>(tab + at[i]), inc);
                }
                if (lane == 0) atomicAdd(reinterpret_cast<uint32_t *>(tab + its), inc * many);
            }
            if (jj + 1 < nj) geno(j0 + jj + 1, g);
            __syncthreads();
            long long s = 0;
            uint32_t v[kItems], most = 0;
#pragma unroll
            for (int i = 0; i < kItems; i++) {
                v[i] = *reinterpret_cast<const uint32_t *>(tab + at[i]);
                most |= (v[i] >> 16) + (v[i] & 0xffffu);
            }
            if (!__any_sync(0xffffffffu, most >= kLogShared)) {
#pragma unroll
                for (int i = 0; i < kItems; i++)
                    s += ln[v[i] >> sh & 0xffffu] - ln[(v[i] >> 16) + (v[i] & 0xffffu)];
            } else {
#pragma unroll
                for (int i = 0; i < kItems; i++)
                    s += __ldg(P.ln + (v[i] >> sh & 0xffffu)) - __ldg(P.ln + ((v[i] >> 16) + (v[i] & 0xffffu)));
            }
            // |s| < 2^52: 32 lanes' lower 26 and upper bits each fit a word
            const uint32_t lo = __reduce_add_sync(0xffffffffu, (uint32_t)s & 0x3ffffffu);
            const int32_t hi = __reduce_add_sync(0xffffffffu, (int32_t)(s >> 26));
            if (lane == 0) part[warp] = ((long long)hi << 26) + lo;
            __syncthreads();
#pragma unroll
            for (int i = 0; i < kItems; i++)
                *reinterpret_cast<uint32_t *>(tab + at[i]) = 0;
            if (t == 0) {
                long long sum = base;
                for (int w = 0; w < warps; w++) sum += part[w];
                S.small = sum < small;
                if (sum >= small) record((float)((double)sum * scale), jj);
            }
            __syncthreads();
            if (S.small) {
                uint32_t again[kWords];
                geno(j0 + jj, again);
#pragma unroll
                for (int i = 0; i < kItems; i++) {
                    at[i] = c7[i] + (again[i / 8] >> (4 * (i % 8)) & 12u);
                    atomicAdd(reinterpret_cast<uint32_t *>(tab + at[i]), inc);
                }
                __syncthreads();
                const double mi = precise_mi(reinterpret_cast<const uint32_t *>(tab), kCells, d.m1, d.m0, d.m, part);
#pragma unroll
                for (int i = 0; i < kItems; i++) *reinterpret_cast<uint32_t *>(tab + at[i]) = 0;
                if (t == 0) record((float)mi, jj);
                __syncthreads();
            }
            if (S.nbuf == kBuffer || (!S.published && P.top_n > 0 && S.list_len + S.nbuf >= P.top_n)) {
                flush(S, sc, rk, P);
                if (t == 0 && S.list_len >= P.top_n) S.published = 1;
                __syncthreads();
            }
        }
        __syncthreads();
        if (t == 0) {
            S.rank = r0 + nj;
            const int from = S.rank < R_e ? next_prefix(S.pre, K - 1, d.n) : -1;
            S.done = from < 0;
            S.from = from;
            S.last = S.pre[K - 2] + 1;
            const float gthr = __uint_as_float(*(volatile uint32_t *)P.global_thr);
            if (gthr > 0.0f) S.thr = fmaxf(S.thr, gthr);
        }
        __syncthreads();
    }
    if (S.nbuf > 0) flush(S, sc, rk, P);
    __syncthreads();
    for (int i = t; i < S.list_len; i += blockDim.x) {
        P.list_score[(size_t)blockIdx.x * P.pool + i] = sc[i];
        P.list_rank[(size_t)blockIdx.x * P.pool + i] = rk[i];
    }
    if (t == 0) P.list_count[blockIdx.x] = S.list_len;
}

// Whether a study's commonest cell is expected to hold kCrowdShare of the
// individuals.
static bool crowds(const DevData &d, int k) { return pow((double)d.top_share, k) >= kCrowdShare; }

// Warps of a CTA: those of cases, then those of controls; and items a thread,
// 8 while that is at most 16 warps.
static int class_warps(int32_t words, int items) { return (words + items - 1) / items; }
static int warps_of(const DevData &d, int items) { return class_warps(d.W1, items) + class_warps(d.Wt - d.W1, items); }
static int items_of(const DevData &d) { return warps_of(d, 8) <= 16 ? 8 : 16; }
static int threads_of(const DevData &d) { return 32 * warps_of(d, items_of(d)); }

static const void *kernel_of(const DevData &d, int k)
{
    static const void *const kernels[3][2][2] = {
        {{(const void *)hist_kernel<6, 8, false>, (const void *)hist_kernel<6, 8, true>},
         {(const void *)hist_kernel<6, 16, false>, (const void *)hist_kernel<6, 16, true>}},
        {{(const void *)hist_kernel<7, 8, false>, (const void *)hist_kernel<7, 8, true>},
         {(const void *)hist_kernel<7, 16, false>, (const void *)hist_kernel<7, 16, true>}},
        {{(const void *)hist_kernel<8, 8, false>, (const void *)hist_kernel<8, 8, true>},
         {(const void *)hist_kernel<8, 16, false>, (const void *)hist_kernel<8, 16, true>}}};
    return k >= 6 && k <= 8 ? kernels[k - 6][items_of(d) == 16][crowds(d, k)] : nullptr;
}

}  // namespace hist

int hist_cand_p2(int pool) { return next_pow2(pool + hist::kBuffer); }

size_t hist_smem_bytes(int k, int pool)
{
    return (size_t)hist::ln_offset(k) + (size_t)hist::kLogShared * 8 + (size_t)hist_cand_p2(pool) * 12;
}

// Orders 6-8 of up to 16384 individuals (1024 threads of 16; a little fewer
// where the classes' last words are not full).
bool hist_applies(const DevData &d, int k, int pool)
{
    if (k < 6 || k > 8 || hist::warps_of(d, 16) > 32) return false;
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return false;
    return hist_smem_bytes(k, pool) + 2048 <= (size_t)optin;
}

size_t hist_geno_words(const DevData &d)
{
    return (size_t)d.n * (hist::items_of(d) / 8) * hist::threads_of(d);
}

int hist_grid(int num_sms, const DevData &d, int k, int pool)
{
    const void *kern = hist::kernel_of(d, k);
    const size_t smem = hist_smem_bytes(k, pool);
    int occ = 0;
    if (!kern || cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, hist::threads_of(d), smem) != cudaSuccess || occ < 1)
        return num_sms;
    return num_sms * occ;
}

cudaError_t launch_hist_search(const DevData &d, int k, uint64_t rank_begin, uint64_t rank_end, int pool, int top_n,
                               uint32_t *global_thr, float *list_score, uint64_t *list_rank, int32_t *list_count,
                               int grid, float *all_scores, uint32_t *geno, long long *ln, cudaStream_t st)
{
    hist::Params p;
    p.d = d;
    p.rank_begin = rank_begin;
    p.rank_end = rank_end;
    p.geno = geno;
    p.ln = ln;
    p.pool = pool;
    p.cand_p2 = hist_cand_p2(pool);
    p.top_n = all_scores ? 0 : top_n;
    p.case_warps = hist::class_warps(d.W1, hist::items_of(d));
    p.global_thr = global_thr;
    p.list_score = list_score;
    p.list_rank = list_rank;
    p.list_count = list_count;
    p.all_scores = all_scores;
    const int items = hist::items_of(d), threads = hist::threads_of(d);
    const void *kern = hist::kernel_of(d, k);
    if (!kern) return cudaErrorInvalidValue;
    const size_t smem = hist_smem_bytes(k, pool);
    const int64_t total = std::max<int64_t>((int64_t)hist_geno_words(d), d.m + 1);
    hist::build_kernel<<<(unsigned)std::min<int64_t>((total + 255) / 256, 1024), 256, 0, st>>>(
        d, threads, p.case_warps, items / 8, geno, ln);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    void *args[] = {&p};
    e = cudaLaunchKernel(kern, dim3((unsigned)grid), dim3((unsigned)threads), args, smem, st);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace epi
