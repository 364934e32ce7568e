// Tensor-core counting path of the exhaustive search (tcgen05, sm_103a).
//
// The last combination level of Section 2.2 (AND of the prefix table with
// the last SNP's table, then popcount) is an exact 0/1 matrix product:
//     count[(p, x'), (j, g)] = sum over individuals s of A[(p, x')][s] * B[(j, g)][s]
// with A[(p, x')] the genotype-table row x' of prefix p (Section 2.1) and
// B[(j, g)] row g of SNP j, summed separately over the case and the control
// individuals.  Both operands hold 0/1 patterns as FP4 E2M1 nibbles
// (kind::mxf4: K = 64 per MMA, twice that of the FP8 kinds, and half their
// operand bytes) and the MMA accumulates in FP32 in tensor memory.  Because
// the product sums over K, any fixed permutation of the individuals inside a K step, applied to both
// operands, leaves the counts unchanged, and the two operands may carry
// different weights per K position as long as their product is constant:
//   * 32-bit word i (of 4) of the 16 bytes of a mask word holds, in nibble b,
//     individual 4 b + i: the A producer turns one mask word into four output
//     words with one AND each (and one shift: nibble bit 3 is the sign);
//   * A's nonzero nibble in word i is 0.5, 1, 2 or 2 (1, 2, 4, 4) and B's is
//     the reciprocal, so every product of two ones is exactly 1.
// kind::mxf4 multiplies every 32 K elements of a row by a power-of-two scale
// kept in tensor memory.  All scales of A are 1; B's case blocks take 2^p and
// its control blocks 1 in the combined-class variant, so one accumulator
// holds ctrl + case 2^p.  Sums of such integers below 2^24 are exact in FP32
// (measured against integer counts up to 2^23.96, and on every table of the
// validation datasets).
// Genotype 2 of the last SNP is obtained by subtraction from the prefix
// row's total, as in the popcount path.
//
// Layout of one tile: M = 128 rows = 4 warps x 32 lanes; each warp holds
// floor(32 / 3^(k-1)) whole prefixes (prefix rows never straddle a warp, so
// the epilogue reduces a prefix within a warp; at order 5 one prefix takes 81
// rows of three warps); N = 240 columns = 120 last SNPs x genotypes {0, 1}
// (combined classes) or 160 columns per class (separate classes); K = 256
// individuals per stage.  Columns come in groups of four: genotype 0 of SNPs
// j, j + 1 (j even), then genotype 1 of both, so the epilogue's packed
// two-lane arithmetic takes two SNPs at a time; a tile's first SNP is even.
// Prefixes are taken in "panel order" (by their last SNP c ascending) so the
// last SNPs of a tile, j > c, form one contiguous range.  A lexicographic rank
// range [r0, r1) of combinations covers the first SNPs s1 in [a, b] (those of
// ranks r0 and r1 - 1); within a panel the prefixes are listed
// lexicographically, so the ones with s1 in [a, b] are contiguous, and the
// epilogue keeps, per prefix, only the last SNPs whose combination's rank lies
// in [r0, r1) (consecutive ranks share their prefix and differ in the last
// SNP, so that is one interval of j).
//
// Warp roles (one CTA per SM, persistent, segments of work items spread over
// the panels; an item = one M tile x one N tile x the whole K range; the
// epilogue/producer split is Roles<K> below):
//   epilogue warps (first): TMEM -> registers, single-precision MI screen,
//               exact-margin candidate selection, per-CTA candidate list;
//               warp w reads TMEM lane quadrant w % 4 for the chunks of 8
//               last SNPs w / 4, w / 4 + G, ... (G warps per quadrant)
//   A producers: prefix rows = AND of the prefix SNPs' bit rows, expanded
//               to FP4 nibbles in the 128-byte-swizzled K-major layout; one
//               thread per row, groups of 4 warps taking the ring's stages
//               in turn, own stages prefetched
//   next warp   TMA producer of B tiles, and writer of the item descriptors
//   last warp   TMEM allocator and MMA issuer (one elected thread)
// Every mbarrier wait is bounded (about 2 s); a wait that gives up sets
// ST_TIMEOUT and all roles leave their loops, drain their own asynchronous
// work and free tensor memory.
#include <cuda.h>
#include <cstring>
#include <cudaTypedefs.h>

#include "epi_host.h"
#include "epi_internal.cuh"
#include "epi_tcgen05.cuh"

namespace epi {

namespace tc {

constexpr int kChunk = 128;            // individuals a class is padded to
constexpr int kRowBytes = 128;         // operand bytes of a row and K stage (256 individuals)
constexpr int kTileBytes = 128 * kRowBytes;   // one A stage

// Tile shapes of the two variants.
//   combined classes (C = true): one accumulator per tile holds
//     ctrl + case 2^p (exact while below 2^24), two of 240 columns in turn;
//   separate classes (C = false): two accumulators per tile, three of 160
//     columns in rotation (the next tile's case accumulator fills while the
//     epilogue reads this tile's two).  480 columns either way: the other 32
//     hold the scale factors.
// The MMA of an N tile that ends the last SNPs is cut to the columns in use
// (a multiple of 16).
template <bool C>
struct Shape {
    static constexpr int J = C ? 120 : 80;          // last SNPs per N tile
    static constexpr int N = 2 * J;                 // tile columns per accumulator
    static constexpr int Stages = C ? 4 : 5;        // K stages in the rings
    static constexpr int BBytes = N * kRowBytes;    // one B stage
    static constexpr int Accs = C ? 2 : 3;          // accumulators in rotation
    static constexpr int AccPerTile = C ? 1 : 2;
};
constexpr int kScaleACol = 480, kScaleBCol = 496;   // 16 tensor-memory columns each

// Epilogue and producer warps (tuning parameters).
#ifndef EPI_TC_EPI_WARPS
#define EPI_TC_EPI_WARPS 8
#endif
#ifndef EPI_TC_PROD_WARPS
#define EPI_TC_PROD_WARPS 4
#endif

struct Roles {
    static constexpr int EpiWarps = EPI_TC_EPI_WARPS;
    static constexpr int ProdWarps = EPI_TC_PROD_WARPS;
    static constexpr int Threads = 32 * (EpiWarps + ProdWarps + 2);   // + the TMA and MMA warps
    static constexpr int EpiThreads = 32 * EpiWarps;
    static constexpr int ProdGroups = ProdWarps / 4;  // one thread per tile row each
    static constexpr int ColGroups = EpiWarps / 4;    // epilogue warps per lane quadrant
    static_assert(EpiWarps % 4 == 0 && ProdWarps % 4 == 0, "roles come in whole lane quadrants");
};
// A producers' load distance in own stages
#ifndef EPI_TC_PREFETCH
#define EPI_TC_PREFETCH 4
#endif
constexpr int kDescDepth = 4;
constexpr int kWaitSlots = 8;
constexpr int kMaxDescSnps = 40;
constexpr unsigned long long kTimeoutNs = 2000000000ull;

struct Desc {
    int32_t j0;          // first last-SNP of the N tile
    int32_t j1;          // pair tiles: the SNP before it
    int32_t nvalid;      // real prefixes in the M tile
    int32_t pad;
    uint64_t single[kMaxDescSnps];   // prefix p's place in the single-count table (groups)
    int32_t snp[kMaxDescSnps];   // prefix p occupies snp[p*(k-1) .. p*(k-1)+k-2] (k - 2 SNPs each with pairs)
};

// One dataset of a launch; a batched launch covers several datasets of the
// same order, CTAs [cta_begin, cta_begin + cta_count) working on this one.
struct DsParams {
    DevData d;
    uint64_t n_prefix;         // prefixes searched (first SNP in [s1_lo, s1_hi])
    uint64_t n_items;
    const uint4 *rows;         // the producers' masks [stage][n][3][2] (16 bytes each)
    const uint64_t *item_cum;  // [n + 1] items of M tiles starting in panels < c
    const uint64_t *pcum;      // [n + 1] prefixes searched in panels < c
    // pair tiles and the single counts behind them (see the pair section
    // below): [n + 1] groups of singles in panels < c; items and operand rows
    // of the pairs whose first SNP is below j1
    const uint64_t *scum;
    const uint64_t *brow;
    float4 *singles;
    int store;                 // 1: write the single counts instead of scoring
    uint64_t rank_begin, rank_end;   // lexicographic ranks searched
    int32_t s1_lo, s1_hi;      // first SNPs of ranks rank_begin and rank_end - 1
    int32_t clip;              // 0: the whole combination range
    int32_t comb_p;            // combined-class variant: control counts in the low comb_p bits
    int top_n;                 // records wanted (0: the pool alone sets the threshold)
    float thr_mul;             // 1 - 4 f32_rel_bound: from a top_n-th best score to a safe threshold
    int chunks, chunks_case;   // 128-individual chunks in total / over the cases
    // screen (see Screen below): MI bound = v vscale + voff; a combination
    // passes when that reaches thr cut_mul - cut_add
    int poly;                  // polynomial bound, else fast logarithms
    float vscale, voff, cut_mul, cut_add;
    float sc_pi, c2, c3, c4, c5a, c5b;
    uint64_t total;            // C(n, k)
    uint32_t *global_thr;
    uint32_t *hist;            // [kTcHistBins] scores of the combinations kept so far, by value
    const CUtensorMap *tmap;   // B-operand map in global memory (batched launches)
    int32_t cta_begin, cta_count;
};

struct Params {
    DsParams one;              // the dataset when the launch has one
    const DsParams *many;      // else [n_ds] in device memory
    const int32_t *cta_ds;     // and the dataset of each CTA
    int pool, cand_p2;
    // the CTA's candidate buffer [cand_p2] in global memory (per CTA, at
    // blockIdx.x * cand_p2) where it does not fit in shared memory; NULL:
    // shared memory
    float *cand_score_g;
    uint64_t *cand_rank_g;
    float *list_score;
    uint64_t *list_rank;
    int32_t *list_count;
    int32_t *status;
    float *scores;                // orders 3-4: every combination's score, by rank (nothing is kept)
    const long long *tlog;        // with scores: n ln n 2^46 for n = 0 .. m, rounded
    TcCollect collect;            // of a collecting launch
    unsigned long long wait_ns;   // limit of the pipeline waits (0: kTimeoutNs)
    uint32_t *dump;            // optional: every table, [rank][2][3^k] (validation)
    unsigned long long *waits; // optional: [grid][8] cycles spent waiting, per role (tracing)
};

// ------------------------------------------------------------------ PTX --
// Limit of the pipeline waits of this CTA (set at start from Params.wait_ns,
// the default kTimeoutNs when 0).  The drain waits at exit always use
// kTimeoutNs, so that no asynchronous copy or MMA is outstanding when the CTA
// leaves.
__shared__ unsigned long long g_wait_limit_ns;
// The item at which every role ends, set where a collecting pass has found
// more than the caller's array holds (none: ~0).
__shared__ volatile uint32_t g_end_item;

// Bounded wait for the phase of parity `parity`; false when it gave up (the
// CTA-wide abort flag is then set).
__device__ __noinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag)
{
    if (mbar_try(bar, parity)) return true;
    const uint64_t t0 = now_ns();
    const unsigned long long limit = g_wait_limit_ns;
    for (;;) {
        if (mbar_try(bar, parity)) return true;
        if (*abort_flag) return false;
        if (now_ns() - t0 > limit) {
            *abort_flag = 1;
            return false;
        }
    }
}

// The wait for an item's descriptor; in a collecting pass also false when the
// pass ends at that item.
template <bool COLLECT>
__device__ __forceinline__ bool wait_desc(uint64_t *bar, uint32_t parity, volatile int *abort_flag, int64_t item)
{
    if constexpr (COLLECT) {
        const uint64_t t0 = now_ns();
        while (!mbar_try(bar, parity)) {
            if (now_ns() - t0 > g_wait_limit_ns) *abort_flag = 1;
            if (*abort_flag || g_end_item == (uint32_t)item) return false;
        }
        return true;
    } else {
        return mbar_wait(bar, parity, abort_flag);
    }
}

// The same, inline and counting its cycles, for the producers' stage loops (a
// call there costs more than the wait itself).
__device__ __forceinline__ bool wait_here(uint64_t *bar, uint32_t parity, volatile int *abort_flag, long long &acc)
{
    if (mbar_test(bar, parity)) return true;
    const long long c0 = clock64();
    const uint64_t n0 = now_ns();
    bool ok = true;
    while (!mbar_try(bar, parity)) {
        if (now_ns() - n0 > g_wait_limit_ns) *abort_flag = 1;
        if (*abort_flag) {
            ok = false;
            break;
        }
    }
    acc += clock64() - c0;
    return ok;
}

// The same for a whole warp in step: the lanes' tests are voted on, so that
// they go on, or give up, together.
__device__ __forceinline__ bool wait_together(uint64_t *bar, uint32_t parity, volatile int *abort_flag, long long &acc)
{
    if (__all_sync(0xffffffffu, mbar_test(bar, parity))) return true;
    const long long c0 = clock64();
    const uint64_t n0 = now_ns();
    bool ok = true;
    while (!__all_sync(0xffffffffu, mbar_try(bar, parity))) {
        if (now_ns() - n0 > g_wait_limit_ns) *abort_flag = 1;
        if (__any_sync(0xffffffffu, *abort_flag)) {
            ok = false;
            break;
        }
    }
    acc += clock64() - c0;
    return ok;
}

// Hot-path wait: one inline non-blocking test; the bounded out-of-line wait
// (and the cycle accounting of the trace) only when the phase is not
// complete yet, so the trace counts every cycle spent waiting.
__device__ __forceinline__ bool wait_fast(uint64_t *bar, uint32_t parity, volatile int *abort_flag, long long &acc)
{
    if (mbar_test(bar, parity)) return true;
    const long long t0 = clock64();
    const bool ok = mbar_wait(bar, parity, abort_flag);
    acc += clock64() - t0;
    return ok;
}

// The issuing warp's wait, inline: a function call in its loop would keep
// every value that lives across it out of the uniform registers the MMAs take
// their operands from.  In a collecting pass also false when it ends at `item`.
template <bool COLLECT>
__device__ __forceinline__ bool wait_inline(uint64_t *bar, uint32_t parity, volatile int *abort_flag, long long &acc,
                                            uint32_t item)
{
    const long long t0 = clock64();
    const uint64_t n0 = now_ns();
    bool ok = true;
    while (!__all_sync(0xffffffffu, mbar_try(bar, parity))) {
        if (now_ns() - n0 > g_wait_limit_ns) *abort_flag = 1;
        if (__any_sync(0xffffffffu, *abort_flag || (COLLECT && g_end_item == item))) {
            ok = false;
            break;
        }
    }
    acc += clock64() - t0;
    return ok;
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
        "[%4];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// Instruction descriptor of kind::mxf4 with F32 accumulation: E2M1 operands,
// both K-major, UE8M0 scales, M = 128 and n columns; bits 4-5 select B's
// pair of scale bytes (0: bytes 0-1, the controls' scale; 2: bytes 2-3, the
// cases').
__host__ __device__ constexpr uint32_t make_idesc(uint32_t n)
{
    return (1u << 7) | (1u << 10) | ((n >> 3) << 17) | (1u << 23) | (1u << 27);
}
constexpr uint32_t kIdescCase = 2u << 4;

// The MMA executed by a whole warp in step; only the elected lane (`leader`
// nonzero) issues it.
__device__ __forceinline__ void mma_f4_warp(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t accumulate,
                                            uint32_t leader, uint32_t idesc, uint32_t sfa, uint32_t sfb)
{
    asm volatile(
        "{\n .reg .pred p, e;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 e, %5, 0;\n"
        " @e tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%6], [%7], p;\n}\n" ::"r"(
            d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(leader), "r"(sfa), "r"(sfb));
}

// 16 tensor-memory columns of this warp's lane quadrant set to v
__device__ __forceinline__ void tmem_fill16(uint32_t taddr, uint32_t v)
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(taddr),
        "r"(v)
        : "memory");
}

__device__ __forceinline__ void mma_commit_warp(uint64_t *bar, uint32_t leader)
{
    asm volatile(
        "{\n .reg .pred e;\n setp.ne.b32 e, %1, 0;\n"
        " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(smem_u32(bar)),
        "r"(leader)
        : "memory");
}

__device__ __forceinline__ uint32_t elect_one()
{
    uint32_t pred;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(pred));
    return pred;
}

__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// lane 0's value in every lane, known to be warp-uniform
__device__ __forceinline__ uint32_t uniform(uint32_t x) { return __shfl_sync(0xffffffffu, x, 0); }

template <int NT>
__device__ __forceinline__ void epi_bar() { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); }

// ------------------------------------------------------------ enumeration --
// Prefixes of order k are the (k-1)-subsets whose last SNP c is <= n-2, in
// panel order: panel c holds the subsets ending in c whose first SNP lies in
// [s1_lo, s1_hi], their first k-2 SNPs in lexicographic order.  pcum[c]
// counts the prefixes of panels < c; q is a prefix's index in this order.
struct PrefixIter {
    int32_t a[kMaxOrderTc];    // first k-2 SNPs (ascending)
    int32_t c;                 // last prefix SNP (panel)
    uint64_t q;                // index in panel order
};

// Subsets of [0, c) of size m with first element >= x: C(c - x, m) (0 when
// c - x < m); for m = 0 the single empty subset, which has no first element
// and counts for every x.
__device__ __forceinline__ uint64_t subsets_from(const DevData &d, int64_t c, int64_t x, int m)
{
    if (m == 0) return 1;
    return c - x >= m ? binom_at(d.binom, d.n, c - x, m) : 0;
}

// Largest x in [lo, hi] for which pred holds (true up to there, pred(lo)
// taken as true), by the whole warp: 32 probes at a time, since each probe
// waits for a load from L2.
template <class F>
__device__ __forceinline__ int64_t warp_last(int64_t lo, int64_t hi, F pred)
{
    const int lane = threadIdx.x & 31;
    while (lo < hi) {
        const int64_t step = (hi - lo + 31) / 32;
        const int64_t c = min(lo + (lane + 1) * step, hi);
        const int n = __popc(__ballot_sync(0xffffffffu, pred(c)));   // the first n probes hold
        hi = n < 32 ? min(lo + (n + 1) * step - 1, hi) : hi;
        lo = min(lo + n * step, hi);
    }
    return lo;
}

// Lexicographic unranking of r among the m-subsets of [0, c) (m <= 3), by the
// whole warp.
__device__ inline void lex_unrank_below(const DevData &d, int64_t c, int m, uint64_t r, int32_t *out)
{
    int64_t start = 0;
    for (int i = 0; i < m; i++) {
        const int rem = m - i;
        const uint64_t all = binom_at(d.binom, d.n, c - start, rem);
        // largest x in [start, c - rem] with fewer than r + 1 subsets whose
        // element i is below x
        const int64_t lo = warp_last(start, c - rem, [&](int64_t x) {
            return all - binom_at(d.binom, d.n, c - x, rem) <= r;
        });
        r -= all - binom_at(d.binom, d.n, c - lo, rem);
        out[i] = (int32_t)lo;
        start = lo + 1;
    }
}

__device__ inline void prefix_unrank(const DsParams &P, int k, uint64_t q, PrefixIter &it)
{
    const DevData &d = P.d;
    // panel: largest c with pcum[c] <= q (a non-empty panel)
    const int64_t lo = warp_last(0, d.n - 2, [&](int64_t x) { return P.pcum[x] <= q; });
    it.c = (int32_t)lo;
    it.q = q;
    const int m2 = k - 2;
    // index within the panel: the subsets whose first SNP is below s1_lo come first
    const uint64_t skip = subsets_from(d, lo, 0, m2) - subsets_from(d, lo, P.s1_lo, m2);
    lex_unrank_below(d, lo, m2, (m2 ? skip : 0) + (q - P.pcum[lo]), it.a);
}

__device__ inline void prefix_next(const DsParams &P, int k, PrefixIter &it)
{
    it.q++;
    const int m2 = k - 2;
    // lexicographic successor within the panel: the last position that can
    // still grow; the first SNP must stay <= s1_hi
    int i = m2 - 1;
    while (i >= 0 && it.a[i] >= it.c - m2 + i) i--;
    if (i > 0 || (i == 0 && it.a[0] + 1 <= P.s1_hi)) {
        it.a[i]++;
        for (int t = i + 1; t < m2; t++) it.a[t] = it.a[t - 1] + 1;
        return;
    }
    // next panel (every panel after a non-empty one is non-empty): its first
    // prefix starts at s1_lo
    it.c++;
    for (int t = 0; t < m2; t++) it.a[t] = P.s1_lo + t;
}

// first (even) last SNP of panel c's N tiles, and their number
__host__ __device__ __forceinline__ int64_t panel_j0(int64_t c) { return (c + 1) & ~(int64_t)1; }
__host__ __device__ __forceinline__ int64_t panel_ntiles(int64_t n, int64_t c, int kj)
{
    return (n - panel_j0(c) + kj - 1) / kj;
}

// ------------------------------------------------------------------ pairs --
// Pair tiles (orders 4-5, whole searches): the last TWO SNPs move to the B
// side.  A tile's rows are (k-2)-prefixes (9 or 27 rows each, 12 or 4 of them)
// and its columns the four joint genotypes (g1, g2 in {0, 1}) of a SNP j1 with
// 60 (or 40) SNPs j2 > j1, an operand built once per search.  A combination
// then takes 128 / 12 x 4 multiply-adds per individual instead of 128 / 4 x 2
// (order 4; order 5: 128 instead of 256), tiles keep all their columns (the
// pairs (j1, j2) of one j1 are many more than the SNPs after a prefix), and
// an A tile serves twice the combinations, which the producers need most.
// The remaining cells of a row follow from its counts with one of the two
// SNPs (the single counts: the same product one order lower, stored by a first
// pass as raw accumulators) and its total:
//     n[g1][2] = n[g1][*] - n[g1][0] - n[g1][1], n[2][g2] likewise, and
//     n[2][2] = n[*][*] - n[0][*] - n[1][*] - n[2][0] - n[2][1].
// Singles table: panel c holds its prefixes in order, each
// single_groups(n, c) groups of two SNPs (from the even panel_j0(c)), a group
// the prefix's rows side by side, a row one float4 per accumulator: genotype 0
// of both SNPs, genotype 1 of both.
__host__ __device__ __forceinline__ int64_t single_groups(int64_t n, int64_t c) { return (n - panel_j0(c) + 1) / 2; }
// operand rows of j1's pairs: 8 per group of two SNPs from the even panel_j0(j1)
__host__ __device__ __forceinline__ int64_t pair_rows(int64_t n, int64_t j1) { return 8 * single_groups(n, j1); }

// -------------------------------------------------------------- epilogue --
// the integer value of an accumulator (below 2^23)
__device__ __forceinline__ uint32_t f2u_exact(float v) { return __float_as_uint(v + 8388608.0f) & 0x7FFFFFu; }

// two floats handled by one instruction (f32x2)
struct F2 {
    uint64_t v;
};
__device__ __forceinline__ F2 f2_pack(float lo, float hi)
{
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_unpack(F2 a, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v));
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c)
{
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b)
{
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b)
{
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 f2_abs(F2 a)
{
    float x, y;
    f2_unpack(a, x, y);
    return f2_pack(fabsf(x), fabsf(y));
}
// 1 / (s + tiny), approximate; finite for s = 0 (cells of no individuals,
// whose terms then are 0)
__device__ __forceinline__ F2 f2_rcp(F2 s, F2 tiny)
{
    float x, y;
    f2_unpack(f2_add(s, tiny), x, y);
    asm("rcp.approx.ftz.f32 %0, %0;" : "+f"(x));
    asm("rcp.approx.ftz.f32 %0, %0;" : "+f"(y));
    return f2_pack(x, y);
}

// The screen: an upper bound of m MI from the cells' totals and case counts.
//
// With s = a + b individuals in a cell, a of them cases, pi = m1 / m and
// x = a / s - pi, m MI = sum over cells of s f(x), f(x) the divergence of a
// Bernoulli(pi + x) from a Bernoulli(pi).  f(x) = c2 x^2 + c3 x^3 + g(x) x^4
// with c2 = 1 / (2 pi (1 - pi)), c3 = (2 pi - 1) / (6 pi^2 (1 - pi)^2) and
// g convex (the fourth derivative of f, 2 / p^3 + 2 / (1 - p)^3, is convex),
// so g lies below its chords: from x = -pi to 0 and from 0 to 1 - pi, whose
// end values have closed forms.  The bound c2 x^2 + c3 x^3 + (c4 + c5a x +
// c5b |x|) x^4 takes one reciprocal per cell and packed multiply-adds where
// exact logarithms take three; on Hardy-Weinberg tables of 1000-16000
// individuals its excess over 2 m MI averages 0.2 (order 3, pi = 0.5) to 1.5
// (order 4, pi = 0.2) while pi lies in [0.2, 0.8], and 2 to 25 at pi = 0.1,
// so outside that interval the logarithms screen.
// Per cell it gets e = 2^(p-1) (a - pi s) and s; the constants absorb the
// power of two.
struct ScreenConst {
    F2 c2, c3, c4, c5a, c5b, tiny;
};
__device__ __forceinline__ F2 cell_bound(F2 e, F2 s, const ScreenConst &c, F2 acc)
{
    const F2 x = f2_mul(e, f2_rcp(s, c.tiny));
    F2 t = f2_fma(c.c5a, x, c.c4);
    t = f2_fma(c.c5b, f2_abs(x), t);
    t = f2_fma(x, t, c.c3);
    t = f2_fma(x, t, c.c2);
    return f2_fma(f2_mul(e, x), t, acc);
}

// t(x) = x log2 x of a count (0 for x = 0)
__device__ __forceinline__ float tlog(float x) { return x * lg2n(fmaxf(x, 1.0f)); }

// t(a) + t(b) - t(a + b) of a cell's counts
__device__ __forceinline__ float cell_log(float a, float b) { return tlog(a) + tlog(b) - tlog(a + b); }

// Compensated sums of the precise scores' terms, over the warp and over a
// prefix's PR row lanes (with plain sums order 2 was 1.5e-7 off 64 bits, and
// 3.6e-8 on the popcount path, whose sum is compensated).
__device__ __forceinline__ float warp_sum(SumF32 v)
{
#pragma unroll
    for (int off = 16; off; off >>= 1) {
        const float s = __shfl_xor_sync(0xffffffffu, v.s, off), c = __shfl_xor_sync(0xffffffffu, v.c, off);
        v.add(s);
        v.c += c;
    }
    return v.value();
}

template <int PR>
__device__ __forceinline__ float seg_sum(SumF32 v, int pos)
{
#pragma unroll
    for (int off = 1; off < PR; off <<= 1) {
        const float s = __shfl_down_sync(0xffffffffu, v.s, off), c = __shfl_down_sync(0xffffffffu, v.c, off);
        if ((pos & (2 * off - 1)) == 0 && pos + off < PR) {
            v.add(s);
            v.c += c;
        }
    }
    return v.value();
}

template <int NT>
__device__ inline void sort_cands_epi(float *sc, uint64_t *rk, int p2, int tid)
{
    for (int kk = 2; kk <= p2; kk <<= 1) {
        for (int jj = kk >> 1; jj > 0; jj >>= 1) {
            for (int i = tid; i < p2; i += NT) {
                const int ixj = i ^ jj;
                if (ixj > i) {
                    const bool up = (i & kk) == 0;
                    const bool sw = up ? cand_better(sc[ixj], rk[ixj], sc[i], rk[i])
                                       : cand_better(sc[i], rk[i], sc[ixj], rk[ixj]);
                    if (sw) {
                        float ts = sc[i]; sc[i] = sc[ixj]; sc[ixj] = ts;
                        uint64_t tr = rk[i]; rk[i] = rk[ixj]; rk[ixj] = tr;
                    }
                }
            }
            epi_bar<NT>();
        }
    }
}

struct EpiState {
    int32_t list_len, nbuf, stop, any;
    float thr;                 // the CTA's own pool threshold
    float next_thr;            // the larger of it and the other CTAs'
    int32_t seen;              // kept combinations at the last look at the histogram
};

// Histogram of the precise scores of every combination any CTA has kept (each
// is kept once): the bins are the scores' leading 16 bits (relative width
// 2^-7) from 2^-16 up.  Its top_n-th best, lowered by four times the score's
// error bound, is a threshold for all CTAs: after the first columns of every
// CTA it comes from 152 times as many combinations as the CTA's own list, so
// few of the later ones are scored precisely (searches with the thresholds of
// the CTAs' own lists and with this: order 2, 6007 x 5003: 2.27 and 0.52 ms;
// order 3, 300 x 2500: 0.69 and 0.38 ms).
constexpr uint32_t kHistFirst = 0x3780u;   // 2^-16 >> 16
__device__ __forceinline__ int hist_bin(float score)
{
    const int b = (int)(__float_as_uint(score) >> 16) - (int)kHistFirst + 1;
    return b < 0 ? 0 : (b >= kTcHistBins ? kTcHistBins - 1 : b);
}
// the threshold the histogram gives, or -1 (all threads of the epilogue; tmp:
// NT / 32 + 2 words of shared memory)
template <int NT>
__device__ inline float hist_threshold(const uint32_t *hist, int top_n, uint32_t *tmp, int tid)
{
    constexpr int kPer = kTcHistBins / NT;
    static_assert(kPer * NT == kTcHistBins && kPer % 4 == 0, "whole vectors per thread");
    const int lane = tid & 31, warp = tid >> 5;
    const int top = kTcHistBins - kPer * (tid + 1);     // this thread's lowest bin (thread 0 has the highest)
    uint32_t c[kPer], sum = 0;
#pragma unroll
    for (int q = 0; q < kPer; q += 4) {
        const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(hist + top + q));
        c[q] = v.x; c[q + 1] = v.y; c[q + 2] = v.z; c[q + 3] = v.w;
        sum += v.x + v.y + v.z + v.w;
    }
    uint32_t inc = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t o = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += o;
    }
    if (tid == 0) tmp[NT / 32] = 0;
    if (lane == 31) tmp[warp] = inc;
    epi_bar<NT>();
    uint32_t before = inc - sum;
    for (int w = 0; w < warp; w++) before += tmp[w];
    const uint32_t need = (uint32_t)top_n;
    if (before < need && before + sum >= need) {
        int b = kPer;
        while (before < need) before += c[--b];
        b += top;
        tmp[NT / 32] = b > 0 ? (uint32_t)(b - 1 + (int)kHistFirst) << 16 : 0u;
    }
    epi_bar<NT>();
    const float t = __uint_as_float(tmp[NT / 32]);
    return t > 0.0f ? t : -1.0f;
}

template <int NT>
__device__ inline void epi_flush(EpiState &S, float *sc, uint64_t *rk, int pool, const DsParams &DS, int tid)
{
    epi_bar<NT>();
    const int live = S.list_len + S.nbuf;
    const int p2 = next_pow2(live < 2 ? 2 : live);
    for (int i = live + tid; i < p2; i += NT) { sc[i] = -1.0f; rk[i] = ~0ull; }
    epi_bar<NT>();
    sort_cands_epi<NT>(sc, rk, p2, tid);
    if (tid == 0) {
        S.list_len = live < pool ? live : pool;
        S.nbuf = 0;
        // at least top_n combinations score >= the top_n-th best: lowered by
        // four times the score's error bound it is safe for the top N and
        // still clears the final margin check
        float t = S.list_len == pool ? sc[pool - 1] : -1.0f;
        if (DS.top_n > 0 && live >= DS.top_n) t = fmaxf(t, sc[DS.top_n - 1] * DS.thr_mul);
        if (t > S.thr) {
            S.thr = t;
            atomicMax(DS.global_thr, __float_as_uint(t));
        }
    }
    epi_bar<NT>();
}

// ---------------------------------------------------------------- kernel --
// Precise single-precision terms of one tile row's three cells (the rare
// candidate path, kept out of line).
__device__ __noinline__ SumF32 row_terms_precise(uint32_t a0, uint32_t b0, uint32_t a1, uint32_t b1, uint32_t a2,
                                                 uint32_t b2, const MiConstF32 mc)
{
    SumF32 v;
    v.add(cell_terms_f32(a0, b0, mc));
    v.add(cell_terms_f32(a1, b1, mc));
    v.add(cell_terms_f32(a2, b2, mc));
    return v;
}

#define TMEM_LD16(taddr, r)                                                                                      \
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, " \
                 "[%16];"                                                                                        \
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), \
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),       \
                   "=r"(r[15])                                                                                   \
                 : "r"(taddr))

// Row values of a chunk: raw accumulators of 8 last SNPs -> the row's part of
// the screen for each, vrow[jj].  Columns 4 h + {0, 1} hold genotype 0 of SNPs
// 2 h and 2 h + 1, columns 4 h + {2, 3} genotype 1.
template <bool C>
struct RowScreen {
    // packed constants; q = 2^(p-1) (1 with separate classes): cases are held
    // times q
    F2 half, neg2, m23, neg_m23, neg1, inv_q, neg_pi;
    ScreenConst sc;
    F2 S, CT;                  // the row's totals: individuals and cases
    uint32_t hi_mask;
    float inv_q1;

    __device__ __forceinline__ void set_row(float cases, float ctrls, float q)
    {
        S = f2_pack(cases + ctrls, cases + ctrls);
        CT = f2_pack(cases * q, cases * q);
    }
    // the two classes of a column pair: individuals s and cases ca.  An
    // accumulator holds v = ctrl + case 2^p < 2^24; v / 2 + 2^23 has the bits
    // of v / 2 (rounded) in its mantissa, and those from bit p - 1 on are the
    // cases (the rounding cannot carry into them: ctrl < 2^p - 1).  (Two
    // products rounded down instead, without the mask: 63.8 instead of 57.7 ms
    // at order 3, 2000 x 4000.)
    __device__ __forceinline__ void split(uint32_t x0, uint32_t x1, F2 &s, F2 &ca) const
    {
        const F2 v = f2_pack(__uint_as_float(x0), __uint_as_float(x1));
        float y0, y1;
        f2_unpack(f2_fma(v, half, m23), y0, y1);
        ca = f2_add(f2_pack(__uint_as_float(__float_as_uint(y0) & hi_mask),
                            __uint_as_float(__float_as_uint(y1) & hi_mask)), neg_m23);
        s = f2_fma(ca, inv_q, f2_fma(ca, neg2, v));
    }
    __device__ __forceinline__ void pair(const uint32_t *cs, const uint32_t *cn, int h, F2 &s0, F2 &s1, F2 &a0,
                                         F2 &a1) const
    {
        if constexpr (C) {
            split(cs[4 * h], cs[4 * h + 1], s0, a0);
            split(cs[4 * h + 2], cs[4 * h + 3], s1, a1);
        } else {
            a0 = f2_pack(__uint_as_float(cs[4 * h]), __uint_as_float(cs[4 * h + 1]));
            a1 = f2_pack(__uint_as_float(cs[4 * h + 2]), __uint_as_float(cs[4 * h + 3]));
            s0 = f2_add(a0, f2_pack(__uint_as_float(cn[4 * h]), __uint_as_float(cn[4 * h + 1])));
            s1 = f2_add(a1, f2_pack(__uint_as_float(cn[4 * h + 2]), __uint_as_float(cn[4 * h + 3])));
        }
    }
    __device__ __forceinline__ void bound(const uint32_t *cs, const uint32_t *cn, float *vrow) const
    {
#pragma unroll
        for (int h = 0; h < 4; h++) {
            F2 s0, s1, a0, a1;
            pair(cs, cn, h, s0, s1, a0, a1);
            const F2 e0 = f2_fma(s0, neg_pi, a0), e1 = f2_fma(s1, neg_pi, a1);
            // genotype 2 by subtraction (exact), so that an empty cell has
            // e = 0 whatever pi
            const F2 s2 = f2_fma(s1, neg1, f2_fma(s0, neg1, S));
            const F2 e2 = f2_fma(s2, neg_pi, f2_fma(a1, neg1, f2_fma(a0, neg1, CT)));
            F2 acc;
            acc.v = 0;
            acc = cell_bound(e0, s0, sc, acc);
            acc = cell_bound(e1, s1, sc, acc);
            acc = cell_bound(e2, s2, sc, acc);
            f2_unpack(acc, vrow[2 * h], vrow[2 * h + 1]);
        }
    }
    // counts of column pair h's cells: a = cases, b = controls by genotype,
    // of SNP 2 h + odd
    __device__ __forceinline__ void counts(const uint32_t *cs, const uint32_t *cn, int h, bool odd, float *a,
                                           float *b) const
    {
        F2 s0, s1, a0, a1;
        pair(cs, cn, h, s0, s1, a0, a1);
        const F2 s2 = f2_fma(s1, neg1, f2_fma(s0, neg1, S));
        const F2 a2 = f2_fma(a1, neg1, f2_fma(a0, neg1, CT));
        const F2 ss[3] = {s0, s1, s2}, aa[3] = {a0, a1, a2};
#pragma unroll
        for (int g = 0; g < 3; g++) {
            float x, y, u, v;
            f2_unpack(aa[g], x, y);
            f2_unpack(ss[g], u, v);
            a[g] = (odd ? y : x) * inv_q1;
            b[g] = (odd ? v : u) - a[g];
        }
    }
    // --- pair tiles: U0, U1 this row's counts with j1's genotypes 0 and 1,
    // V its count with genotype 2 (individuals .s, cases .c)
    struct Cnt {
        F2 s, c;
    };
    Cnt U0, U1, V;
    __device__ __forceinline__ Cnt raw2(uint32_t x0, uint32_t x1, uint32_t y0, uint32_t y1) const
    {
        Cnt r;
        if constexpr (C) {
            split(x0, x1, r.s, r.c);
        } else {
            r.c = f2_pack(__uint_as_float(x0), __uint_as_float(x1));
            r.s = f2_add(r.c, f2_pack(__uint_as_float(y0), __uint_as_float(y1)));
        }
        return r;
    }
    __device__ __forceinline__ Cnt minus2(Cnt a, Cnt b, Cnt d) const
    {
        return Cnt{f2_fma(d.s, neg1, f2_fma(b.s, neg1, a.s)), f2_fma(d.c, neg1, f2_fma(b.c, neg1, a.c))};
    }
    // the nine cells (3 g1 + g2) of two SNPs j2: accumulator columns in pairs
    // (00, 01, 10, 11), s0 / s1 the single counts with them
    __device__ __forceinline__ void nine(const uint32_t *cs, const uint32_t *cn, const float4 &a, const float4 &b,
                                         Cnt *n) const
    {
        n[0] = raw2(cs[0], cs[1], cn[C ? 0 : 0], cn[C ? 0 : 1]);
        n[1] = raw2(cs[2], cs[3], cn[C ? 0 : 2], cn[C ? 0 : 3]);
        n[3] = raw2(cs[4], cs[5], cn[C ? 0 : 4], cn[C ? 0 : 5]);
        n[4] = raw2(cs[6], cs[7], cn[C ? 0 : 6], cn[C ? 0 : 7]);
        const Cnt t0 = raw2(__float_as_uint(a.x), __float_as_uint(a.y), __float_as_uint(b.x), __float_as_uint(b.y));
        const Cnt t1 = raw2(__float_as_uint(a.z), __float_as_uint(a.w), __float_as_uint(b.z), __float_as_uint(b.w));
        n[2] = minus2(U0, n[0], n[1]);
        n[5] = minus2(U1, n[3], n[4]);
        n[6] = minus2(t0, n[0], n[3]);
        n[7] = minus2(t1, n[1], n[4]);
        n[8] = minus2(V, n[6], n[7]);
    }
    __device__ __forceinline__ void pair_bound(const uint32_t *cs, const uint32_t *cn, const float4 &a, const float4 &b,
                                               float &v0, float &v1) const
    {
        Cnt n[9];
        nine(cs, cn, a, b, n);
        F2 acc;
        acc.v = 0;
#pragma unroll
        for (int x = 0; x < 9; x++) acc = cell_bound(f2_fma(n[x].s, neg_pi, n[x].c), n[x].s, sc, acc);
        f2_unpack(acc, v0, v1);
    }
    __device__ __forceinline__ void pair_logs(const uint32_t *cs, const uint32_t *cn, const float4 &a, const float4 &b,
                                              float &v0, float &v1) const
    {
        Cnt n[9];
        nine(cs, cn, a, b, n);
        v0 = v1 = 0.0f;
#pragma unroll
        for (int x = 0; x < 9; x++) {
            float c0, c1, s0, s1;
            f2_unpack(n[x].c, c0, c1);
            f2_unpack(n[x].s, s0, s1);
            c0 *= inv_q1;
            c1 *= inv_q1;
            v0 += cell_log(c0, s0 - c0);
            v1 += cell_log(c1, s1 - c1);
        }
    }
    // this item's j1: its group's float4s and whether it is the odd SNP
    __device__ __forceinline__ void set_first(const float4 &a, const float4 &b, bool odd)
    {
        const uint32_t x0 = __float_as_uint(odd ? a.y : a.x), x1 = __float_as_uint(odd ? a.w : a.z);
        const uint32_t y0 = __float_as_uint(odd ? b.y : b.x), y1 = __float_as_uint(odd ? b.w : b.z);
        U0 = raw2(x0, x0, y0, y0);
        U1 = raw2(x1, x1, y1, y1);
        const Cnt all{S, CT};
        V = minus2(all, U0, U1);
    }
    __device__ __forceinline__ void logs(const uint32_t *cs, const uint32_t *cn, float *vrow) const
    {
#pragma unroll
        for (int jj = 0; jj < 8; jj++) {
            float a[3], b[3];
            counts(cs, cn, jj >> 1, jj & 1, a, b);
            vrow[jj] = cell_log(a[0], b[0]) + cell_log(a[1], b[1]) + cell_log(a[2], b[2]);
        }
    }
};

// One row's nine cells (3 g1 + g2) of a pair, as counts (the rare paths,
// kept out of line): raw accumulators of the joint genotypes 00, 01, 10, 11
// and of j2's single counts (x: the only or the case accumulator, y: the
// control accumulator), counts of the row with j1's genotypes 0 and 1 and
// with genotype 2 (c cases, s individuals), 2^-p and 2^p.
struct PairRow {
    float x[6], y[6];
    float c0, s0, c1, s1, c2, s2;
    float kinv, p2;
};
template <bool C>
__device__ __noinline__ void pair_cells(const PairRow &r, uint32_t *ca, uint32_t *co)
{
    float c[6], t[6];                        // cases, controls
#pragma unroll
    for (int i = 0; i < 6; i++) {
        c[i] = C ? floorf(r.x[i] * r.kinv) : r.x[i];
        t[i] = C ? fmaf(c[i], -r.p2, r.x[i]) : r.y[i];
    }
    const float t0 = r.s0 - r.c0, t1 = r.s1 - r.c1, t2 = r.s2 - r.c2;
    const float cc[9] = {c[0], c[1], r.c0 - c[0] - c[1], c[2], c[3], r.c1 - c[2] - c[3],
                         c[4] - c[0] - c[2], c[5] - c[1] - c[3],
                         r.c2 - (c[4] - c[0] - c[2]) - (c[5] - c[1] - c[3])};
    const float tt[9] = {t[0], t[1], t0 - t[0] - t[1], t[2], t[3], t1 - t[2] - t[3],
                         t[4] - t[0] - t[2], t[5] - t[1] - t[3],
                         t2 - (t[4] - t[0] - t[2]) - (t[5] - t[1] - t[3])};
#pragma unroll
    for (int i = 0; i < 9; i++) {
        ca[i] = f2u_exact(cc[i]);
        co[i] = f2u_exact(tt[i]);
    }
}

// Lexicographic rank of a combination from the sum over its SNPs s_t of
// C(n - 1 - s_t, K - t): total - 1 - sum.
template <int km1>
__device__ __forceinline__ uint64_t prefix_rank_sum(const DevData &d, const int32_t *psnp, int k = km1 + 1)
{
    uint64_t s = 0;
#pragma unroll
    for (int tt = 0; tt < km1; tt++) s += binom_at(d.binom, d.n, d.n - 1 - psnp[tt], k - tt);
    return s;
}

// Last SNPs [jlo, jhi) of a prefix inside the searched rank range: the
// combination (prefix, j) has rank base + j.  Only prefixes whose first SNP
// is the range's first or last can be cut.
template <int km1>
__device__ __forceinline__ void last_snp_range(const DsParams &DS, const DevData &d, const int32_t *psnp, int32_t &jlo,
                                               int32_t &jhi)
{
    jlo = psnp[km1 - 1] + 1;
    jhi = (int32_t)d.n;
    if (DS.clip && (psnp[0] == DS.s1_lo || psnp[0] == DS.s1_hi)) {
        const int64_t base = (int64_t)DS.total - (int64_t)prefix_rank_sum<km1>(d, psnp) - d.n;
        int64_t lo64 = (int64_t)DS.rank_begin - base, hi64 = (int64_t)DS.rank_end - base;
        lo64 = lo64 < (int64_t)jlo ? (int64_t)jlo : (lo64 > d.n ? d.n : lo64);
        hi64 = hi64 > d.n ? d.n : (hi64 < lo64 ? lo64 : hi64);
        jlo = (int32_t)lo64;
        jhi = (int32_t)hi64;
    }
}

#define TMEM_LD8(taddr, r)                                                                                       \
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"                        \
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) \
                 : "r"(taddr))

// COLLECT: every combination that scores at least a threshold instead of the
// best (a kernel of its own: its end in mid-pass, as branches of the search's
// kernel, cost that 0.7 % at order 3, 2000 x 4000, and 1.2 % at order 5,
// 93 x 2001)
template <int K, bool C, bool PAIR, bool COLLECT>
__global__ void __launch_bounds__(Roles::Threads, 1) tc_search_kernel(const __grid_constant__ CUtensorMap tmap_b,
                                                                const Params P)
{
    using S = Shape<C>;
    using R = Roles;
    constexpr int kStages = S::Stages;
    constexpr int kJ = PAIR ? S::N / 4 : S::J;      // last SNPs per N tile
    constexpr int kColsPerSnp = S::N / kJ;
    constexpr int kBBytes = S::BBytes;
    constexpr int kEpiWarps = R::EpiWarps, kProdWarps = R::ProdWarps, kEpiThreads = R::EpiThreads;
    constexpr int kGroups = R::ProdGroups, kCG = R::ColGroups;
    // epilogue: the kQC chunks of 8 last SNPs of a lane quadrant go round-
    // robin to its kCG warps, kIters chunks each (the last may be empty)
    // (pair tiles: chunks of 4 last SNPs, 16 columns; of 2 with separate
    // classes, whose two accumulators and singles would spill)
    constexpr int kCS = PAIR ? (C ? 4 : 2) : 8;
    constexpr int kChunkCols = kCS * kColsPerSnp, kH = kCS / 2;   // columns and groups of two SNPs
    constexpr int kQC = kJ / kCS;
    constexpr int kIters = (kQC + kCG - 1) / kCG;
    constexpr int km1 = PAIR ? K - 2 : K - 1;       // prefix SNPs
    constexpr int kPR = km1 == 1 ? 3 : (km1 == 2 ? 9 : (km1 == 3 ? 27 : 81));
    // order 5: one prefix per tile, its 81 rows over lane quadrants 0-2 (the
    // epilogue sums a combination across warps through shared memory)
    constexpr bool kWide = kPR > 32;
    constexpr int kPPW = kWide ? 0 : 32 / kPR;
    constexpr int kPPT = kWide ? 1 : 4 * kPPW;
    constexpr int kWarpTma = kEpiWarps + kProdWarps;
    constexpr int kWarpMma = kWarpTma + 1;
    // (prefix, last SNP) pairs per warp and chunk; orders 4-5: 8 columns by 4
    // lane parts of the rows
    constexpr int kPairs = (kPPW > 1 ? kPPW : 1) * kCS;
    constexpr int kPairIters = (kPairs + 31) / 32;

    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    unsigned char *stages_a = smem;
    unsigned char *stages_b = smem + kStages * kTileBytes;
    // per epilogue warp, the row values of 8 last SNPs [lane][8] (transposed
    // so that one lane sums one prefix's rows for one last SNP)
    float *wsum = reinterpret_cast<float *>(stages_b + kStages * kBBytes);
    uint32_t *tot = reinterpret_cast<uint32_t *>(wsum + kEpiWarps * 256);   // [2][128][kGroups][2 classes]
    Desc *desc = reinterpret_cast<Desc *>(tot + 2 * 128 * kGroups * 2);
    // (or, when every score is wanted, the n ln n table: nothing is kept then)
    long long *tlog = reinterpret_cast<long long *>(desc + kDescDepth);
    float *sc;
    uint64_t *rk;
    if (P.cand_score_g) {
        sc = P.cand_score_g + (size_t)blockIdx.x * P.cand_p2;
        rk = P.cand_rank_g + (size_t)blockIdx.x * P.cand_p2;
    } else {
        rk = reinterpret_cast<uint64_t *>(desc + kDescDepth);
        sc = reinterpret_cast<float *>(rk + P.cand_p2);
    }

    // full_ab[s]: one group's producer warps and the TMA thread (with its
    // bytes) have filled stage s of both operands; empty_ab[s]: the MMAs that
    // read it are done (one commit per stage)
    __shared__ __align__(8) uint64_t full_ab[kStages], empty_ab[kStages];
    __shared__ __align__(8) uint64_t acc_full[2], acc_empty[S::Accs], tot_full[2], tot_empty[2];
    __shared__ __align__(8) uint64_t desc_full[kDescDepth], desc_empty[kDescDepth], drain_bar;
    __shared__ uint32_t tmem_base_sh;
    // the MMA instruction descriptor of each item (its column count), written
    // with the item's descriptor
    __shared__ uint32_t item_idesc[kDescDepth];
    __shared__ volatile int abort_flag;
    __shared__ volatile int over_flag;               // COLLECT: more found than the caller's array holds
    __shared__ EpiState ES;
    __shared__ uint32_t hist_tmp[kEpiWarps + 1];
    // order 5: per-quadrant sums of the item's last SNPs, and their flags
    __shared__ float wred[kWide ? 4 : 1][kWide ? kJ : 1], wpre[kWide ? 4 : 1][kWide ? kJ : 1];
    __shared__ __align__(8) unsigned char wflag[kWide ? kJ : 1];

    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const DsParams &DS = P.many ? P.many[P.cta_ds[blockIdx.x]] : P.one;
    const DevData d = DS.d;
    const CUtensorMap *tmap = DS.tmap ? DS.tmap : &tmap_b;

    const uint64_t cb = blockIdx.x - (uint64_t)DS.cta_begin, cn_ = (uint64_t)DS.cta_count;
    // Items get cheaper along the panels (fewer last SNPs), so a CTA takes
    // several ranges spread over all of them (up to 16, of 8 items or more,
    // since finding a range's first item takes microseconds): segment q of
    // the dataset's segments x cn goes to CTA q % cn.
    const int segments = (int)max((uint64_t)1, min((uint64_t)16, DS.n_items / (cn_ * 8)));
    auto segment_at = [&](uint64_t q) -> uint64_t {
        return (uint64_t)(((unsigned __int128)DS.n_items * q) / (cn_ * segments));
    };
    int64_t n_my = 0;
    for (int t = 0; t < segments; t++) n_my += (int64_t)(segment_at(cb + cn_ * t + 1) - segment_at(cb + cn_ * t));
    const int chunks = DS.chunks, chunks_case = DS.chunks_case;
    const int nst = (chunks + 1) >> 1;                // K stages of an item

    if (tid == 0) {
        for (int s = 0; s < kStages; s++) {
            mbar_init(&full_ab[s], 4 + 1);            // one producer group + the TMA thread
            mbar_init(&empty_ab[s], 1);
        }
        for (int b = 0; b < S::Accs; b++) mbar_init(&acc_empty[b], kEpiWarps);
        for (int b = 0; b < 2; b++) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&tot_full[b], kProdWarps);
            mbar_init(&tot_empty[b], kEpiWarps);
        }
        for (int q = 0; q < kDescDepth; q++) {
            mbar_init(&desc_full[q], 1);
            mbar_init(&desc_empty[q], kEpiWarps + kProdWarps);
        }
        mbar_init(&drain_bar, 1);
        abort_flag = 0;
        if constexpr (COLLECT) {
            over_flag = 0;
            g_end_item = ~0u;
        }
        g_wait_limit_ns = P.wait_ns ? P.wait_ns : kTimeoutNs;
        ES.list_len = 0; ES.nbuf = 0; ES.stop = 0; ES.any = 0; ES.seen = 0;
        ES.thr = ES.next_thr = COLLECT ? P.collect.thr : -1.0f;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kWarpMma) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_sh)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (P.scores)
        for (int q = tid; q <= (int)d.m; q += R::Threads) tlog[q] = P.tlog[q];
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_sh;
    if (warp < 4) {
        // scale factors (UE8M0, 127 = 1), the same in every byte pair's rows
        // and columns, so their placement does not matter: A all 1; B bytes
        // 0-1 the controls' 1, bytes 2-3 the cases' 2^p
        const uint32_t q = tmem_base + ((uint32_t)(warp * 32) << 16);
        const uint32_t cs = 127u + (uint32_t)DS.comb_p;
        tmem_fill16(q + kScaleACol, 0x7F7F7F7Fu);
        tmem_fill16(q + kScaleBCol, 0x00007F7Fu | (cs << 16) | (cs << 24));
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    if (warp == kWarpTma) {
        // ------------------------------------------------ TMA + descriptors
        // the whole warp runs the loop (its searches probe with all lanes),
        // lane 0 writes, arrives and issues the copies
        if (n_my > 0) {
            // the segment's next item: M tile (prefix iterator) and N tile u
            PrefixIter it;
            int64_t u = 0;
            int seg = -1;
            uint64_t seg_left = 0;
            int32_t j1 = 0, row0 = 0;            // pair tiles: first SNP, its first operand row,
            uint64_t mt = 0, mtiles = 0;         // and the M tile among those of j1
            auto next_segment = [&]() {
                uint64_t w0;
                do {
                    seg++;
                    w0 = segment_at(cb + cn_ * seg);
                    seg_left = segment_at(cb + cn_ * seg + 1) - w0;
                } while (seg_left == 0);
                const int64_t lo = warp_last(0, d.n - 1, [&](int64_t x) { return DS.item_cum[x] <= w0; });
                const int32_t c0 = (int32_t)lo;
                const uint64_t off = w0 - DS.item_cum[c0];
                if constexpr (PAIR) {
                    // M tiles within N tiles within j1
                    j1 = c0;
                    mtiles = (DS.pcum[j1] + kPPT - 1) / kPPT;
                    u = (int64_t)(off / mtiles);
                    mt = off % mtiles;
                    row0 = (int32_t)DS.brow[j1];
                    prefix_unrank(DS, K - 1, mt * (uint64_t)kPPT, it);
                } else {
                    const int64_t nt0 = panel_ntiles(d.n, c0, kJ);
                    const uint64_t tfirst = (DS.pcum[c0] + kPPT - 1) / kPPT;
                    const uint64_t t = tfirst + off / (uint64_t)nt0;
                    u = (int64_t)(off % (uint64_t)nt0);
                    prefix_unrank(DS, K, t * (uint64_t)kPPT, it);
                }
            };
            next_segment();
            int32_t tile_snp[kPPT * km1];
            int32_t nvalid = 0, cmin = it.c;
            // place of this lane's prefixes (lane, lane + 32) in the singles
            uint64_t single[2] = {0, 0};
            auto fill_tile = [&]() {
                nvalid = 0;
                cmin = it.c;
                int32_t my_c[2] = {-1, -1};
                uint64_t my_q[2] = {0, 0};
#pragma unroll
                for (int p = 0; p < kPPT; p++) {
                    if (it.q < DS.n_prefix) {
#pragma unroll
                        for (int s2 = 0; s2 < km1 - 1; s2++) tile_snp[p * km1 + s2] = it.a[s2];
                        tile_snp[p * km1 + km1 - 1] = it.c;
                        if (lane == (p & 31)) { my_c[p >> 5] = it.c; my_q[p >> 5] = it.q; }
                        nvalid++;
                        prefix_next(DS, km1 + 1, it);
                    }
                }
                if (DS.singles) {
#pragma unroll
                    for (int h = 0; h < 2; h++)
                        if (my_c[h] >= 0)
                            single[h] = DS.scum[my_c[h]] +
                                        (my_q[h] - DS.pcum[my_c[h]]) * (uint64_t)single_groups(d.n, my_c[h]);
                }
            };
            fill_tile();
            // item i's descriptor, and the operand row its N tile starts at.
            // Once a collecting epilogue has found too many there is none:
            // every role ends at this item, all stages before it taken (an
            // abort instead would leave this warp's last loads to barriers
            // that the producers no longer reach, two seconds a stage)
            int y_next = 0;
            auto write_desc = [&](int64_t i) -> bool {
                if constexpr (COLLECT) {
                    if (__any_sync(0xffffffffu, over_flag)) {
                        g_end_item = (uint32_t)i;
                        return false;
                    }
                }
                const int dq = (int)(i % kDescDepth);
                const uint32_t ud = (uint32_t)(i / kDescDepth);
                if (!__all_sync(0xffffffffu, mbar_wait(&desc_empty[dq], (ud & 1) ^ 1, &abort_flag))) return false;
                const int32_t tile_j0 = (int32_t)panel_j0(PAIR ? j1 : cmin) + (int32_t)(u * kJ);
                if (DS.singles) {
                    if (lane < kPPT) desc[dq].single[lane] = single[0];
                    if (lane + 32 < kPPT) desc[dq].single[lane + 32] = single[1];
                    __syncwarp();
                }
                if (lane == 0) {
                    Desc &D = desc[dq];
                    D.j0 = tile_j0;
                    D.j1 = j1;
                    D.nvalid = nvalid;
#pragma unroll
                    for (int q = 0; q < kPPT * km1; q++) D.snp[q] = tile_snp[q];
                    // columns in use: 2 (4) per last SNP below n, in steps of 16
                    const int32_t live = kColsPerSnp * ((int32_t)d.n - tile_j0);
                    const uint32_t ncol = live >= S::N ? (uint32_t)S::N : (uint32_t)((live + 15) & ~15);
                    item_idesc[dq] = make_idesc(ncol);
                    mbar_arrive(&desc_full[dq]);
                }
                y_next = PAIR ? row0 + (int)(u * S::N) : 2 * tile_j0;
                return true;
            };
            // the tile after this one (there is one)
            auto next_tile = [&]() {
                if (--seg_left == 0) {
                    next_segment();
                    fill_tile();
                    return;
                }
                if constexpr (PAIR) {
                    if (++mt == mtiles) {
                        // next N tile of j1, or the first of the next SNP:
                        // from the first prefix again
                        mt = 0;
                        if (++u == panel_ntiles(d.n, j1, kJ)) {
                            u = 0;
                            j1++;
                            mtiles = (DS.pcum[j1] + kPPT - 1) / kPPT;
                            row0 = (int32_t)DS.brow[j1];
                        }
                        it.q = 0;
                        it.c = km1 - 1;
#pragma unroll
                        for (int t = 0; t < km1 - 1; t++) it.a[t] = t;
                    }
                    fill_tile();
                } else if (++u == panel_ntiles(d.n, cmin, kJ)) {
                    u = 0;
                    fill_tile();
                }
            };
            uint64_t g = 0;
            int s = 0;
            uint32_t ph = 0;
            long long w_tma = 0;
            bool on = write_desc(0);
            for (int64_t i = 0; i < n_my && on; i++) {
                const int y = y_next;
                // the next item's descriptor before this one's loads, which
                // wait for the ring: its producers start without a gap (the
                // descriptor written after them: 48.5 ms at order 3,
                // 2000 x 4000)
                if (i + 1 < n_my) {
                    next_tile();
                    on = write_desc(i + 1);
                }
                for (int kc = 0; kc < nst; kc++, g++) {
                    if (!__all_sync(0xffffffffu, wait_here(&empty_ab[s], ph ^ 1, &abort_flag, w_tma))) { on = false; break; }
                    if (lane == 0) {
                        mbar_arrive_tx(&full_ab[s], (uint32_t)kBBytes);
                        tma_load_2d(stages_b + s * kBBytes, tmap, kc * kRowBytes, y, &full_ab[s]);
                    }
                    __syncwarp();
                    if (++s == kStages) { s = 0; ph ^= 1; }
                }
            }
            if (P.waits && lane == 0) P.waits[blockIdx.x * kWaitSlots + 6] = (unsigned long long)w_tma;
            for (int q = 0; q < kStages; q++) {
                if (g > (uint64_t)q) {
                    const uint64_t last = ((g - 1 - q) / kStages) * kStages + q;
                    const uint32_t us = (uint32_t)(last / kStages);
                    const uint64_t t0 = now_ns();
                    while (!mbar_try(&full_ab[q], us & 1) && now_ns() - t0 < kTimeoutNs) {}
                }
            }
        }
    } else if (warp == kWarpMma) {
        // ------------------------------------------------------------- MMA
        if (n_my > 0) {
            // The issue loop is run by the whole warp in step; one elected
            // lane issues the MMAs and commits.  Only a few MMAs queue behind
            // the running one, so the tensor pipe idles through whatever this
            // instruction stream does between two MMAs: the next stage's
            // barrier is tested and its operands' descriptors are formed
            // between the MMAs of a stage (measured at order 4, 500 x 8192:
            // testing after the last MMA left 290 cycles a stage exposed), and
            // the class boundary of the separate variant has its own branch.
            const uint32_t leader = elect_one();
            const uint32_t tb = uniform(tmem_base);
            const uint64_t ad0 = sdesc(uniform(smem_u32(stages_a))), bd0 = sdesc(uniform(smem_u32(stages_b)));
            // stage strides in descriptor address units
            constexpr uint32_t kStageDescA = kTileBytes >> 4, kStageDescB = kBBytes >> 4;
            const uint32_t sfa = tb + kScaleACol, sfb = tb + kScaleBCol;
            const int u_chunks = (int)uniform((uint32_t)chunks), u_case = (int)uniform((uint32_t)chunks_case);
            const int u_nst = (u_chunks + 1) >> 1;
            const uint32_t u_items = uniform((uint32_t)n_my);
            int s = 0;
            uint32_t ph = 0;
            int ab = 0;                              // accumulator buffer and the phase of its uses
            uint32_t aph = 0;
            long long w_a = 0, w_b = 0, w_acc = 0;
            const long long t_start = clock64();
            auto next_acc = [&](uint32_t &col) -> bool {
                if (!__all_sync(0xffffffffu, mbar_test(&acc_empty[ab], aph ^ 1)) &&
                    !wait_inline<false>(&acc_empty[ab], aph ^ 1, &abort_flag, w_acc, 0))
                    return false;
                tc_fence_after();
                col = tb + (uint32_t)(ab * S::N);
                if (++ab == S::Accs) { ab = 0; aph ^= 1; }
                return true;
            };
            bool ready = false;                      // stage s, phase ph is known to be full
            for (uint32_t i = 0; i < u_items; i++) {
                uint32_t dcol = 0, idesc = 0;
                if (!next_acc(dcol)) break;
                bool ok = true;
                for (int st = 0; st < u_nst; st++) {
                    if (!__all_sync(0xffffffffu, ready)) {
                        ok = wait_inline<COLLECT>(&full_ab[s], ph, &abort_flag, w_a, i);
                        if (!ok) break;
                    }
                    tc_fence_after();
                    // the item's column count is in place once its first stage is full
                    if (st == 0) idesc = uniform(item_idesc[i % kDescDepth]);
                    const uint64_t ad = ad0 + (uint64_t)(s * kStageDescA), bd = bd0 + (uint64_t)(s * kStageDescB);
                    const int c = 2 * st;
                    const bool second = c + 1 < u_chunks;
                    uint64_t *const freed = &empty_ab[s];
                    if (++s == kStages) { s = 0; ph ^= 1; }
                    if (!C && (c == u_case || c + 1 == u_case) && c > 0) {
                        // the control accumulator starts in this stage
                        if (c + 1 == u_case) {
                            mma_f4_warp(dcol, ad, bd, 1u, leader, idesc, sfa, sfb);
                            mma_f4_warp(dcol, ad + 2, bd + 2, 1u, leader, idesc, sfa, sfb);
                            ok = next_acc(dcol);
                            if (!ok) break;
                            mma_f4_warp(dcol, ad + 4, bd + 4, 0u, leader, idesc, sfa, sfb);
                        } else {
                            ok = next_acc(dcol);
                            if (!ok) break;
                            mma_f4_warp(dcol, ad, bd, 0u, leader, idesc, sfa, sfb);
                            mma_f4_warp(dcol, ad + 2, bd + 2, 1u, leader, idesc, sfa, sfb);
                            if (second) mma_f4_warp(dcol, ad + 4, bd + 4, 1u, leader, idesc, sfa, sfb);
                        }
                        if (second) mma_f4_warp(dcol, ad + 6, bd + 6, 1u, leader, idesc, sfa, sfb);
                        ready = mbar_test(&full_ab[s], ph);
                    } else if (!C && c == 0 && u_case == 1) {
                        // both classes within the first stage
                        mma_f4_warp(dcol, ad, bd, 0u, leader, idesc, sfa, sfb);
                        mma_f4_warp(dcol, ad + 2, bd + 2, 1u, leader, idesc, sfa, sfb);
                        ok = next_acc(dcol);
                        if (!ok) break;
                        mma_f4_warp(dcol, ad + 4, bd + 4, 0u, leader, idesc, sfa, sfb);
                        mma_f4_warp(dcol, ad + 6, bd + 6, 1u, leader, idesc, sfa, sfb);
                        ready = mbar_test(&full_ab[s], ph);
                    } else {
                        const uint32_t id0 = C && c < u_case ? idesc | kIdescCase : idesc;
                        const uint32_t id1 = C && c + 1 < u_case ? idesc | kIdescCase : idesc;
                        mma_f4_warp(dcol, ad, bd, st ? 1u : 0u, leader, id0, sfa, sfb);
                        mma_f4_warp(dcol, ad + 2, bd + 2, 1u, leader, id0, sfa, sfb);
                        ready = mbar_test(&full_ab[s], ph);
                        if (second) {
                            mma_f4_warp(dcol, ad + 4, bd + 4, 1u, leader, id1, sfa, sfb);
                            mma_f4_warp(dcol, ad + 6, bd + 6, 1u, leader, id1, sfa, sfb);
                        }
                    }
                    mma_commit_warp(freed, leader);
                }
                if (!ok) break;
                mma_commit_warp(&acc_full[i & 1], leader);
            }
            if (P.waits && leader) {
                unsigned long long *wp = P.waits + blockIdx.x * kWaitSlots;
                wp[0] = (unsigned long long)w_a;
                wp[1] = (unsigned long long)w_b;
                wp[2] = (unsigned long long)w_acc;
                wp[7] = (unsigned long long)(clock64() - t_start);
            }
            __syncwarp();
            mma_commit_warp(&drain_bar, leader);
            const uint64_t t0 = now_ns();
            while (!mbar_try(&drain_bar, 0) && now_ns() - t0 < kTimeoutNs) {}
        }
    } else if (warp >= kEpiWarps) {
        // ---------------------------------------------------- A producers
        // Thread t owns tile row r = t % 128 in the stages of group t / 128
        // (with two groups they take alternate stages), and writes all 256
        // individuals of the row's stage: eight mask words, each expanded to
        // 16 bytes.
        const int t = tid - kEpiThreads;     // 0 .. 32 kProdWarps - 1
        const int r = t & 127;
        const int grp = t >> 7;
        const int l = r & 31, w = r >> 5;
        // 16-byte piece c of the row is stored at piece c ^ (r % 8): the row's
        // address with r % 8 in the piece bits, xor c
        const uint32_t arow0 = smem_u32(stages_a) + (uint32_t)(r * kRowBytes + ((r & 7) << 4));
        const int64_t stage_stride = 6 * (d.n + 1);
        uint64_t g = 0;                      // stages of the CTA so far (all groups)
        long long w_prod = 0, w_prod_acc = 0;
        // A warp's lanes leave together, by votes: one that left alone would be
        // waited for at the next __syncwarp.
        for (int64_t i = 0; i < n_my; i++) {
            const int dq = (int)(i % kDescDepth);
            const uint32_t ud = (uint32_t)(i / kDescDepth);
            const bool go = wait_desc<COLLECT>(&desc_full[dq], ud & 1, &abort_flag, i) && !abort_flag;
            if (!__all_sync(0xffffffffu, go)) break;
            const Desc &D = desc[dq];
            // the row's SNP rows at stage 0; rows of no prefix read the zero
            // rows kept past the last SNP
            const uint4 *rows[km1];
#pragma unroll
            for (int tt = 0; tt < km1; tt++) rows[tt] = DS.rows + d.n * 6;
            if (kWide ? r < kPR : l < kPPW * kPR) {
                const int p = kWide ? 0 : w * kPPW + l / kPR;
                if (p < D.nvalid) {
                    int rem = kWide ? r : l % kPR, div = kPR / 3;
#pragma unroll
                    for (int tt = 0; tt < km1; tt++) {
                        const int gg = rem / div;
                        rem -= gg * div;
                        div = div > 1 ? div / 3 : 1;
                        rows[tt] = DS.rows + (D.snp[p * km1 + tt] * 3 + gg) * 2;
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&desc_empty[dq]);
            uint32_t t1 = 0, ta = 0;             // individuals of the row: cases, all
            bool ok = true;
            // this group's first stage of the item
            const int st0 = (int)(((uint64_t)grp + kGroups - (g % kGroups)) % kGroups);
            // the prefix SNPs' words for the next own stage (chunk 2 st and,
            // where it exists, 2 st + 1), kept as loaded and ANDed when their
            // stage is produced, so no instruction waits for a load issued for
            // a later stage
            constexpr int kPf = km1 <= 2 ? EPI_TC_PREFETCH : 2;
            static_assert(kPf % 2 == 0, "stages are produced in twos");
            uint4 ring[kPf][2][km1];
            auto fetch = [&](int st, uint4 (*dst)[km1]) {
#pragma unroll
                for (int hh = 0; hh < 2; hh++)
#pragma unroll
                    for (int tt = 0; tt < km1; tt++) dst[hh][tt] = __ldg(rows[tt] + st * stage_stride + hh);
            };
#pragma unroll
            for (int u = 0; u < kPf; u++) fetch(st0 + kGroups * u, ring[u]);
            const uint64_t gs = g + (uint64_t)st0;             // global stage of the first own stage
            int s = (int)(gs % kStages);
            uint32_t ph = (uint32_t)((gs / kStages) & 1);
            // one stage of this row from its words
            auto produce = [&](int st, int slot, const uint4 (*w)[km1]) {
                const uint32_t arow = arow0 + (uint32_t)(slot * kTileBytes);
#pragma unroll
                for (int hh = 0; hh < 2; hh++) {
                    uint4 cur = w[hh][0];
#pragma unroll
                    for (int tt = 1; tt < km1; tt++) {
                        const uint4 v = w[hh][tt];
                        cur.x &= v.x; cur.y &= v.y; cur.z &= v.z; cur.w &= v.w;
                    }
                    const uint32_t wv4[4] = {cur.x, cur.y, cur.z, cur.w};
                    const uint32_t c4 = __popc(wv4[0]) + __popc(wv4[1]) + __popc(wv4[2]) + __popc(wv4[3]);
                    t1 += 2 * st + hh < chunks_case ? c4 : 0u;
                    ta += c4;
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        // output word i = bit i of every nibble of the mask word
                        const uint32_t wv = wv4[q];
                        st_shared_v4(arow ^ (uint32_t)((4 * hh + q) << 4), wv & 0x11111111u, wv & 0x22222222u,
                                     wv & 0x44444444u, (wv >> 1) & 0x44444444u);
                    }
                }
            };
            // Two own stages at a time: the barrier tests, the proxy fence and
            // the arrivals wait for shared memory (about 400 of 930 cycles a
            // stage taken one by one, at order 4)
            for (int sb = st0; sb < nst && ok; sb += kGroups * kPf) {
#pragma unroll
                for (int u = 0; u < kPf; u += 2) {
                    const int st = sb + kGroups * u;
                    if (st >= nst) break;
                    const bool two = st + kGroups < nst;
                    int s2 = s + kGroups;
                    uint32_t ph2 = ph;
                    if (s2 >= kStages) { s2 -= kStages; ph2 ^= 1; }
                    // (one vote for both tests: a vote for each, or one after the
                    // lanes' own waits, took 0.5 to 2 % more at order 4)
                    if (!__all_sync(0xffffffffu, mbar_test(&empty_ab[s], ph ^ 1) &&
                                                     (!two || mbar_test(&empty_ab[s2], ph2 ^ 1)))) {
                        ok = wait_together(&empty_ab[s], ph ^ 1, &abort_flag, w_prod) &&
                             (!two || wait_together(&empty_ab[s2], ph2 ^ 1, &abort_flag, w_prod));
                        if (!ok) break;
                    }
                    produce(st, s, ring[u]);
                    if (two) produce(st + kGroups, s2, ring[u + 1]);
                    fetch(st + kGroups * kPf, ring[u]);
                    fetch(st + kGroups * (kPf + 1), ring[u + 1]);
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) {
                        mbar_arrive(&full_ab[s]);
                        if (two) mbar_arrive(&full_ab[s2]);
                    }
                    // the next own stage: kGroups global stages on from the last
                    s = two ? s2 + kGroups : s2;
                    ph = ph2;
                    if (two && s >= kStages) { s -= kStages; ph ^= 1; }
                }
            }
            if (!ok) break;
            g += (uint64_t)nst;
            const int b = (int)(i & 1);
            const uint32_t ub = (uint32_t)(i >> 1);
            ok = ok && wait_fast(&tot_empty[b], (ub & 1) ^ 1, &abort_flag, w_prod_acc);
            if (!__all_sync(0xffffffffu, ok)) break;
            tot[((b * 128 + r) * kGroups + grp) * 2 + 0] = t1;
            tot[((b * 128 + r) * kGroups + grp) * 2 + 1] = ta - t1;
            __syncwarp();
            if (lane == 0) mbar_arrive(&tot_full[b]);
        }
        if (P.waits && t == 0) {
            P.waits[blockIdx.x * kWaitSlots + 3] = (unsigned long long)w_prod;
            P.waits[blockIdx.x * kWaitSlots + 4] = (unsigned long long)w_prod_acc;
        }
    } else {
        // -------------------------------------------------------- epilogue
        const int quad = warp & 3;           // TMEM lane quadrant
        const int jhalf = warp >> 2;         // column group: chunks jhalf + kCG i of the quadrant
        const int r = quad * 32 + lane;      // tile row = TMEM lane
        const int pos = kWide ? r : lane % kPR;       // row of the prefix's table
        const int pl = kWide ? 0 : lane / kPR;
        const bool lane_real = kWide ? r < kPR : lane < kPPW * kPR;
        const MiConstF32 mc = make_mi_const(d.m, d.m1, d.m0);
        const float p2 = (float)(1u << DS.comb_p);
        RowScreen<C> rs;
        rs.m23 = f2_pack(8388608.0f, 8388608.0f);
        rs.neg_m23 = f2_pack(-8388608.0f, -8388608.0f);
        rs.neg1 = f2_pack(-1.0f, -1.0f);
        const float q1 = C ? 0.5f * p2 : 1.0f;
        rs.half = f2_pack(0.5f, 0.5f);
        rs.neg2 = f2_pack(-2.0f, -2.0f);
        rs.hi_mask = C ? ~((1u << (DS.comb_p - 1)) - 1u) : 0u;
        rs.inv_q1 = 1.0f / q1;
        rs.inv_q = f2_pack(rs.inv_q1, rs.inv_q1);
        rs.neg_pi = f2_pack(-DS.sc_pi, -DS.sc_pi);
        rs.sc.c2 = f2_pack(DS.c2, DS.c2);
        rs.sc.c3 = f2_pack(DS.c3, DS.c3);
        rs.sc.c4 = f2_pack(DS.c4, DS.c4);
        rs.sc.c5a = f2_pack(DS.c5a, DS.c5a);
        rs.sc.c5b = f2_pack(DS.c5b, DS.c5b);
        rs.sc.tiny = f2_pack(1e-30f, 1e-30f);
        const float vscale = DS.vscale, voff = DS.voff;
        // (DS lies in the kernel parameters or in global memory: what the
        // chunk loop needs of it is read once)
        const bool poly = DS.poly != 0, store = !PAIR && DS.store != 0;
        const bool scoring = !PAIR && (K == 3 || K == 4) && P.scores;
        float4 *const singles = DS.singles;
        float *wb = wsum + warp * 256;
        int ab = 0;                          // first accumulator buffer of the item
        float thr = ES.thr;                  // the threshold as of the last item's closing barrier
        long long w_epi = 0;
        for (int64_t i = 0; i < n_my; i++) {
            const int dq = (int)(i % kDescDepth);
            const uint32_t ud = (uint32_t)(i / kDescDepth);
            const int b = (int)(i & 1);
            const uint32_t ub = (uint32_t)(i >> 1);
            bool ok = wait_desc<COLLECT>(&desc_full[dq], ud & 1, &abort_flag, i);
            ok = ok && wait_fast(&acc_full[b], ub & 1, &abort_flag, w_epi);
            ok = ok && wait_fast(&tot_full[b], ub & 1, &abort_flag, w_epi);
            ok = __all_sync(0xffffffffu, ok);
            tc_fence_after();
            // this item's accumulators (case and control with separate classes)
            const int ab1 = C ? ab : (ab + 1 == S::Accs ? 0 : ab + 1);
            const uint32_t tq = tmem_base + ((uint32_t)(quad * 32) << 16);
            const uint32_t ta_case = tq + (uint32_t)(ab * S::N), ta_ctrl = tq + (uint32_t)(ab1 * S::N);
            const int ab_case = ab;
            ab = ab1 + 1 == S::Accs ? 0 : ab1 + 1;
            const Desc &D = desc[dq];
            const int p = quad * kPPW + pl;
            const bool prow = ok && lane_real && p < D.nvalid;
            int32_t psnp[km1];
#pragma unroll
            for (int tt = 0; tt < km1; tt++) psnp[tt] = prow ? D.snp[p * km1 + tt] : 0;
            // the searched last SNPs of the prefixes whose (prefix, last SNP)
            // pairs this lane sums: pair lane + 32 q is prefix (lane + 32 q) / 8
            // of the warp and last SNP (lane + 32 q) % 8 of each chunk (at
            // orders 4-5 the warp's only prefix, last SNP lane % 8)
            int32_t plo[kPairIters], phi[kPairIters];
#pragma unroll
            for (int q = 0; q < kPairIters; q++) {
                const int pp = kPPW > 1 ? (lane + 32 * q) / kCS : 0;
                const int pt = quad * kPPW + pp;
                plo[q] = 1;
                phi[q] = 0;                      // empty: no valid last SNP
                if (ok && (kPPW <= 1 || pp < kPPW) && pt < D.nvalid) {
                    int32_t qs[km1];
#pragma unroll
                    for (int tt = 0; tt < km1; tt++) qs[tt] = D.snp[pt * km1 + tt];
                    if constexpr (PAIR) {
                        // (prefix, j1) is a prefix of the combination
                        if (qs[km1 - 1] < D.j1) { plo[q] = D.j1 + 1; phi[q] = (int32_t)d.n; }
                    } else {
                        last_snp_range<km1>(DS, d, qs, plo[q], phi[q]);
                    }
                }
            }
            {
                uint32_t T1 = 0, T0 = 0;
#pragma unroll
                for (int gq = 0; gq < kGroups; gq++) {
                    T1 += tot[((b * 128 + r) * kGroups + gq) * 2 + 0];
                    T0 += tot[((b * 128 + r) * kGroups + gq) * 2 + 1];
                }
                // rows of no prefix count nothing: their totals are 0
                rs.set_row(u2f_exact(T1), u2f_exact(T0), q1);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&tot_empty[b]);
            // the other CTAs' threshold, for the next item (loaded early)
            const float gthr = tid == 0 ? __uint_as_float(*(volatile uint32_t *)DS.global_thr) : 0.0f;
            float cut = thr * DS.cut_mul - DS.cut_add;
            int list_len = ES.list_len;
            const int32_t j0 = D.j0;
            // before the item's closing barrier: the threshold the other CTAs
            // have reached, and whether a role gave up
            auto refresh = [&]() {
                if (tid == 0) {
                    ES.next_thr = gthr > 0.0f ? fmaxf(ES.thr, gthr) : ES.thr;
                    ES.stop = abort_flag;
                    if constexpr (COLLECT) {
                        // more than the caller's array holds: no further descriptors
                        if (*(volatile unsigned long long *)P.collect.n > P.collect.cap) over_flag = 1;
                        if (g_end_item == (uint32_t)i) ES.stop = 1;
                    }
                }
            };
            // one chunk's accumulators (queued): last SNPs j0 + kCS jcg ..
            auto load_chunk = [&](int jcg, uint32_t *cs, uint32_t *cn) {
                if constexpr (kChunkCols == 16) {
                    TMEM_LD16(ta_case + (uint32_t)(16 * jcg), cs);
                    if constexpr (!C) TMEM_LD16(ta_ctrl + (uint32_t)(16 * jcg), cn);
                } else {
                    TMEM_LD8(ta_case + (uint32_t)(8 * jcg), cs);
                    if constexpr (!C) TMEM_LD8(ta_ctrl + (uint32_t)(8 * jcg), cn);
                }
            };
            auto release_acc = [&]() {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&acc_empty[ab_case]);
                    if constexpr (!C) mbar_arrive(&acc_empty[ab1]);
                }
            };
            // validation: every table of the chunk, as counts
            auto dump_chunk = [&](int jb, const uint32_t *cs, const uint32_t *cn) {
                if (!prow) return;
                int32_t jlo, jhi;
                last_snp_range<km1>(DS, d, psnp, jlo, jhi);
#pragma unroll 1
                for (int jj = 0; jj < 8; jj++) {
                    const int32_t j = jb + jj;
                    if (j < jlo || j >= jhi) continue;
                    float a[3] = {}, bb[3] = {};
#pragma unroll
                    for (int h = 0; h < 4; h++)
                        if (h == jj >> 1) rs.counts(cs, cn, h, jj & 1, a, bb);
                    constexpr int cells = kPR * 3;
                    uint32_t *o = P.dump + (DS.total - 1 - prefix_rank_sum<km1>(d, psnp) - (uint64_t)(d.n - 1 - j)) *
                                               2 * cells;
#pragma unroll
                    for (int g3 = 0; g3 < 3; g3++) {
                        o[pos * 3 + g3] = f2u_exact(a[g3]);
                        o[cells + pos * 3 + g3] = f2u_exact(bb[g3]);
                    }
                }
            };
            // precise single-precision terms of this row for column jsel
            auto row_precise = [&](const uint32_t *cs, const uint32_t *cn, int jsel) -> SumF32 {
                float a[3] = {}, bb[3] = {};
#pragma unroll
                for (int h = 0; h < 4; h++)
                    if (h == jsel >> 1) rs.counts(cs, cn, h, jsel & 1, a, bb);
                return row_terms_precise(f2u_exact(a[0]), f2u_exact(bb[0]), f2u_exact(a[1]), f2u_exact(bb[1]),
                                         f2u_exact(a[2]), f2u_exact(bb[2]), mc);
            };
            // combination of tile prefix pt and last SNP j into the buffer
            auto keep = [&](float score, int pt, int32_t j) {
                if (score >= thr) {
                    int32_t qs[km1];
#pragma unroll
                    for (int tt = 0; tt < km1; tt++) qs[tt] = D.snp[pt * km1 + tt];
                    uint64_t rank = DS.total - 1 - prefix_rank_sum<km1>(d, qs, K) - (uint64_t)(d.n - 1 - j);
                    if constexpr (PAIR) rank -= binom_at(d.binom, d.n, d.n - 1 - D.j1, 2);
                    if constexpr (COLLECT) {
                        const unsigned long long at = atomicAdd(P.collect.n, 1ull);
                        if (at < P.collect.cap) P.collect.ranks[at] = rank;
                    } else {
                        const int slot = list_len + atomicAdd(&ES.nbuf, 1);
                        if (DS.top_n > 0) atomicAdd(DS.hist + hist_bin(score), 1u);
                        sc[slot] = score;
                        rk[slot] = rank;
                    }
                }
            };
            // the threshold of everything kept so far, by all CTAs
            auto share_threshold = [&]() {
                epi_bar<kEpiThreads>();
                const int kept = ES.list_len + ES.nbuf;
                if (DS.top_n > 0) {
                    __threadfence();
                    const float t = hist_threshold<kEpiThreads>(DS.hist, DS.top_n, hist_tmp, tid) * DS.thr_mul;
                    if (tid == 0) {
                        ES.seen = kept;
                        if (t > ES.thr) {
                            ES.thr = t;
                            atomicMax(DS.global_thr, __float_as_uint(t));
                        }
                    }
                }
                epi_bar<kEpiThreads>();
                thr = fmaxf(thr, ES.thr);
            };
            // Without a threshold every combination needs its precise score:
            // all prefixes of the warp at once, column by column (one flagged
            // pair at a time, as below, the first items of a CTA took
            // milliseconds at order 2), summed as the flagged ones are.
            bool cold = thr < 0.0f && !store && !scoring;
            // 8 row values per lane -> transposed sums: the lane of pair
            // (prefix pp, last SNP jj) adds rows pp kPR .. of column jj (all
            // banks distinct); at orders 4-5 four lanes share a column
            auto store_rows = [&](const float *vrow) {
                reinterpret_cast<float4 *>(wb + lane * 8)[0] = make_float4(vrow[0], vrow[1], vrow[2], vrow[3]);
                reinterpret_cast<float4 *>(wb + lane * 8)[1] = make_float4(vrow[4], vrow[5], vrow[6], vrow[7]);
                __syncwarp();
            };
            auto column_sum = [&]() -> float {
                constexpr int kPart = kWide ? 8 : 7;
                const int part = lane >> 3;
                float v = 0.0f, w2 = 0.0f;
#pragma unroll
                for (int rr = 0; rr < kPart; rr++) {
                    const int row = part * kPart + rr;
                    const float x = (kWide || row < kPR) ? wb[row * 8 + (lane & 7)] : 0.0f;
                    if (rr & 1) w2 += x;
                    else v += x;
                }
                v += w2;
                v += __shfl_xor_sync(0xffffffffu, v, 8);
                v += __shfl_xor_sync(0xffffffffu, v, 16);
                return v;
            };
            if constexpr (kWide) {
                // order 5: the item's sums of each quadrant's rows, then one
                // pass over its last SNPs, then (rarely) the precise scores
                // of the flagged ones
#pragma unroll 1
                for (int jcg = jhalf; jcg < kQC; jcg += kCG) {
                    const int32_t jb = j0 + 8 * jcg;
                    float v = 0.0f;
                    if (ok && quad < 3 && jb < (int32_t)d.n) {
                        uint32_t cs[16], cn[C ? 1 : 16];
                        load_chunk(jcg, cs, cn);
                        tmem_wait_ld();
                        if (P.dump) dump_chunk(jb, cs, cn);
                        if (cold) {
#pragma unroll 1
                            for (int jj = 0; jj < 8; jj++) {
                                const float e = warp_sum(prow ? row_precise(cs, cn, jj) : SumF32());
                                if (lane == jj) v = e;
                            }
                        } else {
                            float vrow[8];
                            if (poly) rs.bound(cs, cn, vrow);
                            else rs.logs(cs, cn, vrow);
                            store_rows(vrow);
                            v = column_sum();
                            __syncwarp();
                        }
                    }
                    if (lane < 8) wred[quad][8 * jcg + lane] = v;
                }
                epi_bar<kEpiThreads>();
                bool any = false;
                // the tile's one prefix is every thread's
                int32_t qs[km1], plo_any = 1, phi_any = 0;
#pragma unroll
                for (int tt = 0; tt < km1; tt++) qs[tt] = D.snp[tt];
                if (ok) last_snp_range<km1>(DS, d, qs, plo_any, phi_any);
                for (int q = tid; q < kJ; q += kEpiThreads) {
                    const float tv = wred[0][q] + wred[1][q] + wred[2][q];
                    const int32_t j = j0 + q;
                    bool f = false;
                    if (j >= plo_any && j < phi_any) {
                        if (cold) keep(__fdiv_rn(tv, mc.fm), 0, j);
                        else f = fmaf(tv, vscale, voff) >= cut;
                    }
                    wflag[q] = f ? 1 : 0;
                    any |= f;
                }
                if (any) ES.any = 1;
                epi_bar<kEpiThreads>();
                if (ES.any) {
#pragma unroll 1
                    for (int jcg = jhalf; jcg < kQC; jcg += kCG) {
                        const unsigned long long fl = *reinterpret_cast<const unsigned long long *>(&wflag[8 * jcg]);
                        if (!fl || quad == 3) continue;
                        uint32_t cs[16], cn[C ? 1 : 16];
                        load_chunk(jcg, cs, cn);
                        tmem_wait_ld();
#pragma unroll 1
                        for (int jj = 0; jj < 8; jj++) {
                            if (!wflag[8 * jcg + jj]) continue;
                            const float e = warp_sum(prow ? row_precise(cs, cn, jj) : SumF32());
                            if (lane == 0) wpre[quad][8 * jcg + jj] = e;
                        }
                    }
                }
                release_acc();
                if (ES.any) {
                    epi_bar<kEpiThreads>();
                    for (int q = tid; q < kJ; q += kEpiThreads) {
                        if (!wflag[q]) continue;
                        keep(__fdiv_rn(wpre[0][q] + wpre[1][q] + wpre[2][q], mc.fm), 0, j0 + q);
                    }
                }
                refresh();
                epi_bar<kEpiThreads>();
                if (tid == 0) ES.any = 0;
            } else if constexpr (PAIR) {
                // Chunks of kCS last SNPs: kH groups of two, each 8 columns and
                // one float4 (two with separate classes) of single counts per
                // row, loaded one chunk ahead
                constexpr int kAcc = C ? 1 : 2;
                const int live_chunks = ok ? min(kQC, ((int32_t)d.n - j0 + kCS - 1) / kCS) : 0;
                const int mine = (live_chunks - jhalf + kCG - 1) / kCG;
                const bool row_in = prow && psnp[km1 - 1] < D.j1;
                // rows outside read one place of the table (their values are dropped)
                const int32_t base = row_in ? (int32_t)panel_j0(psnp[km1 - 1]) : 0;
                const float4 *sp = singles + (row_in ? (D.single[p] * kPR + pos) * kAcc : 0);
                const int64_t gstep = row_in ? (int64_t)kPR * kAcc : 0;
                auto load_singles = [&](int32_t j, float4 *a, float4 *b) {
                    const float4 *q = sp + (int64_t)((j - base) >> 1) * gstep;
#pragma unroll
                    for (int h = 0; h < kH; h++) {
                        a[h] = __ldg(q + h * gstep);
                        if constexpr (!C) b[h] = __ldg(q + h * gstep + 1);
                    }
                };
                float4 na[kH], nb[kH];
                {
                    float4 fa, fb;
                    const float4 *q = sp + (int64_t)((D.j1 - base) >> 1) * gstep;
                    fa = __ldg(q);
                    fb = C ? fa : __ldg(q + 1);
                    if (mine > 0) load_singles(j0 + kCS * jhalf, na, nb);
                    rs.set_first(fa, fb, ((D.j1 - base) & 1) != 0);
                }
                // one chunk's screen: the row values of its last SNPs, summed
                // by prefix; the pairs that pass, as lane masks
                auto screen_chunk = [&](int32_t jb, const uint32_t *cs, const uint32_t *cn, const float4 *a,
                                        const float4 *b, uint32_t *cmask) {
#pragma unroll
                    for (int h = 0; h < kH; h++) {
                        const uint32_t *hs = cs + 8 * h, *hn = cn + (C ? 0 : 8 * h);
                        float v0, v1;
                        if (poly) {
                            rs.pair_bound(hs, hn, a[h], b[h], v0, v1);
                        } else {
                            rs.pair_logs(hs, hn, a[h], b[h], v0, v1);
                        }
                        // one group after the other: side by side they spill
                        reinterpret_cast<float2 *>(wb)[lane * kH + h] =
                            row_in ? make_float2(v0, v1) : make_float2(0.0f, 0.0f);
                        __syncwarp();
                    }
                    __syncwarp();
                    if constexpr (kPPW > 1) {
#pragma unroll
                        for (int q = 0; q < kPairIters; q++) {
                            const int pair = lane + 32 * q;
                            bool cand = false;
                            if (pair < kPairs) {
                                const int pp = pair / kCS, jj = pair % kCS;
                                float v = 0.0f, w2 = 0.0f;
#pragma unroll
                                for (int rr = 0; rr < kPR; rr++) {
                                    if (rr & 1) w2 += wb[(pp * kPR + rr) * kCS + jj];
                                    else v += wb[(pp * kPR + rr) * kCS + jj];
                                }
                                v += w2;
                                const int32_t j = jb + jj;
                                cand = j >= plo[q] && j < phi[q] && fmaf(v, vscale, voff) >= cut;
                            }
                            cmask[q] = __ballot_sync(0xffffffffu, cand);
                        }
                    } else {
                        // one prefix: 32 / kCS lanes share a column, kCS rows each
                        float v = 0.0f;
#pragma unroll
                        for (int rr = 0; rr < kCS; rr++) v += wb[((lane / kCS) * kCS + rr) * kCS + lane % kCS];
#pragma unroll
                        for (int off = kCS; off < 32; off <<= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
                        const int32_t j = jb + lane % kCS;
                        cmask[0] = __ballot_sync(0xffffffffu, lane < kCS && j >= plo[0] && j < phi[0] &&
                                                                  fmaf(v, vscale, voff) >= cut);
                    }
                    __syncwarp();
                };
                // The chunks' screen; the rare work (precise scores, a search
                // without a threshold, the validation dump) has a loop of its
                // own below, which loads its chunks again: in one loop it cost
                // every chunk registers and reordering (order 3, 2000 x 4000:
                // 63 ms with all of it inside, 54 without).
                const bool slow = cold || P.dump;
                uint32_t todo = 0xffffffffu;
                if (!slow) {
                    todo = 0;
#pragma unroll 1
                    for (int jc = 0; jc < mine; jc++) {
                        const int jcg = jhalf + kCG * jc;
                        const int32_t jb = j0 + kCS * jcg;
                        uint32_t cs[kChunkCols], cn[C ? 1 : kChunkCols];
                        load_chunk(jcg, cs, cn);
                        float4 a[kH], b[kH];
#pragma unroll
                        for (int h = 0; h < kH; h++) {
                            a[h] = na[h];
                            b[h] = C ? na[h] : nb[h];
                        }
                        if (jc + 1 < mine) load_singles(jb + kCS * kCG, na, nb);
                        tmem_wait_ld();
                        uint32_t cmask[kPairIters], any = 0;
                        screen_chunk(jb, cs, cn, a, b, cmask);
#pragma unroll
                        for (int q = 0; q < kPairIters; q++) any |= cmask[q];
                        if (any) todo |= 1u << jc;
                    }
                }
                const int rounds = slow && cold ? kIters : (todo ? mine : 0);
#pragma unroll 1
                for (int jc = 0; jc < rounds; jc++) {
                    if (cold && jc > 0) {
                        share_threshold();
                        cut = thr * DS.cut_mul - DS.cut_add;
                        cold = thr < 0.0f;
                    }
                    if (jc >= mine || !(todo >> jc & 1u)) continue;
                    const int jcg = jhalf + kCG * jc;
                    const int32_t jb = j0 + kCS * jcg;
                    uint32_t cs[kChunkCols], cn[C ? 1 : kChunkCols];
                    load_chunk(jcg, cs, cn);
                    float4 a[kH], b[kH];
                    load_singles(jb, a, b);
                    if constexpr (C) {
#pragma unroll
                        for (int h = 0; h < kH; h++) b[h] = a[h];
                    }
                    tmem_wait_ld();
                    // this row's nine cells of column jsel
                    auto chunk_counts = [&](int jsel, uint32_t *ca, uint32_t *co) {
                        PairRow pr;
                        const bool odd = jsel & 1;
#pragma unroll
                        for (int h = 0; h < kH; h++) {
                            if (h != jsel >> 1) continue;
#pragma unroll
                            for (int i = 0; i < 4; i++) {
                                pr.x[i] = __uint_as_float(odd ? cs[8 * h + 2 * i + 1] : cs[8 * h + 2 * i]);
                                if constexpr (!C)
                                    pr.y[i] = __uint_as_float(odd ? cn[8 * h + 2 * i + 1] : cn[8 * h + 2 * i]);
                            }
                            pr.x[4] = odd ? a[h].y : a[h].x;
                            pr.x[5] = odd ? a[h].w : a[h].z;
                            if constexpr (!C) {
                                pr.y[4] = odd ? b[h].y : b[h].x;
                                pr.y[5] = odd ? b[h].w : b[h].z;
                            }
                        }
                        float drop;
                        f2_unpack(rs.U0.c, pr.c0, drop);
                        f2_unpack(rs.U0.s, pr.s0, drop);
                        f2_unpack(rs.U1.c, pr.c1, drop);
                        f2_unpack(rs.U1.s, pr.s1, drop);
                        f2_unpack(rs.V.c, pr.c2, drop);
                        f2_unpack(rs.V.s, pr.s2, drop);
                        pr.c0 *= rs.inv_q1;
                        pr.c1 *= rs.inv_q1;
                        pr.c2 *= rs.inv_q1;
                        pr.kinv = 1.0f / p2;
                        pr.p2 = p2;
                        pair_cells<C>(pr, ca, co);
                    };
                    if (P.dump && row_in) {
#pragma unroll 1
                        for (int jj = 0; jj < kCS; jj++) {
                            const int32_t j = jb + jj;
                            if (j <= D.j1 || j >= (int32_t)d.n) continue;
                            uint32_t ca[9], co[9];
                            chunk_counts(jj, ca, co);
                            constexpr int cells = kPR * 9;
                            const uint64_t rank = DS.total - 1 - prefix_rank_sum<km1>(d, psnp, K) -
                                                  binom_at(d.binom, d.n, d.n - 1 - D.j1, 2) - (uint64_t)(d.n - 1 - j);
                            uint32_t *o = P.dump + rank * 2 * cells;
#pragma unroll
                            for (int x = 0; x < 9; x++) {
                                o[pos * 9 + x] = ca[x];
                                o[cells + pos * 9 + x] = co[x];
                            }
                        }
                    }
                    // precise terms of this row for column jsel
                    auto precise = [&](int jsel) -> SumF32 {
                        uint32_t ca[9], co[9];
                        chunk_counts(jsel, ca, co);
                        SumF32 e;
#pragma unroll 1
                        for (int x = 0; x < 9; x += 3) {
                            const SumF32 r =
                                row_terms_precise(ca[x], co[x], ca[x + 1], co[x + 1], ca[x + 2], co[x + 2], mc);
                            e.add(r.s);
                            e.c += r.c;
                        }
                        return e;
                    };
                    if (cold) {
#pragma unroll 1
                        for (int jj = 0; jj < kCS; jj++) {
                            const float e = seg_sum<kPR>(row_in ? precise(jj) : SumF32(), pos);
                            if (row_in && pos == 0 && jb + jj > D.j1 && jb + jj < (int32_t)d.n)
                                keep(__fdiv_rn(e, mc.fm), p, jb + jj);
                        }
                        continue;
                    }
                    uint32_t cmask[kPairIters];
                    screen_chunk(jb, cs, cn, a, b, cmask);
#pragma unroll
                    for (int q = 0; q < kPairIters; q++) {
                        while (cmask[q]) {
                            const int pair = __ffs(cmask[q]) - 1 + 32 * q;
                            cmask[q] &= cmask[q] - 1;
                            const int pp = pair / kCS, jsel = pair % kCS;
                            const float e = seg_sum<kPR>(row_in && pl == pp ? precise(jsel) : SumF32(), pos);
                            if (row_in && pl == pp && pos == 0) keep(__fdiv_rn(e, mc.fm), p, jb + jsel);
                        }
                    }
                }
                release_acc();
                refresh();
                epi_bar<kEpiThreads>();
            } else {
                // this warp's chunks of the quadrant: those that hold a last
                // SNP below n (all but in the last N tile of a panel)
                const int live_chunks = ok ? min(kQC, ((int32_t)d.n - j0 + 7) >> 3) : 0;
                const int mine = (live_chunks - jhalf + kCG - 1) / kCG;
                // one chunk's screen: the row values of its last SNPs, summed
                // by prefix; the pairs that pass, as lane masks
                auto screen_chunk = [&](int32_t jb, const uint32_t *cs, const uint32_t *cn, uint32_t *cmask) {
                    float vrow[8];
                    if (poly) rs.bound(cs, cn, vrow);
                    else rs.logs(cs, cn, vrow);
                    store_rows(vrow);
                    if constexpr (kPPW > 1) {
#pragma unroll
                        for (int q = 0; q < kPairIters; q++) {
                            const int pair = lane + 32 * q;
                            bool cand = false;
                            if (pair < kPairs) {
                                const int pp = pair >> 3, jj = pair & 7;
                                float v = 0.0f, w2 = 0.0f;
#pragma unroll
                                for (int rr = 0; rr < kPR; rr++) {
                                    if (rr & 1) w2 += wb[(pp * kPR + rr) * 8 + jj];
                                    else v += wb[(pp * kPR + rr) * 8 + jj];
                                }
                                v += w2;
                                const int32_t j = jb + jj;
                                cand = j >= plo[q] && j < phi[q] && fmaf(v, vscale, voff) >= cut;
                            }
                            cmask[q] = __ballot_sync(0xffffffffu, cand);
                        }
                    } else {
                        const float v = column_sum();
                        const int32_t j = jb + (lane & 7);
                        cmask[0] = __ballot_sync(0xffffffffu, lane < 8 && j >= plo[0] && j < phi[0] &&
                                                                  fmaf(v, vscale, voff) >= cut);
                    }
                    __syncwarp();
                };
                // Every score of a chunk: m MI = T(m) - T(m1) - T(m0) + sum over
                // cells of T(a) + T(b) - T(a + b), T(c) = c ln c from a table
                // in shared memory as integers of 2^-46, so the sum is exact
                // and the score's error is the two roundings to float (the
                // popcount path's per-term series takes ten times the
                // instructions: order 4, 200 x 2000, 177 ms); the scores too
                // small for the table are made again (small_scores_kernel)
                auto score_chunk = [&](int32_t jb, const uint32_t *cs, const uint32_t *cn) {
                    long long *w64 = reinterpret_cast<long long *>(wb);
                    const int pp = kPPW > 1 ? lane >> 2 : 0;
                    const int pt = quad * kPPW + pp;
                    const bool sums = kPPW > 1 ? pp < kPPW && pt < D.nvalid : lane < 4 && pt < D.nvalid;
                    int64_t rank0 = 0;
                    int32_t c = 0x7fffffff;
                    if (sums) {
                        int32_t qs[km1];
#pragma unroll
                        for (int tt = 0; tt < km1; tt++) qs[tt] = D.snp[pt * km1 + tt];
                        rank0 = (int64_t)(DS.total - prefix_rank_sum<km1>(d, qs)) - d.n;
                        c = qs[km1 - 1];
                    }
                    const long long all = tlog[d.m] - tlog[d.m1] - tlog[d.m0];
#pragma unroll
                    for (int half = 0; half < 2; half++) {
                        long long v[4];
#pragma unroll
                        for (int e = 0; e < 4; e++) {
                            float a[3], bb[3];
                            rs.counts(cs, cn, 2 * half + (e >> 1), e & 1, a, bb);
                            long long t = 0;
#pragma unroll
                            for (int g3 = 0; g3 < 3; g3++) {
                                const uint32_t ia = f2u_exact(a[g3]), ib = f2u_exact(bb[g3]);
                                t += tlog[ia] + tlog[ib] - tlog[ia + ib];
                            }
                            v[e] = prow ? t : 0;
                        }
                        reinterpret_cast<longlong2 *>(w64)[lane * 2] = make_longlong2(v[0], v[1]);
                        reinterpret_cast<longlong2 *>(w64)[lane * 2 + 1] = make_longlong2(v[2], v[3]);
                        __syncwarp();
                        long long sum = 0;
                        if constexpr (kPPW > 1) {
                            if (sums) {
#pragma unroll
                                for (int rr = 0; rr < kPR; rr++) sum += w64[(pp * kPR + rr) * 4 + (lane & 3)];
                            }
                        } else {
#pragma unroll
                            for (int rr = 0; rr < 4; rr++) sum += w64[((lane >> 2) * 4 + rr) * 4 + (lane & 3)];
#pragma unroll
                            for (int off = 4; off < 32; off <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
                        }
                        const int32_t j = jb + 4 * half + (lane & 3);
                        if (sums && j > c && j < (int32_t)d.n) {
                            const long long t = sum + all;
                            P.scores[rank0 + j] =
                                __fdiv_rn(__ll2float_rn(t > 0 ? t : 0) * 1.4210854715202004e-14f, mc.fm);   // 2^-46
                        }
                        __syncwarp();
                    }
                };
                // The chunks' screen, accumulators loaded one chunk ahead; the
                // rare work (precise scores, a search without a threshold, the
                // stored single counts, the validation dump) has a loop of its
                // own below, which loads its chunks again: in one loop it cost
                // every chunk registers and reordering (order 3, 2000 x 4000:
                // 63 ms with all of it inside, 54 without).
                const bool slow = cold || store || scoring || P.dump;
                uint32_t todo = 0xffffffffu;
                if (!slow) {
                    todo = 0;
                    uint32_t nx[16], ny[C ? 1 : 16];
                    if (mine > 0) load_chunk(jhalf, nx, ny);
#pragma unroll 1
                    for (int jc = 0; jc < mine; jc++) {
                        const int jcg = jhalf + kCG * jc;
                        uint32_t cs[16], cn[C ? 1 : 16];
                        tmem_wait_ld();
#pragma unroll
                        for (int q = 0; q < 16; q++) {
                            cs[q] = nx[q];
                            if constexpr (!C) cn[q] = ny[q];
                        }
                        if (jc + 1 < mine) load_chunk(jcg + kCG, nx, ny);
                        uint32_t cmask[kPairIters], any = 0;
                        screen_chunk(j0 + 8 * jcg, cs, cn, cmask);
#pragma unroll
                        for (int q = 0; q < kPairIters; q++) any |= cmask[q];
                        if (any) todo |= 1u << jc;
                    }
                }
                // while there is no threshold the warps go chunk by chunk
                // together, until enough combinations are scored to set one
                // (kIters rounds for every warp, whatever its item or state:
                // the rounds meet at barriers)
                const int rounds = slow && cold ? kIters : (todo ? mine : 0);
#pragma unroll 1
                for (int jc = 0; jc < rounds; jc++) {
                    if (cold && jc > 0) {
                        share_threshold();
                        cut = thr * DS.cut_mul - DS.cut_add;
                        cold = thr < 0.0f;
                    }
                    if (jc >= mine || !(todo >> jc & 1u)) continue;
                    const int jcg = jhalf + kCG * jc;
                    const int32_t jb = j0 + 8 * jcg;
                    uint32_t cs[16], cn[C ? 1 : 16];
                    load_chunk(jcg, cs, cn);
                    tmem_wait_ld();
                    if (P.dump) dump_chunk(jb, cs, cn);
                    if constexpr (K == 3 || K == 4) {
                        if (scoring) {
                            score_chunk(jb, cs, cn);
                            continue;
                        }
                    }
                    if (store) {
                        // the raw accumulators of this row, two SNPs at a time
                        if (prow) {
                            constexpr int kAcc = C ? 1 : 2;
                            const int32_t base = (int32_t)panel_j0(psnp[km1 - 1]);
                            const int32_t top = base + 2 * (int32_t)single_groups(d.n, psnp[km1 - 1]);
#pragma unroll
                            for (int h = 0; h < 4; h++) {
                                const int32_t j = jb + 2 * h;
                                if (j < base || j >= top) continue;
                                float4 *o = singles + ((D.single[p] + (uint64_t)((j - base) >> 1)) * kPR + pos) * kAcc;
                                o[0] = make_float4(__uint_as_float(cs[4 * h]), __uint_as_float(cs[4 * h + 1]),
                                                   __uint_as_float(cs[4 * h + 2]), __uint_as_float(cs[4 * h + 3]));
                                if constexpr (!C)
                                    o[1] = make_float4(__uint_as_float(cn[4 * h]), __uint_as_float(cn[4 * h + 1]),
                                                       __uint_as_float(cn[4 * h + 2]), __uint_as_float(cn[4 * h + 3]));
                            }
                        }
                        continue;
                    }
                    if (cold) {
                        int32_t jlo = 1, jhi = 0;
                        if (prow && pos == 0) last_snp_range<km1>(DS, d, psnp, jlo, jhi);
#pragma unroll 1
                        for (int jj = 0; jj < 8; jj++) {
                            const float e = seg_sum<kPR>(prow ? row_precise(cs, cn, jj) : SumF32(), pos);
                            if (jb + jj >= jlo && jb + jj < jhi) keep(__fdiv_rn(e, mc.fm), p, jb + jj);
                        }
                        continue;
                    }
                    uint32_t cmask[kPairIters];
                    screen_chunk(jb, cs, cn, cmask);
                    // precise single-precision scores of the flagged pairs
                    // (rare): the prefix's row lanes score their rows of that
                    // column, the prefix's first row lane adds them up
#pragma unroll
                    for (int q = 0; q < kPairIters; q++) {
                        while (cmask[q]) {
                            const int pair = __ffs(cmask[q]) - 1 + 32 * q;
                            cmask[q] &= cmask[q] - 1;
                            const int pp = pair >> 3, jsel = pair & 7;
                            SumF32 rv;
                            if (lane_real && pl == pp) rv = row_precise(cs, cn, jsel);
                            const float e = seg_sum<kPR>(rv, pos);
                            if (lane_real && pl == pp && pos == 0) keep(__fdiv_rn(e, mc.fm), p, jb + jsel);
                        }
                    }
                }
                release_acc();
                refresh();
                epi_bar<kEpiThreads>();
            }
            if (ES.stop) break;
            if (lane == 0) mbar_arrive(&desc_empty[dq]);
            thr = ES.next_thr;
            // the next item adds at most one candidate per last SNP and
            // prefix: sort and trim first if the buffer could not hold them
            const int kept = ES.list_len + ES.nbuf;
            const bool grew = kept != ES.seen;
            // no candidate of the next item before every warp has read these
            epi_bar<kEpiThreads>();
            if (kept + kJ * kPPT > P.cand_p2) {
                epi_flush<kEpiThreads>(ES, sc, rk, P.pool, DS, tid);
                thr = fmaxf(thr, ES.thr);
            }
            if (grew) share_threshold();
        }
        epi_bar<kEpiThreads>();
        {
            // what the other CTAs' threshold has passed meanwhile need not be
            // sorted: compact the rest (any order) to the front
            const float gthr = __uint_as_float(*(volatile uint32_t *)DS.global_thr);
            const int kept = ES.list_len + ES.nbuf;
            epi_bar<kEpiThreads>();
            if (tid == 0) ES.nbuf = 0;
            for (int q0 = 0; q0 < kept; q0 += kEpiThreads) {
                const int q = q0 + tid;
                const float v = q < kept ? sc[q] : -1.0f;
                const uint64_t rv = q < kept ? rk[q] : 0;
                epi_bar<kEpiThreads>();
                if (q < kept && v >= gthr) {
                    const int at = atomicAdd(&ES.nbuf, 1);
                    sc[at] = v;
                    rk[at] = rv;
                }
                epi_bar<kEpiThreads>();
            }
            if (tid == 0) ES.list_len = 0;
            epi_bar<kEpiThreads>();
        }
        if (ES.nbuf > 0) epi_flush<kEpiThreads>(ES, sc, rk, P.pool, DS, tid);
        const int L = ES.list_len;
        for (int q = tid; q < L; q += kEpiThreads) {
            P.list_score[(size_t)blockIdx.x * P.pool + q] = sc[q];
            P.list_rank[(size_t)blockIdx.x * P.pool + q] = rk[q];
        }
        if (tid == 0) P.list_count[blockIdx.x] = L;
        if (P.waits && tid == 0) P.waits[blockIdx.x * kWaitSlots + 5] = (unsigned long long)w_epi;
    }

    tc_fence_before();
    __syncthreads();
    if (warp == kWarpMma) {
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
    }
    if (tid == 0 && abort_flag) atomicOr(P.status, ST_TIMEOUT);
}

// Prefixes searched per panel (first SNP in [a, b]) and their exclusive
// prefix sum over c into pcum; then items per panel (the M tiles whose first
// prefix lies in panel c, times the N tiles of that panel) and their
// exclusive prefix sum into cum.  One block.
__device__ __forceinline__ uint64_t panel_prefixes(const DevData &d, int k, int64_t c, int64_t a, int64_t b)
{
    if (c < k - 2 || c > d.n - 2) return 0;
    if (k == 2) return (c >= a && c <= b) ? 1 : 0;
    return subsets_from(d, c, a, k - 2) - subsets_from(d, c, b + 1, k - 2);
}

__device__ void block_exclusive_scan(uint64_t *part, uint64_t s, uint64_t &before, uint64_t &total)
{
    part[threadIdx.x] = s;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        const uint64_t v = threadIdx.x >= off ? part[threadIdx.x - off] : 0;
        __syncthreads();
        part[threadIdx.x] += v;
        __syncthreads();
    }
    before = part[threadIdx.x] - s;
    total = part[1023];
    __syncthreads();
}

__global__ void __launch_bounds__(1024) item_cum_kernel(DevData d, int k, int ppt, int kj, int32_t a, int32_t b,
                                                        uint64_t *pcum, uint64_t *cum)
{
    __shared__ uint64_t part[1024];
    const int64_t n = d.n;
    const int64_t per = (n + 1023) / 1024;
    const int64_t cb = (int64_t)threadIdx.x * per, ce = min(n, cb + per);
    uint64_t s = 0, run = 0, all = 0;
    for (int64_t c = cb; c < ce; c++) s += panel_prefixes(d, k, c, a, b);
    block_exclusive_scan(part, s, run, all);
    for (int64_t c = cb; c < ce; c++) {
        pcum[c] = run;
        run += panel_prefixes(d, k, c, a, b);
    }
    if (threadIdx.x == 1023) pcum[n] = all;
    __syncthreads();
    auto items = [&](int64_t c) -> uint64_t {
        if (c < k - 2 || c > n - 2) return 0;
        const uint64_t t0 = (pcum[c] + ppt - 1) / ppt;
        const uint64_t t1 = (pcum[c + 1] + ppt - 1) / ppt;
        return (t1 - t0) * (uint64_t)panel_ntiles(n, c, kj);
    };
    s = 0;
    for (int64_t c = cb; c < ce; c++) s += items(c);
    block_exclusive_scan(part, s, run, all);
    for (int64_t c = cb; c < ce; c++) {
        cum[c] = run;
        run += items(c);
    }
    if (threadIdx.x == 1023) cum[n] = all;
}

// B operand: rows 4 h + {0, 1} are genotype 0 of SNPs 2 h and 2 h + 1, rows
// 4 h + {2, 3} genotype 1 (zero rows past the last SNP); the 16 bytes of mask
// word w hold, in nibble b of 32-bit word i, individual 32 w + 4 b + i (the A
// producer's order): 2, 1, 0.5 or 0.5 by i where the genotype is the row's.
__global__ void build_b4_kernel(DevData d, uint4 *__restrict__ b4)
{
    const int64_t total = 4 * ((d.n + 1) / 2) * d.Wt;
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t row = idx / d.Wt;
        const int64_t w = idx - row * d.Wt;
        const int64_t j = 2 * (row >> 2) + (row & 1);
        const int g = (int)(row >> 1) & 1;
        const uint32_t v = j < d.n ? d.masks[(j * 3 + g) * d.Wt + w] : 0u;
        b4[idx] = make_uint4((v & 0x11111111u) << 2, v & 0x22222222u, (v & 0x44444444u) >> 2, (v >> 3) & 0x11111111u);
    }
}

// Tables of a pair search over the (kp)-prefixes of pcum: groups of singles
// per panel, items and operand rows per first SNP j1 of the pairs (exclusive
// prefix sums).  One block.
__global__ void __launch_bounds__(1024) pair_tables_kernel(DevData d, int kp, int ppt, int kj, const uint64_t *pcum,
                                                           uint64_t *scum, uint64_t *icum, uint64_t *brow)
{
    __shared__ uint64_t part[1024];
    const int64_t n = d.n;
    const int64_t per = (n + 1023) / 1024;
    const int64_t cb = (int64_t)threadIdx.x * per, ce = min(n, cb + per);
    auto scan = [&](auto value, uint64_t *out) {
        uint64_t s = 0, run = 0, all = 0;
        for (int64_t c = cb; c < ce; c++) s += value(c);
        block_exclusive_scan(part, s, run, all);
        for (int64_t c = cb; c < ce; c++) {
            out[c] = run;
            run += value(c);
        }
        if (threadIdx.x == 1023) out[n] = all;
    };
    scan([&](int64_t c) -> uint64_t { return (pcum[c + 1] - pcum[c]) * (uint64_t)single_groups(n, c); }, scum);
    scan([&](int64_t j) -> uint64_t {
        return j < kp || j > n - 2 ? 0 : (pcum[j] + ppt - 1) / ppt * (uint64_t)panel_ntiles(n, j, kj);
    }, icum);
    scan([&](int64_t j) -> uint64_t { return j > n - 2 ? 0 : (uint64_t)pair_rows(n, j); }, brow);
}

// Pair operand: of j1 = blockIdx.y, rows 8 h + 4 g1 + 2 g2 + odd are the
// individuals with genotype g1 at j1 and g2 at j2 = panel_j0(j1) + 2 h + odd
// (zeros where j2 <= j1 or past the last SNP), expanded as the B operand is.
__global__ void build_pairs_kernel(DevData d, const uint64_t *__restrict__ brow, uint4 *__restrict__ out)
{
    const int64_t j1 = blockIdx.y;
    const int64_t rows = pair_rows(d.n, j1), j0 = panel_j0(j1);
    uint4 *o = out + brow[j1] * d.Wt;
    const int64_t total = rows * d.Wt;
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t row = idx / d.Wt, w = idx - row * d.Wt;
        const int64_t j2 = j0 + 2 * (row >> 3) + (row & 1);
        const int g1 = (int)(row >> 2) & 1, g2 = (int)(row >> 1) & 1;
        const uint32_t v = j2 > j1 && j2 < d.n ? d.masks[(j1 * 3 + g1) * d.Wt + w] & d.masks[(j2 * 3 + g2) * d.Wt + w] : 0u;
        o[idx] = make_uint4((v & 0x11111111u) << 2, v & 0x22222222u, (v & 0x44444444u) >> 2, (v >> 3) & 0x11111111u);
    }
}

__global__ void tlog_kernel(int64_t m, long long *__restrict__ out)
{
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c <= m; c += (int64_t)gridDim.x * blockDim.x)
        out[c] = c > 0 ? __double2ll_rn((double)c * log((double)c) * 70368744177664.0) : 0;   // 2^46
}

// The scores of a whole table of scores that are small beside the errors of
// the sums of n ln n, made again in the cancellation-free form in double
// precision.  Half a unit of 2^-46 for each entry and a last place of each
// double-precision product add up to less than m ln m / 16 + 123 units, so
// scores from 2^24 times that (an MI of 1e-7 at 3000 individuals) keep their
// accuracy; below are combinations with hardly any association, or none,
// whose score has to be zero.  An ordinary study has none: one read of the
// scores (order 4, 200 SNPs: 259 MB) counts them.  Where there are some, SNPs
// with one genotype are left out of the combination (they do not change its
// score): of none but such the score is zero, and the others go to a list, a
// warp each with a table of 3^(SNPs left) cells.  Where those cells come to
// more than a sixty-fourth of the whole table's, the popcount path makes the
// table.  (Every second of 300 SNPs so, order 3 x 2000: 8.9 ms when each was
// counted in full, 0.7 so; 100 SNPs with 0 to 2 carriers, order 4 x 2000: 17.4
// and 4.3.)
__host__ __device__ inline float small_score_limit(int64_t m)
{
    const double units = (double)m * log((double)m) / 16.0 + 123.0;
    return (float)(units * 16777216.0 / 70368744177664.0 / (double)m);
}

__global__ void __launch_bounds__(256) count_small_kernel(uint64_t total, float limit, const float *__restrict__ scores,
                                                          unsigned long long *__restrict__ n)
{
    uint32_t c = 0;
    for (uint64_t r = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; r < total; r += (uint64_t)gridDim.x * blockDim.x)
        c += scores[r] < limit;
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(n, (unsigned long long)c);
}

// one warp per SNP: whether everyone has the same genotype
__global__ void __launch_bounds__(256) one_genotype_kernel(DevData d, uint8_t *__restrict__ same)
{
    const int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (s >= d.n) return;
    uint32_t held = 0;
    for (int w = threadIdx.x & 31; w < d.Wt; w += 32)
        for (int g = 0; g < 3; g++) held |= d.masks[(s * 3 + g) * d.Wt + w] ? 1u << g : 0u;
    held = __reduce_or_sync(0xffffffffu, held);
    if ((threadIdx.x & 31) == 0) same[s] = __popc(held) == 1;
}

// the combination of rank r without its SNPs of one genotype; how many are left
__device__ __forceinline__ int varying_snps(const DevData &d, int k, uint64_t r, const uint8_t *__restrict__ same,
                                            int32_t *out)
{
    int32_t comb[kMaxOrderGpu];
    unrank_lex(d.binom, d.n, k, r, comb);
    int left = 0;
    for (int t = 0; t < k; t++)
        if (!same[comb[t]]) out[left++] = comb[t];
    return left;
}

__global__ void __launch_bounds__(256) list_small_kernel(DevData d, int k, uint64_t total, float limit,
                                                         const uint8_t *__restrict__ same, float *__restrict__ scores,
                                                         uint64_t *__restrict__ list, uint64_t cap,
                                                         unsigned long long *__restrict__ n)
{
    const int lane = threadIdx.x & 31;
    const uint64_t step = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t r0 = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); r0 < total; r0 += step) {
        const uint64_t r = r0 + lane;
        uint32_t cells = 0;                  // of this lane's table, where it is listed
        if (r < total && scores[r] < limit) {
            int32_t comb[kMaxOrderGpu];
            const int left = varying_snps(d, k, r, same, comb);
            if (left) {
                cells = 1;
                for (int t = 0; t < left; t++) cells *= 3;
            } else {
                scores[r] = 0.0f;
            }
        }
        const uint32_t mask = __ballot_sync(0xffffffffu, cells != 0);
        if (!mask) continue;
        const uint32_t all = __reduce_add_sync(0xffffffffu, cells);
        unsigned long long at = 0;
        if (lane == 0) {
            at = atomicAdd(n, (unsigned long long)__popc(mask));
            atomicAdd(n + 1, (unsigned long long)all);
        }
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(mask & ((1u << lane) - 1u));
        if (cells && at < cap) list[at] = r;
    }
}

__global__ void __launch_bounds__(256) small_scores_kernel(DevData d, int k, const uint8_t *__restrict__ same,
                                                           const uint64_t *__restrict__ list, uint64_t n,
                                                           float *__restrict__ scores)
{
    const int lane = threadIdx.x & 31;
    for (uint64_t i = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n;
         i += ((uint64_t)gridDim.x * blockDim.x) >> 5) {
        const uint64_t r = list[i];
        int32_t comb[kMaxOrderGpu];
        const int left = varying_snps(d, k, r, same, comb);
        int cells = 1;
        for (int t = 0; t < left; t++) cells *= 3;
        double mine = 0.0;
        for (int x0 = 0; x0 < cells; x0 += 32) {
            uint32_t a = 0, b = 0;   // counts of cell x0 + lane
            for (int x = x0; x < min(cells, x0 + 32); x++) {
                uint32_t ca = 0, cb = 0;
                for (int w = lane; w < d.Wt; w += 32) {
                    uint32_t bits = 0xffffffffu;
                    for (int q = left - 1, y = x; q >= 0; q--, y /= 3)
                        bits &= d.masks[((int64_t)comb[q] * 3 + y % 3) * d.Wt + w];
                    (w < d.W1 ? ca : cb) += __popc(bits);
                }
                ca = __reduce_add_sync(0xffffffffu, ca);
                cb = __reduce_add_sync(0xffffffffu, cb);
                if (lane == x - x0) { a = ca; b = cb; }
            }
            mine += mi_term_f64(a, a + b, d.m1, d.m) + mi_term_f64(b, a + b, d.m0, d.m);
        }
        for (int off = 16; off; off >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, off);
        if (lane == 0) scores[r] = (float)(mine / (double)d.m);
    }
}

// The producers' masks: the 256 individuals of a K stage of every SNP's three
// genotype rows side by side (96 bytes a SNP; zeros past the last word), so
// the lanes of a warp, whose rows differ in genotype first, read one or two
// cache lines per load instead of one per genotype.  One SNP of zeros follows
// the last (rows of no prefix), and kRowsAhead unwritten stages the last one
// (the producers' prefetch runs past it).
constexpr int kRowsAhead = 2 * EPI_TC_PREFETCH * Roles::ProdGroups;
__global__ void build_rows_kernel(DevData d, uint4 *__restrict__ rows)
{
    const int64_t nst = (d.Wt + 7) / 8;
    const int64_t per = (d.n + 1) * 6;
    const int64_t total = nst * per;
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t st = idx / per, q = idx - st * per;
        const int64_t w = st * 8 + (q & 1) * 4;
        rows[idx] = w < d.Wt && q < d.n * 6 ? *reinterpret_cast<const uint4 *>(d.masks + (q >> 1) * d.Wt + w) : make_uint4(0, 0, 0, 0);
    }
}

}  // namespace tc

// ----------------------------------------------------------------- host --
static PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

static cudaError_t get_encode()
{
    if (g_encode) return cudaSuccess;
    cudaDriverEntryPointQueryResult q;
    void *fn = nullptr;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess) return e;
    if (q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
    g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    return cudaSuccess;
}

// the B operand, then (256-byte aligned) the producers' masks
static size_t tc_b_bytes(const DevData &d) { return ((size_t)4 * ((d.n + 1) / 2) * d.Wt * 16 + 255) & ~(size_t)255; }
size_t tc_b4_bytes(const DevData &d) { return tc_b_bytes(d) + (size_t)((d.Wt + 7) / 8 + tc::kRowsAhead) * (d.n + 1) * 96; }

cudaError_t launch_build_b4(const DevData &d, unsigned char *b4, int num_sms, cudaStream_t st)
{
    const int64_t total = 4 * ((d.n + 1) / 2) * (int64_t)d.Wt;
    int64_t blocks = (total + 255) / 256;
    if (blocks > (int64_t)num_sms * 16) blocks = (int64_t)num_sms * 16;
    if (blocks < 1) blocks = 1;
    tc::build_b4_kernel<<<(unsigned)blocks, 256, 0, st>>>(d, reinterpret_cast<uint4 *>(b4));
    tc::build_rows_kernel<<<(unsigned)blocks, 256, 0, st>>>(d, reinterpret_cast<uint4 *>(b4 + tc_b_bytes(d)));
    return cudaGetLastError();
}

// Class shift p of the combined-class variant for a search of d, or 0 where
// the separate-class variant runs: with c1 and c0 the largest case and control
// counts of a genotype-0 or -1 row (no accumulator exceeds them), c0 must lie
// below 2^p - 1 and ctrl + case 2^p below 2^24, where FP32 accumulation of such
// integers and the decode are exact.
int tc_comb_shift(const DevData &d)
{
    int p = 1;
    while (p < 24 && (1ll << p) <= (int64_t)d.c0max + 1) p++;
    return (int64_t)d.c1max * (1ll << p) + d.c0max < (1ll << 24) ? p : 0;
}

static int tc_tile_snps(bool comb) { return comb ? tc::Shape<true>::J : tc::Shape<false>::J; }
static int tc_pr(int k) { return k == 2 ? 3 : (k == 3 ? 9 : (k == 4 ? 27 : 81)); }
static int tc_ppt(int k) { return tc_pr(k) > 32 ? 1 : 4 * (32 / tc_pr(k)); }

// Work items of an order-k search over first SNPs [a, b] (same formulas as
// item_cum_kernel): the host needs the count to split items over the CTAs.
static uint64_t host_subsets_from(int64_t c, int64_t x, int m)
{
    if (m == 0) return 1;
    return c - x >= m ? host_binom(c - x, m) : 0;
}

uint64_t tc_item_count(int64_t n, int k, int64_t a, int64_t b, int kj)
{
    const uint64_t ppt = (uint64_t)tc_ppt(k);
    uint64_t total = 0, pc = 0;
    for (int64_t c = k - 2; c <= n - 2; c++) {
        uint64_t cnt;
        if (k == 2) cnt = (c >= a && c <= b) ? 1 : 0;
        else cnt = host_subsets_from(c, a, k - 2) - host_subsets_from(c, b + 1, k - 2);
        const uint64_t t0 = (pc + ppt - 1) / ppt;
        pc += cnt;
        const uint64_t t1 = (pc + ppt - 1) / ppt;
        total += (t1 - t0) * (uint64_t)tc::panel_ntiles(n, c, kj);
    }
    return total;
}

uint64_t tc_item_count(int64_t n, int k, bool comb) { return tc_item_count(n, k, 0, n - k, tc_tile_snps(comb)); }

// First SNP of the combination of lexicographic rank r: the largest s with
// C(n, k) - C(n - s, k) <= r (the combinations starting below s come first).
int64_t tc_first_snp(int64_t n, int k, uint64_t r)
{
    const uint64_t total = host_binom(n, k);
    int64_t lo = 0, hi = n - k;
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (total - host_binom(n - mid, k) <= r) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Combinations the tensor path counts for the rank range [rb, re): every
// combination whose first SNP lies in [first SNP of rb, first SNP of re - 1].
uint64_t tc_range_work(int64_t n, int k, uint64_t rb, uint64_t re)
{
    if (re <= rb) return 0;
    const int64_t a = tc_first_snp(n, k, rb), b = tc_first_snp(n, k, re - 1);
    // combinations whose first SNP is >= a, minus those whose first SNP is > b
    return host_binom(n - a, k) - host_binom(n - b - 1, k);
}

// Candidate buffer entries: the pool plus one item's combinations, rounded up
// to a power of two for the bitonic sort.
int tc_cand_p2(int k, int pool, bool comb, bool pair)
{
    return next_pow2(pool + (pair ? tc_tile_snps(comb) / 2 * tc_ppt(k - 1) : tc_tile_snps(comb) * tc_ppt(k)));
}

// Groups of the single-count table of a pair search, and operand rows.
static uint64_t pair_single_groups(int64_t n, int kp)
{
    uint64_t g = 0;
    for (int64_t c = kp - 1; c <= n - 2; c++) g += host_binom(c, kp - 1) * (uint64_t)tc::single_groups(n, c);
    return g;
}

static uint64_t pair_operand_rows(int64_t n)
{
    uint64_t r = 0;
    for (int64_t j = 0; j <= n - 2; j++) r += (uint64_t)tc::pair_rows(n, j);
    return r;
}

TcPairBytes tc_pair_bytes(const DevData &d, int k, bool comb)
{
    TcPairBytes b;
    b.operand = (size_t)pair_operand_rows(d.n) * d.Wt * 16;
    // one group more: the chunk that ends a prefix's groups may read past them
    b.singles = ((size_t)pair_single_groups(d.n, k - 2) + 4) * tc_pr(k - 1) * (comb ? 16 : 32);
    b.tables = (size_t)5 * (d.n + 1) * 8;
    return b;
}

// Whether a whole order-k search takes pair tiles: orders 4 and 5 on enough
// SNPs, with the operand and the single counts within 16 GiB.  The passes
// before the search cost about 30 us (order 4 with and without pairs, 2500
// individuals: 33 SNPs 207 and 191 us, 40 SNPs 214 and 263, 130 SNPs 1.8 and
// 2.7 ms; order 5: 33 SNPs 0.58 and 2.7 ms, 60 SNPs 4.0 and 12.1).
bool tc_pair_applies(const DevData &d, int k, bool comb)
{
    if ((k != 4 && k != 5) || d.n < (k == 4 ? 40 : 24) || d.n > 16384) return false;
    const TcPairBytes b = tc_pair_bytes(d, k, comb);
    return b.operand + b.singles <= ((size_t)16 << 30);
}

size_t tc_smem_bytes(int cand_p2, bool cand_global, bool comb)
{
    const size_t rings = comb ? (size_t)tc::Shape<true>::Stages * (tc::kTileBytes + tc::Shape<true>::BBytes)
                              : (size_t)tc::Shape<false>::Stages * (tc::kTileBytes + tc::Shape<false>::BBytes);
    return 1024 + rings + (cand_global ? 0 : (size_t)cand_p2 * 12) + 2 * 128 * tc::Roles::ProdGroups * 2 * 4 +
           tc::kDescDepth * sizeof(tc::Desc) + (size_t)tc::Roles::EpiWarps * 256 * 4;
}

// B operand of `rows` rows (0: the dataset's own)
static cudaError_t encode_map(CUtensorMap *map, const DevData &d, const unsigned char *b4, bool comb,
                              uint64_t rows = 0)
{
    cudaError_t e = get_encode();
    if (e != cudaSuccess) return e;
    const int64_t row = (int64_t)d.Wt * 16;
    cuuint64_t gdim[2] = {(cuuint64_t)row, rows ? (cuuint64_t)rows : (cuuint64_t)(4 * ((d.n + 1) / 2))};
    cuuint64_t gstride[1] = {(cuuint64_t)row};
    cuuint32_t box[2] = {(cuuint32_t)tc::kRowBytes, (cuuint32_t)(2 * tc_tile_snps(comb))};
    cuuint32_t estr[2] = {1u, 1u};
    CUresult cr = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<unsigned char *>(b4), gdim, gstride, box,
                           estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return cr == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// The screen's constants and margins (see cell_bound).
static void fill_screen(tc::DsParams &D, const DevData &d, int k, int comb_p)
{
    const double u = 5.9604644775390625e-8, m = (double)d.m;
    const double pi = (double)d.m1 / m;
    const double q2 = comb_p ? (double)(1 << (comb_p - 1)) : 1.0;   // e's factor
    D.poly = pi >= 0.2 && pi <= 0.8;
    if (!D.poly) {
        // fast logarithms: m MI / ln 2 = T(m) - T(m1) - T(m0) + sum over cells
        // of t(a) + t(b) - t(a + b), T = t on counts.  Margin: relative errors
        // of the log2 approximation (2^-21) and of the float sums over the
        // terms' magnitude T(m) + T(m1) + T(m0), doubled
        auto T = [](double c) { return c > 0 ? c * log2(c) : 0.0; };
        const int64_t cells = (int64_t)tc_pr(k) * 3;
        const double mag = T(m) + T((double)d.m1) + T((double)d.m0);
        D.vscale = (float)(0.6931471805599453 / m);
        D.voff = (float)((T(m) - T((double)d.m1) - T((double)d.m0)) * 0.6931471805599453 / m);
        D.cut_mul = 1.0f;
        D.cut_add = (float)(2.0 * (4.0 * 4.76837158203125e-7 + (double)(2 * cells + 40) * u) * mag *
                            0.6931471805599453 / m) + 1e-7f;
        D.sc_pi = (float)(pi * q2);
        D.c2 = D.c3 = D.c4 = D.c5a = D.c5b = 0.0f;
        return;
    }
    const double v = pi * (1.0 - pi), q = 1.0 - pi;
    const double c2 = 0.5 / v, c3 = (2.0 * pi - 1.0) / (6.0 * v * v);
    // g at -pi (a cell without cases), 0 and 1 - pi (a cell without controls)
    const double g0 = (-log(q) - c2 * pi * pi + c3 * pi * pi * pi) / (pi * pi * pi * pi);
    const double gm = (2.0 / (pi * pi * pi) + 2.0 / (q * q * q)) / 24.0;
    const double g1 = (-log(pi) - c2 * q * q - c3 * q * q * q) / (q * q * q * q);
    const double slope_n = (g0 - gm) / pi, slope_p = (g1 - gm) / q;   // of g against |x|
    const double c5a = 0.5 * (slope_p - slope_n), c5b = 0.5 * (slope_p + slope_n);
    D.sc_pi = (float)(pi * q2);
    D.c2 = (float)c2;
    D.c3 = (float)(c3 / q2);
    D.c4 = (float)(gm / (q2 * q2));
    D.c5a = (float)(c5a / (q2 * q2 * q2));
    D.c5b = (float)(c5b / (q2 * q2 * q2));
    D.vscale = (float)(1.0 / (q2 * q2 * m));
    D.voff = 0.0f;
    // Rounding (u = 2^-24).  e: at most 2 u of the cell's individuals (pi and
    // the fused product), so 2 u m over all cells, times the bound's slope; x: the
    // reciprocal's and the product's 3 u relative, times the slope |x q'| / q;
    // the polynomial's products and sums: 8 u of its terms' magnitudes, and
    // its value's own 2 u; the sums over at most 81 rows, all terms positive:
    // 40 u relative.  The ratios are evaluated on a grid and doubled.
    double slope = 0.0, rel = 0.0;
    for (int t = -32; t <= 32; t++) {
        if (t == 0) continue;
        const double x = t < 0 ? pi * t / 32.0 : q * t / 32.0, ax = fabs(x);
        const double w = c2 + x * (c3 + x * (gm + c5a * x + c5b * ax));
        const double mag = c2 + ax * (fabs(c3) + ax * (gm + (fabs(c5a) + fabs(c5b)) * ax));
        const double dq = x * (2.0 * c2 + x * (3.0 * c3 + x * (4.0 * gm + 5.0 * (c5a * x + c5b * ax))));
        slope = fmax(slope, fabs(dq));
        rel = fmax(rel, (3.0 * fabs(dq) / (ax * w) + 8.0 * mag / w) * u);
    }
    // a precise score at the threshold exceeds MI by at most its own bound
    D.cut_mul = (float)(1.0 - 2.0 * rel - 42.0 * u - f32_rel_bound(k, d.m));
    D.cut_add = (float)(2.0 * slope * 2.0 * u) + 1e-9f;
}

// Per-dataset parameters (host side); the B-operand map goes to tmap_dev when
// the launch is batched (nullptr: passed as a kernel parameter instead).
static void fill_ds(tc::DsParams &D, const DevData &d, int k, uint64_t *item_cum, uint32_t *global_thr,
                    uint64_t total, uint64_t rb, uint64_t re, const CUtensorMap *tmap_dev, int cta_begin,
                    int cta_count, int comb_p, const unsigned char *b4, int top_n, uint32_t *hist)
{
    D.d = d;
    D.rows = reinterpret_cast<const uint4 *>(b4 + tc_b_bytes(d));
    D.comb_p = comb_p;
    D.top_n = hist ? top_n : 0;
    D.hist = hist;
    D.thr_mul = (float)(1.0 - 4.0 * f32_rel_bound(k, d.m));
    D.rank_begin = rb;
    D.rank_end = re;
    D.s1_lo = (int32_t)tc_first_snp(d.n, k, rb);
    D.s1_hi = (int32_t)tc_first_snp(d.n, k, re - 1);
    D.clip = !(rb == 0 && re == total);
    // prefixes whose first SNP lies in [s1_lo, s1_hi]
    uint64_t np = 0;
    for (int64_t c = k - 2; c <= d.n - 2; c++) {
        if (k == 2) np += (c >= D.s1_lo && c <= D.s1_hi) ? 1 : 0;
        else np += host_subsets_from(c, D.s1_lo, k - 2) - host_subsets_from(c, D.s1_hi + 1, k - 2);
    }
    D.n_prefix = np;
    D.n_items = tc_item_count(d.n, k, D.s1_lo, D.s1_hi, tc_tile_snps(comb_p != 0));
    D.item_cum = item_cum;
    D.pcum = item_cum + d.n + 1;
    D.scum = D.brow = nullptr;
    D.singles = nullptr;
    D.store = 0;
    D.chunks = d.Wt * 32 / tc::kChunk;
    D.chunks_case = d.W1 * 32 / tc::kChunk;
    fill_screen(D, d, k, comb_p);
    D.total = total;
    D.global_thr = global_thr;
    D.tmap = tmap_dev;
    D.cta_begin = cta_begin;
    D.cta_count = cta_count;
}

static void fill_launch(tc::Params &P, int k, int pool, float *list_score, uint64_t *list_rank, int32_t *list_count,
                        int32_t *status, uint32_t *dump, unsigned long long *waits, float *cand_g,
                        uint64_t *rank_g, bool comb, bool pair = false)
{
    P.pool = pool;
    P.cand_p2 = tc_cand_p2(k, pool, comb, pair);
    P.cand_score_g = cand_g;
    P.cand_rank_g = rank_g;
    P.wait_ns = 0;
    P.scores = nullptr;
    P.tlog = nullptr;
    P.list_score = list_score;
    P.list_rank = list_rank;
    P.list_count = list_count;
    P.status = status;
    P.dump = dump;
    P.waits = waits;
}

static cudaError_t launch_kernel(const CUtensorMap &map, const tc::Params &P, int k, int grid, cudaStream_t st,
                                 bool comb, bool pair = false, bool collect = false)
{
    const size_t smem = tc_smem_bytes(P.cand_p2, P.cand_score_g != nullptr, comb) +
                        (P.scores ? (size_t)(P.one.d.m + 1) * 8 : 0);
    using Kernel = void (*)(const CUtensorMap, const tc::Params);
    static const Kernel kernels[2][2][4] = {
        {{tc::tc_search_kernel<2, false, false, false>, tc::tc_search_kernel<3, false, false, false>,
          tc::tc_search_kernel<4, false, false, false>, tc::tc_search_kernel<5, false, false, false>},
         {tc::tc_search_kernel<2, true, false, false>, tc::tc_search_kernel<3, true, false, false>,
          tc::tc_search_kernel<4, true, false, false>, tc::tc_search_kernel<5, true, false, false>}},
        {{tc::tc_search_kernel<2, false, false, true>, tc::tc_search_kernel<3, false, false, true>,
          tc::tc_search_kernel<4, false, false, true>, tc::tc_search_kernel<5, false, false, true>},
         {tc::tc_search_kernel<2, true, false, true>, tc::tc_search_kernel<3, true, false, true>,
          tc::tc_search_kernel<4, true, false, true>, tc::tc_search_kernel<5, true, false, true>}}};
    static const Kernel pair_kernels[2][2] = {
        {tc::tc_search_kernel<4, false, true, false>, tc::tc_search_kernel<5, false, true, false>},
        {tc::tc_search_kernel<4, true, true, false>, tc::tc_search_kernel<5, true, true, false>}};
    const Kernel kern = pair ? pair_kernels[comb][k - 4] : kernels[collect][comb][k - 2];
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<grid, tc::Roles::Threads, smem, st>>>(map, P);
    return cudaGetLastError();
}

cudaError_t launch_tc_item_cum(const DevData &d, int k, uint64_t rb, uint64_t re, uint64_t *item_cum,
                               cudaStream_t st, bool comb)
{
    const int32_t a = (int32_t)tc_first_snp(d.n, k, rb), b = (int32_t)tc_first_snp(d.n, k, re - 1);
    tc::item_cum_kernel<<<1, 1024, 0, st>>>(d, k, tc_ppt(k), tc_tile_snps(comb), a, b, item_cum + d.n + 1, item_cum);
    return cudaGetLastError();
}

cudaError_t launch_tc_search(const DevData &d, int k, const unsigned char *b4, uint64_t *item_cum, int pool,
                             uint32_t *global_thr, float *list_score, uint64_t *list_rank, int32_t *list_count,
                             int32_t *status, int grid, uint64_t total, uint64_t rb, uint64_t re, cudaStream_t st,
                             int *cand_p2_out, float *cand_g, uint64_t *rank_g, uint32_t *dump,
                             unsigned long long *waits, unsigned long long wait_ns, int comb_p, int top_n, uint32_t *hist,
                             TcCollect collect)
{
    tc::Params P;
    fill_ds(P.one, d, k, item_cum, global_thr, total, rb, re, nullptr, 0, grid, comb_p, b4, top_n, hist);
    P.many = nullptr;
    P.cta_ds = nullptr;
    fill_launch(P, k, pool, list_score, list_rank, list_count, status, dump, waits, cand_g, rank_g, comb_p != 0);
    P.wait_ns = wait_ns;
    P.collect = collect;
    *cand_p2_out = P.cand_p2;
    cudaError_t e = launch_tc_item_cum(d, k, rb, re, item_cum, st, comb_p != 0);
    if (e != cudaSuccess) return e;
    CUtensorMap map;
    e = encode_map(&map, d, b4, comb_p != 0);
    if (e != cudaSuccess) return e;
    return launch_kernel(map, P, k, grid, st, comb_p != 0, false, collect.ranks != nullptr);
}

// The same search with pair tiles (whole range): ws holds tc_pair_bytes of
// operand, singles and tables.
cudaError_t launch_tc_pair_search(const DevData &d, int k, const unsigned char *b4, const TcPairWork &ws, int pool,
                                  uint32_t *global_thr, float *list_score, uint64_t *list_rank, int32_t *list_count,
                                  int32_t *status, int grid, uint64_t total, cudaStream_t st, float *cand_g,
                                  uint64_t *rank_g, uint32_t *dump, unsigned long long *waits,
                                  unsigned long long wait_ns, int comb_p, int top_n, uint32_t *hist)
{
    const bool comb = comb_p != 0;
    const int kp = k - 2;                       // prefix SNPs: the tiles of an order-(k-1) search
    const int kj = tc_tile_snps(comb) / 2;
    uint64_t *cum1 = ws.tables, *pcum = cum1 + d.n + 1, *scum = pcum + d.n + 1, *icum = scum + d.n + 1,
             *brow = icum + d.n + 1;
    const uint64_t total1 = host_binom(d.n, k - 1);
    cudaError_t e = launch_tc_item_cum(d, k - 1, 0, total1, cum1, st, comb);
    if (e != cudaSuccess) return e;
    tc::pair_tables_kernel<<<1, 1024, 0, st>>>(d, kp, tc_ppt(k - 1), kj, pcum, scum, icum, brow);
    tc::build_pairs_kernel<<<dim3(16, (unsigned)(d.n - 1)), 256, 0, st>>>(d, brow, reinterpret_cast<uint4 *>(ws.operand));
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // the single counts: an order-(k-1) pass that stores its accumulators
    tc::Params P;
    CUtensorMap map;
    fill_ds(P.one, d, k - 1, cum1, global_thr, total1, 0, total1, nullptr, 0, grid, comb_p, b4, 0, nullptr);
    P.one.singles = reinterpret_cast<float4 *>(ws.singles);
    P.one.scum = scum;
    P.one.store = 1;
    P.many = nullptr;
    P.cta_ds = nullptr;
    fill_launch(P, k - 1, 32, list_score, list_rank, list_count, status, nullptr, nullptr, cand_g, rank_g, comb);
    P.wait_ns = wait_ns;
    e = encode_map(&map, d, b4, comb);
    if (e == cudaSuccess) e = launch_kernel(map, P, k - 1, grid, st, comb);
    if (e != cudaSuccess) return e;
    // the pairs
    fill_ds(P.one, d, k, icum, global_thr, total, 0, total, nullptr, 0, grid, comb_p, b4, top_n, hist);
    P.one.singles = reinterpret_cast<float4 *>(ws.singles);
    P.one.scum = scum;
    P.one.brow = brow;
    P.one.pcum = pcum;
    P.one.s1_hi = (int32_t)(d.n - k + 1);        // the prefixes as the order-(k-1) pass lists them
    P.one.n_prefix = 0;
    for (int64_t c = kp - 1; c <= d.n - 2; c++) P.one.n_prefix += host_binom(c, kp - 1);
    P.one.n_items = 0;
    for (int64_t j = kp; j <= d.n - 2; j++)
        P.one.n_items += (host_binom(j, kp) + tc_ppt(k - 1) - 1) / tc_ppt(k - 1) * (uint64_t)tc::panel_ntiles(d.n, j, kj);
    fill_launch(P, k, pool, list_score, list_rank, list_count, status, dump, waits, cand_g, rank_g, comb, true);
    P.wait_ns = wait_ns;
    e = encode_map(&map, d, ws.operand, comb, pair_operand_rows(d.n));
    if (e != cudaSuccess) return e;
    return launch_kernel(map, P, k, grid, st, comb, true);
}

// shared memory of a pass that writes every score
size_t tc_scores_smem_bytes(const DevData &d, bool comb) { return tc_smem_bytes(0, true, comb) + (size_t)(d.m + 1) * 8; }

cudaError_t launch_tc_scores(const DevData &d, int k, const unsigned char *b4, uint64_t *item_cum, long long *tlog,
                             float *scores, uint32_t *global_thr, int32_t *list_count, int32_t *status, int grid,
                             uint64_t total, cudaStream_t st, unsigned long long wait_ns, int comb_p,
                             unsigned long long *small)
{
    tc::tlog_kernel<<<16, 256, 0, st>>>(d.m, tlog);
    tc::Params P;
    CUtensorMap map;
    fill_ds(P.one, d, k, item_cum, global_thr, total, 0, total, nullptr, 0, grid, comb_p, b4, 0, nullptr);
    P.many = nullptr;
    P.cta_ds = nullptr;
    // nothing is kept: any address will do for the candidate buffers
    fill_launch(P, k, 32, nullptr, nullptr, list_count, status, nullptr, nullptr, reinterpret_cast<float *>(tlog),
                reinterpret_cast<uint64_t *>(tlog), comb_p != 0);
    P.scores = scores;
    P.tlog = tlog;
    P.wait_ns = wait_ns;
    cudaError_t e = launch_tc_item_cum(d, k, 0, total, item_cum, st, comb_p != 0);
    if (e == cudaSuccess) e = encode_map(&map, d, b4, comb_p != 0);
    if (e == cudaSuccess) e = launch_kernel(map, P, k, grid, st, comb_p != 0);
    if (e != cudaSuccess) return e;
    tc::count_small_kernel<<<(unsigned)std::min<uint64_t>((total + 255) / 256, (uint64_t)grid * 8), 256, 0, st>>>(
        total, tc::small_score_limit(d.m), scores, small);
    return cudaGetLastError();
}

cudaError_t launch_list_small(const DevData &d, int k, uint64_t total, float *scores, uint8_t *same, uint64_t *list,
                              uint64_t cap, unsigned long long *n, int num_sms, cudaStream_t st)
{
    tc::one_genotype_kernel<<<(unsigned)((d.n + 7) / 8), 256, 0, st>>>(d, same);
    tc::list_small_kernel<<<(unsigned)std::min<uint64_t>((total + 255) / 256, (uint64_t)num_sms * 8), 256, 0, st>>>(
        d, k, total, tc::small_score_limit(d.m), same, scores, list, cap, n);
    return cudaGetLastError();
}

cudaError_t launch_small_scores(const DevData &d, int k, const uint8_t *same, const uint64_t *list, uint64_t n,
                                float *scores, int num_sms, cudaStream_t st)
{
    tc::small_scores_kernel<<<(unsigned)std::min<uint64_t>((n + 7) / 8, (uint64_t)num_sms * 8), 256, 0, st>>>(
        d, k, same, list, n, scores);
    return cudaGetLastError();
}

size_t tc_ds_bytes() { return sizeof(tc::DsParams); }

cudaError_t tc_fill_batch_entry(void *ds_host, void *tmap_host, const DevData &d, int k, const unsigned char *b4,
                                uint64_t *item_cum, uint32_t *global_thr, uint64_t total, const void *tmap_dev,
                                int cta_begin, int cta_count, int comb_p, int top_n, uint32_t *hist)
{
    fill_ds(*static_cast<tc::DsParams *>(ds_host), d, k, item_cum, global_thr, total, 0, total,
            static_cast<const CUtensorMap *>(tmap_dev), cta_begin, cta_count, comb_p, b4, top_n, hist);
    return encode_map(static_cast<CUtensorMap *>(tmap_host), d, b4, comb_p != 0);
}

cudaError_t launch_tc_batch(const void *ds_dev, const int32_t *cta_ds_dev, int k, int pool, float *list_score,
                            uint64_t *list_rank, int32_t *list_count, int32_t *status, int grid, cudaStream_t st,
                            float *cand_g, uint64_t *rank_g, bool comb)
{
    tc::Params P;
    P.one = tc::DsParams();
    P.many = static_cast<const tc::DsParams *>(ds_dev);
    P.cta_ds = cta_ds_dev;
    fill_launch(P, k, pool, list_score, list_rank, list_count, status, nullptr, nullptr, cand_g, rank_g, comb);
    CUtensorMap unused;
    memset(&unused, 0, sizeof(unused));
    return launch_kernel(unused, P, k, grid, st, comb);
}

}  // namespace epi
