// Stage "prep" on the tensor cores (bf16 keys of 64 and 128 dimensions, E4M3 codes of 128): one streaming pass over the candidate keys
// that leaves, per key, r_i = 1 / (||k_i|| + eps), Kbar_i . Kbar_i and the threshold slices, per key tile sum_i r_i k_i, and, while
// the keys are at hand, Eq. 2-3's pooled logits.
//
//   norms     on the CUDA cores, one thread per row, the row read from shared memory once, packed fp32
//   key sums  ONE small product per unit: the key tile as TMA leaves it (rows of 128 d-elements, 128-byte swizzle) is used TRANSPOSED
//             as the A operand (MN-major: M = d, K = the 128 rows), the B operand holds r_i in three bf16 parts (N = 16, rows 0..2),
//             so D[c][0..2] sum to sum_i r_i k_i[c] to fp32 accuracy
//   logits    one product per tile: the tile as the A operand (a key per TMEM lane), the G * alpha query rows of the head as B; the thread
//             that owns a key takes the maximum (or the mean) over the group from its lane
//
// The logits used to be formed by the first scoring pass, beside its own columns of the same product.  That pass is bound by its
// epilogue, this one by HBM with its issue slots idle, and without the query columns three accumulators of the first pass fit (prep and
// first pass, 4096 heads of 4216 tokens: 771 + 994 us, now 891 + 792; 7168 of 2168 with seven query heads: 710 + 934, 761 + 713;
// 8192 of 2168 tokens of 64 dimensions: 546 + 786, 574 + 573; 256 of 1144 no difference).
//
// 64 dimensions: a unit of work is two tiles of a head, one behind the other in the same 32 KB: the two halves of the key sums' M, with
// their r_i as rows 0..2 and 3..5 of the B operand.  Codes: the tile arrives as stored (16 KB) and the thread that owns a row
// widens it into one of the groups' bf16 operand tiles, taking the norm on the way; with `copy` the same tile goes out by a TMA
// store as the head's part of the scoring copy, for the scoring kernels that need one (4096 heads of 4216 tokens: 743 us, 1381 with the
// copy).
//
// The threshold test of Section 3.3, S[j][i] > T, as the sign of k_i . k_j - T / (r_i r_j): the scoring kernels append one K = 16
// step to a tile product whose operands are the slices.  1 / r = ||k|| + eps in three bf16 parts (their sum has fp32 accuracy) as
// (n1, n2, n3, n1, n2, n1, 0 ...) for a key row; its dot product with a row's (-t1, -t1, -t1, -t2, -t2, -t3, 0 ...), the parts of T / r,
// is -T / (r_i r_j) up to terms of size 2^-24.
//
// One persistent block per SM with a contiguous range of the units (head-major), so that a head's queries are fetched once per
// block.  Warp 0 = TMA producer (a ring of up to six tiles: what bounds the kernel is how many bytes an SM has under way); it hands
// each unit's descriptor on with its data.  Warp 1 = issuer of the logits' products and TMEM owner, warp 2 = issuer of the key sums', then
// groups of four warps that take the units in turn: a unit's time is a chain of latencies (landing, norms, product, TMEM loads), which
// four groups overlap (with three 4096 heads of 4216 tokens in 8 bits took 779 us, 743 with four; 8192 of 2168 tokens of 64 dimensions 574,
// 550; with 128 dimensions in bf16, at its bytes, no difference).
#include <algorithm>

#include "rkv_prep.cuh"

namespace rkv {

namespace {

using namespace sm100;

constexpr int kMaxGroups = 4;
constexpr int kGroupWarp0 = 3;
constexpr int kThreads = (kGroupWarp0 + 4 * kMaxGroups) * 32;
constexpr int kBoxBytes = kTile * 64 * 2;                  // one TMA box: 128 rows of 128 bytes
constexpr int kOperandBytes = 2 * kBoxBytes;               // a unit as the tensor cores read it
constexpr int kSumB = 8 * 16 * 32;                         // B operand of the key sums: 8 K-steps x [16 n][16 k] bf16, 32-byte rows (32-byte swizzle)
constexpr int kMaxStages = 8;
constexpr uint32_t kTmemCols = 512;
constexpr int kSmemLimit = 227 * 1024;
// From more units a block on the next kernel is let in when nothing is left to ask for, below by this one's end: the head sums waiting
// beside the last units cost 256 heads of 9 tiles (16 units a block) 123.0 us a call, 121.4 without; 1024 of 2 tiles (14) 124.0, 122.6;
// of 4096 heads of 33 tiles in 8 bits (913) the stage takes 764 us when they come after it, 747 beside it.
constexpr int kManyUnits = 32;

template <int D, bool kCodes>
struct Form {
    static constexpr int kSub = kHeadDim / D;                        // tiles of a unit
    static constexpr int kStageBytes = kCodes ? kBoxBytes : kOperandBytes;
};

enum {
    kBarFull = 0,                            // [kMaxStages] unit landed
    kBarEmpty = kBarFull + kMaxStages,       // [kMaxStages] ... and no longer read (both products; codes: the 4 warps that widened it)
    kBarQFull = kBarEmpty + kMaxStages,      // [kMaxStages] a head's queries landed (choose_plan says how many of them are used)
    kBarQEmpty = kBarQFull + kMaxStages,     // [kMaxStages] ... no longer read
    kBarReady = kBarQEmpty + kMaxStages,     // [kMaxGroups] r_i (codes: and the operand tile) written by the group's 4 warps
    kBarLogits = kBarReady + kMaxGroups,     // [kMaxGroups] logits in TMEM
    kBarSums = kBarLogits + kMaxGroups,      // [kMaxGroups] key sums in TMEM
    kBarTaken = kBarSums + kMaxGroups,       // [kMaxGroups] both taken out (4 warps)
    kBarStored = kBarTaken + kMaxGroups,     // [kMaxGroups] copy: the operand tile has been read by its store
    kBarDrain = kBarStored + kMaxGroups,
    kNumBars
};

// How a block's shared memory is cut up.
struct Plan {
    int stages, q_bytes, off_own, off_q, off_sum, off_bar, off_units, off_misc, total;
};
template <int D, bool kCodes>
__host__ __device__ inline Plan make_plan(int q_rows_pad, int groups, int q_bufs)
{
    Plan pl;
    pl.q_bytes = q_rows_pad * D * 2;
    const int own = kCodes ? groups * kOperandBytes : 0;
    const int fixed = own + q_bufs * pl.q_bytes + groups * kSumB + kNumBars * 8 + 16 + (kMaxStages + kMaxGroups) * 16 + 32 + 1024;      // + alignment slack
    const int stages = (kSmemLimit - fixed) / Form<D, kCodes>::kStageBytes;
    pl.stages = stages > kMaxStages ? kMaxStages : stages;
    pl.off_own = pl.stages * Form<D, kCodes>::kStageBytes;
    pl.off_q = pl.off_own + own;
    pl.off_sum = pl.off_q + q_bufs * pl.q_bytes;
    pl.off_bar = pl.off_sum + groups * kSumB;
    pl.off_units = pl.off_bar + (kNumBars * 8 + 15) / 16 * 16;
    pl.off_misc = pl.off_units + (kMaxStages + kMaxGroups) * 16;
    pl.total = pl.off_misc + 32 + 1024;
    return pl;
}
// The groups: as many as have room for their accumulators (64 dimensions: three from 64 query rows on, two from 80), and no more than there
// are stages.  A group waits for unit k by the parity of its stage's phase, which is exact once the unit before in that stage, k -
// stages, has landed; what a group knows to have landed is everything up to its own unit before, k - groups (its key sums were
// issued in order).
//
// The rings: q_bufs heads' queries and so many units as fit beside them.  A unit can be asked for once its head's queries can, that is
// when the head q_bufs before it is done with: of heads of u units (q_bufs - 1) u + 1 units can be under way, and no more than there are
// stages.  The plan is the one with the most units under way, the fewest query blocks among those.
template <int D, bool kCodes>
void choose_plan(int q_rows_pad, int units_per_head, int *groups, int *q_bufs)
{
    int best = 0;
    *groups = 1 + std::min(kMaxGroups, (int)kTmemCols / (16 + Form<D, kCodes>::kSub * q_rows_pad));
    while (best == 0) {
        --*groups;
        for (int n = 2; n <= kMaxStages; ++n) {
            const int stages = make_plan<D, kCodes>(q_rows_pad, *groups, n).stages;
            const int under_way = std::min(stages, q_rows_pad ? (n - 1) * units_per_head + 1 : stages);
            if ((stages >= *groups || *groups == 1) && under_way > best) best = under_way, *q_bufs = n;
        }
    }
}

// One unit of the work list: which head-problem, which tiles, how many candidate rows from its first tile on.
struct PrepUnit {
    int head, tile, n, rows_here;
};

// kSub: tiles of a unit.  With write_meta the length is recorded, and reported where it is invalid.
template <int kSub>
__device__ __forceinline__ PrepUnit prep_unit_at(const Params &p, int idx, bool write_meta)
{
    PrepUnit w;
    const int units = (p.tiles + kSub - 1) / kSub;
    w.tile = idx % units * kSub;
    w.head = idx / units;                 // head-problem index b * hkv + h
    const int b = w.head / p.hkv;
    int L = p.seq_lens[b];
    int budget_b = p.budgets ? p.budgets[b] : p.budget;             // Section 4.2's per-sequence (ratio) budgets
    if (L < 0 || L > p.cap || budget_b <= p.alpha || budget_b > p.budget) {
        if (write_meta) report(p.status, RKV_ERR_INVALID_ARG);
        L = kMetaInvalid;
        budget_b = p.budget;
    }
    if (write_meta && w.tile == 0 && w.head % p.hkv == 0) {
        p.meta[b] = L;
        p.meta[p.batch + b] = budget_b;
    }
    w.n = candidates_from_meta(L, budget_b, p.alpha);
    w.rows_here = min(max(w.n - w.tile * kTile, 0), kSub * kTile);
    return w;
}

// Where the lengths are recorded and the counters cleared ahead of the prep kernel (Params::lengths_done).
constexpr int kLengthThreads = 256;
__global__ void __launch_bounds__(kLengthThreads) lengths_kernel(Params p)
{
    pdl_trigger();
    pdl_wait();
    clear_counters(p);
    const int b = blockIdx.x * kLengthThreads + threadIdx.x;
    if (b < p.batch) prep_unit_at<1>(p, b * p.hkv * p.tiles, true);
}

// sum_i r_i k_i of a unit: the eight K = 16 steps of D[c][nn] = sum_i K[i][c] R[nn][i], the key rows as an MN-major operand.
// A: 64-element (128-byte) atoms along M 16 KB apart (the second box), 8-row groups along K 1 KB apart, 16 rows of 128 bytes per
// step.  B: 32-byte rows, 8-row groups 256 bytes apart, 32-byte swizzle, 512 bytes per step.
__device__ __forceinline__ void umma_sums(uint32_t d_tmem, uint32_t a_addr, uint32_t b_addr, uint32_t idesc)
{
    const uint32_t a_lo = ((a_addr & 0x3FFFFu) >> 4) | ((16384u >> 4) << 16), a_hi = (1024u >> 4) | (1u << 14) | (2u << 29);
    const uint32_t b_lo = ((b_addr & 0x3FFFFu) >> 4) | (1u << 16), b_hi = (256u >> 4) | (1u << 14) | (6u << 29);
#pragma unroll
    for (int ks = 0; ks < 8; ++ks)
        asm volatile(
            "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
            "setp.ne.b32 p, %6, 0;\n\t"
            "mov.b64 da, {%1, %2};\n\tmov.b64 db, {%3, %4};\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n\t}"
            ::"r"(d_tmem), "r"(a_lo + 128u * ks), "r"(a_hi), "r"(b_lo + 32u * ks), "r"(b_hi), "r"(idesc), "r"(ks)
            : "memory");
}

// The threshold slices of row lr of key tile `tile` (what they are for: see above): 1 / r as
// (n1, n2, n3, n1, n2, n1, 0 ...), and for the head's last key tile -T / r as (-t1, -t1, -t1, -t2, -t2, -t3, 0 ...).
__device__ __forceinline__ void write_slices(const Params &p, int head, int tile, int lr, int n, float r)
{
    auto split3 = [](float rest, uint32_t (&part)[3]) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const __nv_bfloat16 h16 = __float2bfloat16_rn(rest);
            part[c] = (uint32_t)__bfloat16_as_ushort(h16);
            rest -= __bfloat162float(h16);
        }
    };
    uint32_t part[3];
    split3(r > 0.f ? __fdiv_rn(1.0f, r) : 0.f, part);
    uint4 *dst = reinterpret_cast<uint4 *>(p.norm_split + ((size_t)head * p.cap_pad + tile * kTile + lr) * sm100::kSliceElems);
    dst[0] = make_uint4(part[0] | (part[1] << 16), part[2] | (part[0] << 16), part[1] | (part[0] << 16), 0u);
    if (tile != (n + kTile - 1) / kTile - 1) return;
    split3(r > 0.f ? -__fdiv_rn(p.sim_threshold, r) : 0.f, part);
    uint4 *thr = reinterpret_cast<uint4 *>(p.thr_split + ((size_t)head * kTile + lr) * sm100::kSliceElems);
    thr[0] = make_uint4(part[0] | (part[0] << 16), part[0] | (part[1] << 16), part[1] | (part[2] << 16), 0u);
}

// widen16, and the squares of the values onto four packed sums
__device__ __forceinline__ void widen16_squares(const uint4 &codes, uint4 *lo, uint4 *hi, float2 (&sq2)[4])
{
    const uint32_t w[4] = {codes.x, codes.y, codes.z, codes.w};
    uint32_t out[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const __half2_raw pair = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)((w[q >> 1] >> (16 * (q & 1))) & 0xFFFFu), __NV_E4M3);
        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&pair));
        sq2[q & 3] = __ffma2_rn(f, f, sq2[q & 3]);
        const __nv_bfloat162 b2 = __floats2bfloat162_rn(f.x, f.y);
        out[q] = *reinterpret_cast<const uint32_t *>(&b2);
    }
    *lo = make_uint4(out[0], out[1], out[2], out[3]);
    *hi = make_uint4(out[4], out[5], out[6], out[7]);
}

// pool_logits for other window lengths than eight, a column per load ...
__device__ __forceinline__ void pool_columns(uint32_t qbase, bool row_ok, float *logits, int G, int alpha, int cap_pad, bool mean, float scale)
{
    const float kInf = __int_as_float(0x7f800000);
    for (int j = 0; j < alpha; ++j) {
        float best = -kInf, sum = 0.f;
        for (int g0 = 0; g0 < G; g0 += 4) {
            uint32_t tq[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) tmem_ld1(qbase + min(g0 + u, G - 1) * alpha + j, tq[u]);
            asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(tq[0]), "+r"(tq[1]), "+r"(tq[2]), "+r"(tq[3]) :: "memory");
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                best = fmaxf(best, __uint_as_float(tq[u]));
                sum += (g0 + u < G) ? __uint_as_float(tq[u]) : 0.f;
            }
        }
        if (row_ok) logits[(size_t)j * cap_pad] = mean ? sum * scale / (float)G : best * scale;
    }
}
// ... and four where the length is a multiple of that (808 sequences of 1564 tokens, window 12: the stage 204 us, 153; 3380 of 777 tokens of 64
// dimensions 208, 163).  A function of its own, not inlined: beside the code for windows of eight it cost that 5 %.  (Codes, whose
// kernel is short of registers, take single columns: the call alone cost them 738 -> 783 us.)
__device__ __noinline__ void pool_any_window(uint32_t qbase, bool row_ok, float *logits, int G, int alpha, int cap_pad, bool mean, float scale)
{
    const float kInf = __int_as_float(0x7f800000);
    if (alpha % 4 == 0) {                           // four positions of four query heads per round trip
        for (int j0 = 0; j0 < alpha; j0 += 4) {
            float best[4], sum[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) best[j] = -kInf, sum[j] = 0.f;
            for (int g0 = 0; g0 < G; g0 += 4) {
                uint32_t t[4][4];
#pragma unroll
                for (int u = 0; u < 4; ++u) tmem_ld4(qbase + min(g0 + u, G - 1) * alpha + j0, t[u]);
#pragma unroll
                for (int u = 0; u < 4; ++u) tmem_wait4(t[u]);
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        best[j] = fmaxf(best[j], __uint_as_float(t[u][j]));
                        sum[j] += (g0 + u < G) ? __uint_as_float(t[u][j]) : 0.f;
                    }
            }
            if (row_ok)
#pragma unroll
                for (int j = 0; j < 4; ++j) logits[(size_t)(j0 + j) * cap_pad] = mean ? sum[j] * scale / (float)G : best[j] * scale;
        }
        return;
    }
    pool_columns(qbase, row_ok, logits, G, alpha, cap_pad, mean, scale);
}

// Eq. 2-3 for one key from its accumulator row at `qbase` (G groups of alpha columns): the pooled logits into logits[j * cap_pad].
template <bool kCodes>
__device__ __forceinline__ void pool_logits(const Params &p, uint32_t qbase, bool row_ok, float *logits)
{
    const float kInf = __int_as_float(0x7f800000), scale = p.logit_scale;            // 1 / sqrt(d)
    const int G = p.group;
    if (p.alpha == 8) {
        float pooled[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) pooled[j] = p.gqa_mean_pool ? 0.f : -kInf;
        for (int g0 = 0; g0 < G; g0 += 4) {           // four query heads per round trip to TMEM
            uint32_t t0[8], t1[8], t2[8], t3[8];
            tmem_ld8(qbase + g0 * 8, t0);
            tmem_ld8(qbase + min(g0 + 1, G - 1) * 8, t1);         // heads beyond the group re-read its last one
            tmem_ld8(qbase + min(g0 + 2, G - 1) * 8, t2);
            tmem_ld8(qbase + min(g0 + 3, G - 1) * 8, t3);
            tmem_wait8(t0);
            tmem_wait8(t1);
            tmem_wait8(t2);
            tmem_wait8(t3);
            if (p.gqa_mean_pool) {                    // the variant: sum over the group (scaled to the mean below)
                const bool h1 = g0 + 1 < G, h2 = g0 + 2 < G, h3 = g0 + 3 < G;
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    pooled[j] += (__uint_as_float(t0[j]) + (h1 ? __uint_as_float(t1[j]) : 0.f)) +
                                 ((h2 ? __uint_as_float(t2[j]) : 0.f) + (h3 ? __uint_as_float(t3[j]) : 0.f));
                continue;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j)
                pooled[j] = fmaxf(fmaxf(pooled[j], __uint_as_float(t0[j])),
                                  max3(__uint_as_float(t1[j]), __uint_as_float(t2[j]), __uint_as_float(t3[j])));
        }
        const float scale_q = p.gqa_mean_pool ? scale / (float)G : scale;
        if (row_ok)
#pragma unroll
            for (int j = 0; j < 8; ++j) logits[(size_t)j * p.cap_pad] = pooled[j] * scale_q;
        return;
    }
    if (kCodes) pool_columns(qbase, row_ok, logits, G, p.alpha, p.cap_pad, p.gqa_mean_pool != 0, scale);
    else pool_any_window(qbase, row_ok, logits, G, p.alpha, p.cap_pad, p.gqa_mean_pool != 0, scale);
}

// map_k: the stored keys.  map_wide, copy: see above.  table: the block table of the stored keys.  q_rows_pad: 0 where another kernel forms the
// logits.  groups, q_bufs: see choose_plan.
template <int D, bool kCodes>
__global__ void __launch_bounds__(kThreads, 1)
prep_sm100_kernel(Params p, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_q,
                  const __grid_constant__ CUtensorMap map_wide, const int32_t *table, int copy, int total, int q_rows_pad, int groups, int q_bufs)
{
    using F = Form<D, kCodes>;
    constexpr int kSub = F::kSub;
    constexpr int kChunks = D / 8;                           // 16-byte vectors of a bf16 row
    extern __shared__ uint8_t prep_raw[];
    uint8_t *smem = align_smem(prep_raw);
    const uint32_t sbase = smem_u32(smem);
    const Plan pl = make_plan<D, kCodes>(q_rows_pad, groups, q_bufs);
    const uint32_t stages = (uint32_t)pl.stages;
    int *misc = reinterpret_cast<int *>(smem + pl.off_misc);           // TMEM base, abort flag, units and query blocks asked for
    volatile int *abort_flag = misc + 1;
    // descriptors {head, first tile, n, candidate rows from that tile on}: of the units in the ring, and of those that the groups work on
    int4 *unit_at = reinterpret_cast<int4 *>(smem + pl.off_units), *group_unit = unit_at + kMaxStages;
    auto bar = [&](int i) -> uint32_t { return sbase + pl.off_bar + 8u * (uint32_t)i; };
    const ErrSink sink = prep_sink(p);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int first = (int)((long long)blockIdx.x * total / gridDim.x), units = (int)((long long)(blockIdx.x + 1) * total / gridDim.x) - first;
    const uint32_t group_cols = 16u + (uint32_t)(kSub * q_rows_pad);   // TMEM columns of a group: key sums, then logits

    if (threadIdx.x == 0) {
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(bar(kBarFull + s), 1);
            mbar_init(bar(kBarEmpty + s), kCodes ? 4 : 2);
            mbar_init(bar(kBarQFull + s), 1);
            mbar_init(bar(kBarQEmpty + s), 1);
        }
        for (int s = 0; s < kMaxGroups; ++s) {
            mbar_init(bar(kBarReady + s), 4);
            mbar_init(bar(kBarLogits + s), 1);
            mbar_init(bar(kBarSums + s), 1);
            mbar_init(bar(kBarTaken + s), 4);
            mbar_init(bar(kBarStored + s), 1);
        }
        mbar_init(bar(kBarDrain), 2);
        misc[1] = misc[2] = misc[3] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        prefetch_map(&map_k);
        if (q_rows_pad) prefetch_map(&map_q);
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(misc)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // rows 3 kSub..15 of the key sums' B operands stay zero; the others are rewritten in full for every unit
    for (int x = threadIdx.x; x < groups * kSumB / 16; x += kThreads) reinterpret_cast<uint4 *>(smem + pl.off_sum)[x] = make_uint4(0u, 0u, 0u, 0u);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(misc);
    pdl_wait();                             // the set-up above touches no global memory
    if (!p.lengths_done) clear_counters(p);

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0) {
            auto row0 = [&](int head, int tile) -> int {
                return table ? table[(size_t)head * (p.cap / kTile) + tile] * kTile : head * p.cap + tile * kTile;
            };
            int q_head = -1, qn = 0, qb = 0, q_phase = 1, k = 0, seq = -1;
            PrepUnit w = prep_unit_at<kSub>(p, first, false);
            for (; k < units; ++k) {
                const uint32_t s = (uint32_t)k % stages, full = bar(kBarFull + s);
                if (k > 0) {
                    w.tile += kSub;
                    if (w.tile >= p.tiles) {
                        w.tile = 0;
                        ++w.head;
                    }
                }
                if (w.head / p.hkv != seq) {                  // another sequence: its length
                    seq = w.head / p.hkv;
                    w.n = prep_unit_at<kSub>(p, first + k, !p.lengths_done).n;
                }
                w.rows_here = min(max(w.n - w.tile * kTile, 0), kSub * kTile);
                if (!mbar_wait(bar(kBarEmpty + s), (((uint32_t)k / stages) & 1u) ^ 1u, abort_flag, sink)) break;
                unit_at[s] = make_int4(w.head, w.tile, w.n, w.rows_here);
                if (w.rows_here <= 0) {                       // the phase completes without a copy
                    mbar_arrive(full);
                    continue;
                }
                const bool both = kSub == 1 || w.rows_here > kTile;
                const uint32_t dst = sbase + s * F::kStageBytes;
                const int y = row0(w.head, w.tile);
                mbar_expect_tx(full, both ? F::kStageBytes : F::kStageBytes / 2);
                tma_load_2d(dst, &map_k, 0, y, full);
                if (D == 128 && !kCodes) tma_load_2d(dst + kBoxBytes, &map_k, 64, y, full);
                if (kSub == 2 && both) tma_load_2d(dst + kBoxBytes, &map_k, 0, row0(w.head, w.tile + 1), full);
                if (q_rows_pad && w.head != q_head) {         // (the keys first: they do not wait for a query block to come free)
                    if (!mbar_wait(bar(kBarQEmpty + qb), (uint32_t)q_phase, abort_flag, sink)) {
                        ++k;                                  // the unit's keys are under way
                        break;
                    }
                    const uint32_t q_full = bar(kBarQFull + qb), q_dst = sbase + pl.off_q + qb * pl.q_bytes;
                    const int q_row = (w.head / p.hkv * p.hq + w.head % p.hkv * p.group) * p.alpha;
                    mbar_expect_tx(q_full, (uint32_t)pl.q_bytes);
#pragma unroll
                    for (int x = 0; x < D / 64; ++x) tma_load_2d(q_dst + x * q_rows_pad * 128, &map_q, x * 64, q_row, q_full);
                    q_head = w.head;
                    ++qn;
                    if (++qb == q_bufs) qb = 0, q_phase ^= 1;
                }
            }
            misc[2] = k;
            misc[3] = qn;
            if (units > kManyUnits) pdl_trigger();
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------------------ products for the logits
        if (lane == 0) {
            const uint32_t idesc_q = instr_desc(kTile, q_rows_pad);
            int q_head = -1, q_next = 0, q_phase = 0, g = 0;
            uint32_t turn = 0, s = 0, round = 0, q_bar = 0, q = 0;
            for (int k = 0; k < units; ++k) {
                if (!(kCodes ? mbar_wait(bar(kBarReady + g), turn & 1u, abort_flag, sink) : mbar_wait(bar(kBarFull + s), round & 1u, abort_flag, sink))) break;
                const int4 w = kCodes ? group_unit[g] : unit_at[s];
                if (!mbar_wait(bar(kBarTaken + g), (turn & 1u) ^ 1u, abort_flag, sink)) break;
                if (!q_rows_pad || w.w <= 0) {
                    mbar_arrive(bar(kBarLogits + g));
                    if (!kCodes) mbar_arrive(bar(kBarEmpty + s));
                } else {
                    if (w.x != q_head) {
                        if (!mbar_wait(bar(kBarQFull + q_next), (uint32_t)q_phase, abort_flag, sink)) break;
                        q_head = w.x;
                        q_bar = bar(kBarQEmpty + q_next);
                        q = sbase + pl.off_q + q_next * pl.q_bytes;
                        if (++q_next == q_bufs) q_next = 0, q_phase ^= 1;
                    }
                    tc_fence_after();
                    const uint32_t tile = kCodes ? sbase + pl.off_own + g * kOperandBytes : sbase + s * F::kStageBytes;
                    const uint32_t d_tmem = tmem + g * group_cols + 16u;
                    if (D == 64) {
                        umma_tile_k64(d_tmem, tile, q, idesc_q);
                        if (w.w > kTile) umma_tile_k64(d_tmem + (uint32_t)q_rows_pad, tile + kBoxBytes, q, idesc_q);
                    } else {
                        umma_tile_k128_halves(d_tmem, tile, kBoxBytes, q, (uint32_t)q_rows_pad * 128, idesc_q);
                    }
                    umma_commit(bar(kBarLogits + g));
                    if (!kCodes) umma_commit(bar(kBarEmpty + s));
                    if ((w.y + kSub) * kTile >= w.z) umma_commit(q_bar);         // the head's last candidates
                }
                if (++g == groups) g = 0, ++turn;
                if (++s == stages) s = 0, ++round;
            }
        }
        __syncwarp();
    } else if (warp == 2) {
        // ------------------------------------------------------------------ products for the key sums
        if (lane == 0) {
            // f32 accumulate, bf16 x bf16, A MN-major (bit 15), B K-major, M = 128, N = 16
            const uint32_t idesc_s = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | ((16u >> 3) << 17) | ((128u >> 4) << 24);
            int g = 0;
            uint32_t turn = 0, s = 0;
            for (int k = 0; k < units; ++k) {
                if (!mbar_wait(bar(kBarReady + g), turn & 1u, abort_flag, sink)) break;
                const int4 w = group_unit[g];
                const uint32_t tile = kCodes ? sbase + pl.off_own + g * kOperandBytes : sbase + s * F::kStageBytes;
                if (w.w <= 0) {
                    mbar_arrive(bar(kBarSums + g));
                    if (!kCodes) mbar_arrive(bar(kBarEmpty + s));
                } else {
                    tc_fence_after();
                    umma_sums(tmem + g * group_cols, tile, sbase + pl.off_sum + g * kSumB, idesc_s);
                    umma_commit(bar(kBarSums + g));
                    if (!kCodes) umma_commit(bar(kBarEmpty + s));
                    if (kCodes && copy) {
                        // the tile, as the head's rows [128 tile, 128 tile + 128) of the scoring copy (contiguous, head after head)
                        const int yw = w.x * p.cap + w.y * kTile;
#pragma unroll
                        for (int x = 0; x < 2; ++x)
                            asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                                         ::"l"(reinterpret_cast<uint64_t>(&map_wide)), "r"(64 * x), "r"(yw), "r"(tile + x * kBoxBytes) : "memory");
                    }
                }
                if (kCodes && copy) {
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");      // one group per unit, empty or not
                    asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    if (k > 0) mbar_arrive(bar(kBarStored + (g == 0 ? groups : g) - 1));
                }
                if (++g == groups) g = 0, ++turn;
                if (++s == stages) s = 0;
            }
            if (kCodes && copy) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");      // the stores are through before the block leaves
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------------ groups: a thread per row, later per dimension
        const int g = (warp - kGroupWarp0) >> 2, quad = warp & 3, rt = quad * 32 + lane;
        const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16) + g * group_cols;
        uint8_t *bop = smem + pl.off_sum + g * kSumB;
        for (int k = g; g < groups && k < units; k += groups) {
            const uint32_t s = (uint32_t)k % stages, turn = (uint32_t)(k / groups);
            bool ok = mbar_wait(bar(kBarFull + s), ((uint32_t)k / stages) & 1u, abort_flag, sink);
            if (kCodes && copy && ok) ok = mbar_wait(bar(kBarStored + g), (turn & 1u) ^ 1u, abort_flag, sink);
            if (!__all_sync(0xffffffffu, ok)) break;
            const int4 desc = unit_at[s];
            const PrepUnit w{desc.x, desc.y, desc.z, desc.w};
            if (rt == 0) group_unit[g] = desc;
            // ---- norms; rows that are not candidates are cleared for the key sums (they may hold anything, and 0 x NaN would spoil them; a
            // row's logits are its own)
            float r[kSub], sq[kSub];
#pragma unroll
            for (int u = 0; u < kSub; ++u) {
                r[u] = sq[u] = 0.f;
                if (w.rows_here <= 0) continue;
                const bool row_ok = u * kTile + rt < w.rows_here;
                float2 sq2[4];                       // four independent chains of packed multiply-adds
#pragma unroll
                for (int e = 0; e < 4; ++e) sq2[e] = make_float2(0.f, 0.f);
                [[maybe_unused]] auto add = [&](const uint4 &vec) {
                    float f[8];
                    Elem<__nv_bfloat16>::unpack(vec, f);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 f2 = make_float2(f[2 * e], f[2 * e + 1]);
                        sq2[e] = __ffma2_rn(f2, f2, sq2[e]);
                    }
                };
                if constexpr (kCodes) {
                    const uint8_t *raw = smem + s * F::kStageBytes + rt * 128;
                    uint4 in[8];
#pragma unroll
                    for (int c = 0; c < 8; ++c) in[c] = row_ok ? *reinterpret_cast<const uint4 *>(raw + ((c ^ (rt & 7)) << 4)) : make_uint4(0u, 0u, 0u, 0u);
                    uint8_t *row_smem = smem + pl.off_own + g * kOperandBytes + rt * 128;
#pragma unroll
                    for (int c = 0; c < 8; ++c) {            // 16 codes -> bf16 chunks 2 c, 2 c + 1, the squares on the way
                        uint4 lo, hi;
                        widen16_squares(in[c], &lo, &hi, sq2);
                        uint8_t *half = row_smem + (c >> 2) * kBoxBytes;
                        *reinterpret_cast<uint4 *>(half + ((((2 * c) & 7) ^ (rt & 7)) << 4)) = lo;
                        *reinterpret_cast<uint4 *>(half + ((((2 * c + 1) & 7) ^ (rt & 7)) << 4)) = hi;
                    }
                } else {
                    // chunk c of the row: the first box, or with 128 dimensions the second as well
                    uint8_t *row_smem = smem + s * F::kStageBytes + u * kBoxBytes + rt * 128;
                    if (row_ok) {
#pragma unroll
                        for (int c = 0; c < kChunks; ++c)
                            add(*reinterpret_cast<const uint4 *>(row_smem + (c >> 3) * kBoxBytes + (((c & 7) ^ (rt & 7)) << 4)));
                    } else {
#pragma unroll
                        for (int c = 0; c < kChunks; ++c)
                            *reinterpret_cast<uint4 *>(row_smem + (c >> 3) * kBoxBytes + ((c & 7) << 4)) = make_uint4(0u, 0u, 0u, 0u);
                    }
                }
                if (row_ok) {
                    sq[u] = ((sq2[0].x + sq2[0].y) + (sq2[1].x + sq2[1].y)) + ((sq2[2].x + sq2[2].y) + (sq2[3].x + sq2[3].y));
                    const float nrm = sq[u] > 0.f ? sq[u] * rsqrtf(sq[u]) : 0.f;
                    r[u] = __fdividef(1.0f, nrm + p.eps);
                }
                // r in three bf16 parts: row rt of the B operand's K dimension, rows 3 u..3 u + 2 of its N dimension
                float rest = r[u];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const __nv_bfloat16 h16 = __float2bfloat16_rn(rest);
                    const int nn = 3 * u + c;        // (32-byte rows, 32-byte swizzle: rows 4..7 have their 16-byte halves swapped)
                    *reinterpret_cast<__nv_bfloat16 *>(bop + (rt >> 4) * 512 + nn * 32 + ((((rt & 15) >> 3) ^ (nn >> 2)) << 4) + (rt & 7) * 2) = h16;
                    rest -= __bfloat162float(h16);
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");       // generic writes -> tensor-core (and TMA) reads
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(bar(kBarReady + g));
                if (kCodes) mbar_arrive(bar(kBarEmpty + s));
            }
            // ---- what a row leaves behind, written while the products run
#pragma unroll
            for (int u = 0; u < kSub; ++u) {
                const int tile = w.tile + u, row = tile * kTile + rt;
                if (kSub > 1 && tile >= p.tiles) break;
                p.inv_norm[(size_t)w.head * p.cap_pad + row] = r[u];
                p.self_dot[(size_t)w.head * p.cap_pad + row] = (r[u] * r[u]) * sq[u];     // Kbar_i . Kbar_i
                if (p.tri) write_slices(p, w.head, tile, rt, w.n, r[u]);
            }
            if (!__all_sync(0xffffffffu, mbar_wait(bar(kBarLogits + g), turn & 1u, abort_flag, sink))) break;
            if (q_rows_pad && w.rows_here > 0) {
                tc_fence_after();
#pragma unroll
                for (int u = 0; u < kSub; ++u) {
                    if (u > 0 && w.rows_here <= u * kTile) break;
                    pool_logits<kCodes>(p, lane_base + 16u + (uint32_t)(u * q_rows_pad), u * kTile + rt < w.rows_here,
                                p.logits + (size_t)w.head * p.alpha * p.cap_pad + (w.tile + u) * kTile + rt);
                }
            }
            if (!__all_sync(0xffffffffu, mbar_wait(bar(kBarSums + g), turn & 1u, abort_flag, sink))) break;
            float tsum = 0.f;
            if (w.rows_here > 0) {
                tc_fence_after();
                uint32_t acc[8];
                tmem_ld8(lane_base, acc);            // lane = column c of the keys (of tile c / D of the unit)
                tmem_wait8(acc);
                tsum = kSub > 1 && rt >= D ? (__uint_as_float(acc[3]) + __uint_as_float(acc[4])) + __uint_as_float(acc[5])
                                           : (__uint_as_float(acc[0]) + __uint_as_float(acc[1])) + __uint_as_float(acc[2]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kBarTaken + g));
            if (kSub == 1 || w.tile + rt / D < p.tiles) p.tile_sum[((size_t)w.head * p.tiles + w.tile) * D + rt] = tsum;
        }
    }

    // ---------------------------------------------------------------------- common exit
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {                      // error path: what is under way lands, and the block's units are given up
        if ((warp == 1 || warp == 2) && lane == 0) {
            umma_commit(bar(kBarDrain));
            drain(bar(kBarDrain), 0);
        }
        if (threadIdx.x == 0) {
            for (int k = max(misc[2] - (int)stages, 0); k < misc[2]; ++k) drain(bar(kBarFull + (uint32_t)k % stages), ((uint32_t)k / stages) & 1u);
            for (int q = max(misc[3] - q_bufs, 0); q < misc[3]; ++q) drain(bar(kBarQFull + q % q_bufs), (uint32_t)(q / q_bufs) & 1u);
            for (int k = 0; k < units; ++k) {
                const PrepUnit w = prep_unit_at<kSub>(p, first + k, !p.lengths_done);
                for (int u = 0; u < kSub && w.tile + u < p.tiles; ++u) p.inv_norm[(size_t)w.head * p.cap_pad + (w.tile + u) * kTile] = kGaveUp;
            }
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

template <int D, bool kCodes>
cudaError_t launch_for(const Params &p, cudaStream_t s)
{
    using F = Form<D, kCodes>;
    static PerDevice done;
    int dev = 0, sms = 0;
    cudaError_t e = device_sms(&dev, &sms);
    if (e != cudaSuccess || (e = allow_smem_once(done, dev, prep_sm100_kernel<D, kCodes>, kSmemLimit)) != cudaSuccess) return e;
    // the logits are left to the other scoring kernels where those form them, and to a later call that scores
    const int q_rows_pad = p.form_logits ? (p.group * p.alpha + 15) / 16 * 16 : 0;
    const int copy = kCodes ? p.fused_codes : 0;
    const int32_t *table = copy ? p.fuse_table : p.block_table;
    const uint64_t rows = table ? (uint64_t)p.pool_pages * kTile : (uint64_t)p.batch * p.hkv * p.cap;
    CUtensorMap map_k, map_q, map_wide;
    const bool ok = (kCodes ? make_map_row128(&map_k, copy ? p.fuse_src : p.k_cache, rows, true) : make_map_rows(&map_k, p.k_cache, rows, D, kTile)) &&
                    make_map_rows(&map_q, p.q_window, (uint64_t)p.batch * p.hq * p.alpha, D, (uint32_t)std::max(q_rows_pad, 16)) &&
                    (!copy || make_map(&map_wide, p.k_cache, (uint64_t)p.batch * p.hkv * p.cap + kTile, kTile));
    if (!ok) return cudaErrorInvalidValue;
    if (!copy) map_wide = map_k;
    const int total = (p.tiles + F::kSub - 1) / F::kSub * p.batch * p.hkv;
    int groups = 1, q_bufs = 2;
    choose_plan<D, kCodes>(q_rows_pad, (p.tiles + F::kSub - 1) / F::kSub, &groups, &q_bufs);
    return launch_early(prep_sm100_kernel<D, kCodes>, (unsigned)std::min(total, sms), kThreads, (size_t)make_plan<D, kCodes>(q_rows_pad, groups, q_bufs).total, s,
                        1, p, map_k, map_q, map_wide, table, copy, total, q_rows_pad, groups, q_bufs);
}

}  // namespace

cudaError_t launch_prep_sm100(const Params &p, cudaStream_t s)
{
    cudaError_t e = cudaSuccess;
    if (p.lengths_done)
        e = launch_early(lengths_kernel, (unsigned)((p.batch + kLengthThreads - 1) / kLengthThreads), kLengthThreads, 0, s, 1, p);
    if (e != cudaSuccess) return e;
    e = p.fused_codes || p.codes ? launch_for<128, true>(p, s) : p.d == 64 ? launch_for<64, false>(p, s) : launch_for<128, false>(p, s);
    return e == cudaSuccess ? launch_head_sum(p, s) : e;
}

// The queries belong to the stage that scores: where that is called by itself, the prep kernel goes over the keys once more with the
// lengths recorded before, and leaves the logits beside what it left then.  (The head sums' kernel is what sees that a block gave up.)
cudaError_t launch_logits_sm100(Params p, cudaStream_t s)
{
    p.lengths_done = p.form_logits = 1;
    p.seq_lens = p.meta;
    p.budgets = p.meta + p.batch;
    const cudaError_t e = p.d == 64 ? launch_for<64, false>(p, s) : launch_for<128, false>(p, s);
    return e == cudaSuccess ? launch_head_sum(p, s) : e;
}

}  // namespace rkv
