// Stage "scores", first pass, for bf16 caches of 64 and 128 dimensions and E4M3 codes of 128: every candidate token against the LAST key tile of its head
// (Eq. 5 and the start of Section 3.3's scan, which runs from the last position downwards) and against the head's key sum (Eq. 6).
// tcgen05.mma with TMEM accumulators, fed by TMA, one persistent block per SM.
//
// The pass is a single sweep over the keys, so it is organised as a stream: the 128-row key tiles of a head flow
// through a ring of shared-memory stages as the A operand (one token per TMEM lane), while ONE B operand block of the
// head stays put: the rows of its last key tile, then 16 rows that hold sum_j Kbar_j split into bf16 parts.  Per streamed tile the
// tensor cores form one product of N = 128 + 16, plus one K = 16 step on the key columns that folds the
// threshold test into the accumulator (slices of both operands written by the prep stage):
//
//   columns [0, 128)         h = k_i . k_j - T / (r_i r_j) for the 128 keys j of the last tile: S[j][i] > T exactly
//                            when h > 0.  The thread that owns token i scans them from the last position downwards,
//                            "the first beta hits" are Section 3.3's partners; a partner's value is T + h r_i r_j
//   columns [128, 144)       k_i . s in three parts, which gives sum_j S[j][i] = Kbar_i . (sum_j Kbar_j) - Kbar_i . Kbar_i without
//                            forming the matrix
//
// Out, per token: the column sum minus the removed entries (sbar), the partners still lacking (a bit, and for beta > 1 how many).
//
// What bounds it: with 128 dimensions the keys' bytes (4096 heads of 4216 tokens: 792 us for 5.0 GB), with 64 the integer instructions
// of the screening (8192 heads of 2168 tokens: 573; 4096 of 4216 in 8 bits: 615, and 765 on their widened copy).  While the query rows rode in the B block too (the logits are the prep stage's
// now) the product had 128 + G alpha + 16 columns, so that only two accumulators fitted, and the epilogue formed the logits: 994 and 786.
//
// Work item = (head, range of row tiles); items are handed out by a global ticket counter, head-major.  The operands
// that stay put are double-buffered across items, so the next item's copies run under the current item's products.
// Warp roles (448 threads): warp 0 = tickets + TMA producer, warp 1 = MMA issuer and TMEM owner, warps 2..13 = epilogue
// in three groups of four (warp w may touch TMEM lanes 32 (w % 4) .. +31); group g drains accumulator buffer g, i.e.
// every third tile of the stream.  Every wait on an mbarrier is bounded; on expiry the block records
// RKV_ERR_TIMEOUT, stops issuing work and leaves through the common exit that frees TMEM.  No TMA multicast, no
// cluster launch.
#include "rkv_sm100.cuh"

namespace rkv {

namespace {

using namespace sm100;

constexpr int kHalfBytes = kTile * 64 * 2;       // one TMA box: 128 rows x 64 bf16 (128-byte swizzled rows)
constexpr int kSliceBytes = kTile * 32;          // the extra K = 16 slice of an operand: 128 rows x 32 bytes (32-byte swizzle)
constexpr int kMaxStagesA = 8;
constexpr int kMostTurns = 4;                    // partners of a chunk that are taken out one by one
constexpr uint32_t kGroups = 3;                  // accumulator buffers, and the groups of four epilogue warps that drain one each
constexpr uint32_t kAccCols = 160;               // 128 key columns + 16, up to a multiple of 32
constexpr uint32_t kTmemColsP1 = 512;
static_assert(kGroups * kAccCols <= kTmemColsP1, "TMEM columns");
constexpr int kThreadsP1 = 64 + 128 * (int)kGroups;
constexpr int kSmemLimit = 227 * 1024;

enum {
    kBarSlotFull = 0,                            // [2] item descriptor written and its resident operands landed
    kBarSlotEmpty = kBarSlotFull + 2,            // [2] ... no longer read: the MMA thread and the epilogue warps
    kBarAFull = kBarSlotEmpty + 2,               // [kMaxStagesA] streamed tile landed
    kBarAEmpty = kBarAFull + kMaxStagesA,        // [kMaxStagesA] ... and consumed by the products
    kBarAccFull = kBarAEmpty + kMaxStagesA,      // [kGroups] accumulator buffer written
    kBarAccEmpty = kBarAccFull + 3,              // [kGroups] ... and drained by its 4 epilogue warps
    kNumBarsP1 = kBarAccEmpty + 3
};

// Shared memory (offsets from a 1024-byte aligned base).
template <int D>
struct Lay {
    static constexpr int kTileBytes = kTile * D * 2;                   // an operand tile: one 64-column box or two
    // B block: rows [0, 128) the last key tile, then 16 rows of the key sum; as 64-column boxes, one behind the other; then the slice
    // of the last key tile
    static constexpr int kSumBytes = 16 * D * 2, kSlotBytes = kTileBytes + kSumBytes, kBoxBytes = kSlotBytes / (D / 64);
    static constexpr int kSlotStride = kSlotBytes + kSliceBytes;
    static constexpr int kFixed = 2 * (kSlotStride + kTile * 4) + kNumBarsP1 * 8 + 2 * 16 + 32 + 1024;      // + alignment slack
    static constexpr int kFit = (kSmemLimit - kFixed) / (kTileBytes + kSliceBytes);
    static constexpr int kStages = kFit > kMaxStagesA ? kMaxStagesA : kFit;                                // ring depth
    static constexpr int kOffAug = kStages * kTileBytes;               // a slice per stage
    static constexpr int kOffSlot = kOffAug + kStages * kSliceBytes;   // 2 B blocks
    static constexpr int kOffRj = kOffSlot + 2 * kSlotStride;          // 2 x 128 floats: r_j of the last key tile
    static constexpr int kOffBar = kOffRj + 2 * kTile * 4;
    static constexpr int kOffItems = (kOffBar + kNumBarsP1 * 8 + 15) / 16 * 16;
    static constexpr int kOffMisc = kOffItems + 2 * 16;
    static constexpr int kBytes = kOffMisc + 16 + 1024;
    static_assert(kBoxBytes % 1024 == 0 && kBytes <= kSmemLimit, "shared memory");
};

// Item descriptor (int4): {head, first row tile, one past the last row tile, n}.  x < 0: no more items.
// kCodes: E4M3 codes of 128 dimensions, whose rows are as long as those of 64 dimensions in bf16 (D = 64).  kRule: the retention rule is on.  kOne: beta = 1.  kMany: beta > kMostTurns, the form that can also take a chunk's partners out in one sum
// (each without the others' code: the roles share the instruction cache).
template <int D, bool kCodes, bool kRule, bool kOne, bool kMany>
__global__ void __launch_bounds__(kThreadsP1, 1)
scores_stream_sm100_kernel(Params p, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_hs,
                           const __grid_constant__ CUtensorMap map_ns, const __grid_constant__ CUtensorMap map_ts, int splits,
                           unsigned long long total_items)
{
    using L = Lay<D>;
    constexpr uint32_t kStages = L::kStages;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = align_smem(smem_raw);
    const uint32_t sbase = smem_u32(smem);
    int4 *items = reinterpret_cast<int4 *>(smem + L::kOffItems);
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(smem + L::kOffMisc);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + L::kOffMisc + 4);
    volatile int *bail = reinterpret_cast<volatile int *>(smem + L::kOffMisc + 8);
    const uint32_t bar0 = sbase + L::kOffBar;
    auto bar = [bar0](uint32_t idx) -> uint32_t { return bar0 + 8u * idx; };

    // Once a bounded wait of this call has run out, the blocks still to start return at once.
    const ErrSink sink = make_sink(p);
    pdl_wait();
    if (threadIdx.x == 0) *bail = call_aborted(p) ? 1 : 0;
    __syncthreads();
    if (*bail) return;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(bar(kBarSlotFull + s), 1);
            mbar_init(bar(kBarSlotEmpty + s), 1 + 4 * kGroups);
        }
        for (uint32_t s = 0; s < kGroups; ++s) {
            mbar_init(bar(kBarAccFull + s), 1);
            mbar_init(bar(kBarAccEmpty + s), 4);
        }
        for (int s = 0; s < kMaxStagesA; ++s) {
            mbar_init(bar(kBarAFull + s), 1);
            mbar_init(bar(kBarAEmpty + s), 1);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_holder)), "r"(kTmemColsP1) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    unsigned long long tiles_done = 0ull;

    if (warp == 0) {
        // ------------------------------------------------------------------ tickets + TMA producer
        if (lane == 0) {
            uint32_t k_item = 0, acount = 0;
            bool ok = true;
            // the next ticket is drawn while the current item is set up (a block draws one ticket too many)
            unsigned long long next_ticket = atomicAdd(&p.counters[1], 1ull);
            while (ok) {
                const unsigned long long ticket = next_ticket;
                if (ticket >= total_items) break;
                next_ticket = atomicAdd(&p.counters[1], 1ull);
                const int head = (int)(ticket / (unsigned)splits);
                const int part = (int)(ticket % (unsigned)splits);
                const int n = seq_candidates(p, head / p.hkv);
                if (n == 0) continue;
                const int n_tiles = (n + kTile - 1) / kTile;
                const int t0 = (int)((long long)part * n_tiles / splits), t1 = (int)((long long)(part + 1) * n_tiles / splits);
                if (t0 >= t1) continue;                                        // more parts than tiles

                const uint32_t slot = k_item & 1;
                if (!mbar_wait(bar(kBarSlotEmpty + slot), ((k_item >> 1) & 1) ^ 1, abort_flag, sink)) break;
                items[slot] = make_int4(head, t0, t1, n);
                const uint32_t slot_addr = sbase + L::kOffSlot + slot * L::kSlotStride;
                const uint32_t full = bar(kBarSlotFull + slot);
                // the descriptor is published by this arrival; the barrier completes when the operands have landed too
                mbar_expect_tx(full, (uint32_t)L::kSumBytes + (kRule ? (uint32_t)(L::kTileBytes + kSliceBytes + kTile * 4) : 0u));
                // behind the key tile's rows: 16 rows holding sum_j Kbar_j split into bf16 parts; every 64-column box
#pragma unroll
                for (int x = 0; x < D / 64; ++x) tma_load_2d(slot_addr + x * L::kBoxBytes + kTile * 128, &map_hs, x * 64, head * (kCodes ? kSumHeadBytes / 128 : 16), full);
                if (kRule) {
                    const int y = (int)tile_row0(p, head, n_tiles - 1);
#pragma unroll
                    for (int x = 0; x < D / 64; ++x) tma_load_2d(slot_addr + x * L::kBoxBytes, &map_k, x * 64, y, full);
                    // the tile's extra slice: -T / r_j of its keys in three bf16 parts
                    tma_load_2d(slot_addr + L::kSlotBytes, &map_ts, 0, head * kTile, full);
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 ::"r"(sbase + L::kOffRj + slot * kTile * 4),
                                   "l"(p.inv_norm + (size_t)head * p.cap_pad + (size_t)(n_tiles - 1) * kTile),
                                   "r"((uint32_t)(kTile * 4)), "r"(full)
                                 : "memory");
                }
                for (int t = t0; t < t1; ++t) {
                    const uint32_t s = acount % kStages;
                    if (!mbar_wait(bar(kBarAEmpty + s), ((acount / kStages) & 1) ^ 1, abort_flag, sink)) {
                        ok = false;
                        break;
                    }
                    const uint32_t dst = sbase + s * L::kTileBytes;
                    const int y = (int)tile_row0(p, head, t);
                    mbar_expect_tx(bar(kBarAFull + s), L::kTileBytes + (kRule ? kSliceBytes : 0));
                    tma_load_2d(dst, &map_k, 0, y, bar(kBarAFull + s));
                    if (D == 128) tma_load_2d(dst + kHalfBytes, &map_k, 64, y, bar(kBarAFull + s));
                    if (kRule)      // the tile's extra slice: 1 / r_i of its keys in three bf16 parts
                        tma_load_2d(sbase + L::kOffAug + s * kSliceBytes, &map_ns, 0, head * p.cap_pad + t * kTile,
                                    bar(kBarAFull + s));
                    ++acount;
                }
                ++k_item;
            }
            // terminator: tells the other roles that no item follows (skipped when the block is aborting)
            if (!*abort_flag) {
                const uint32_t slot = k_item & 1;
                if (mbar_wait(bar(kBarSlotEmpty + slot), ((k_item >> 1) & 1) ^ 1, abort_flag, sink)) {
                    items[slot] = make_int4(-1, 0, 0, 0);
                    mbar_arrive(bar(kBarSlotFull + slot));
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            // one product per streamed tile: N = the 128 keys of the last tile + the key sum (that alone while the rule is off)
            const uint32_t idesc_ks = kCodes ? instr_desc_codes(kTile, kTile + 16) : instr_desc(kTile, kTile + 16);
            const uint32_t idesc_s = kCodes ? instr_desc_codes(kTile, 16) : instr_desc(kTile, 16);
            const uint32_t idesc_k = instr_desc(kTile, kTile);
            uint32_t k_item = 0, acount = 0;
            bool ok = true;
            while (ok) {
                const uint32_t slot = k_item & 1;
                if (!mbar_wait(bar(kBarSlotFull + slot), (k_item >> 1) & 1, abort_flag, sink)) break;
                const int4 d = items[slot];
                if (d.x < 0) break;
                const uint32_t b_block = sbase + L::kOffSlot + slot * L::kSlotStride;
                for (int t = d.y; t < d.z; ++t) {
                    const uint32_t s = acount % kStages;
                    if (!mbar_wait(bar(kBarAFull + s), (acount / kStages) & 1, abort_flag, sink)) {
                        ok = false;
                        break;
                    }
                    const uint32_t a = acount % kGroups;           // tile c of the stream uses accumulator buffer c % kGroups
                    if (!mbar_wait(bar(kBarAccEmpty + a), ((acount / kGroups) & 1) ^ 1, abort_flag, sink)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t tile = sbase + s * L::kTileBytes;
                    const uint32_t d_tmem = tmem_base + a * kAccCols;
                    if (kRule) {
                        if (D == 128) umma_tile_k128_halves(d_tmem, tile, kHalfBytes, b_block, L::kBoxBytes, idesc_ks);
                        else umma_tile_row128<kCodes>(d_tmem, tile, b_block, idesc_ks);
                        // ... - T / (r_i r_j) onto the key columns: the accumulator's sign is the threshold test
                        umma_k16_sw32(d_tmem, sbase + L::kOffAug + s * kSliceBytes, b_block + L::kSlotBytes, idesc_k);
                        ++tiles_done;
                    } else {
                        if (D == 128) umma_tile_k128_halves(d_tmem + 128, tile, kHalfBytes, b_block + kTile * 128, L::kBoxBytes, idesc_s);
                        else umma_tile_row128<kCodes>(d_tmem + 128, tile, b_block + kTile * 128, idesc_s);
                    }
                    umma_commit(bar(kBarAccFull + a));
                    umma_commit(bar(kBarAEmpty + s));              // the stage may be refilled once these products have read it
                    ++acount;
                }
                if (!ok) break;
                umma_commit(bar(kBarSlotEmpty + slot));            // so may the item's resident operands
                ++k_item;
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------------ epilogue warps
        const uint32_t grp = (uint32_t)(warp - 2) >> 2;      // accumulator buffer this warp drains
        const int quad = warp & 3;               // TMEM lane quadrant this warp may access
        const int lrow = quad * 32 + lane;       // row within the 128-row tile
        const uint32_t lane_base = tmem_base + ((uint32_t)(quad * 32) << 16) + grp * kAccCols;
        uint32_t k_item = 0, ccount = 0;         // ccount: tiles of the stream so far (all of them, not only this group's)
        bool ok = true;

        while (ok) {
            const uint32_t slot = k_item & 1;
            if (!mbar_wait(bar(kBarSlotFull + slot), (k_item >> 1) & 1, abort_flag, sink)) break;
            const int4 d = items[slot];
            if (d.x < 0) break;
            const int head = d.x, n = d.w;
            const int last_tile = (n + kTile - 1) / kTile - 1;
            const int jbase = last_tile * kTile;
            const float *inv_norm = p.inv_norm + (size_t)head * p.cap_pad;
            const float *rj = reinterpret_cast<const float *>(smem + L::kOffRj + slot * kTile * 4);
            const float *self_dot = p.self_dot + (size_t)head * p.cap_pad;
            const float sum_scale = kCodes ? *reinterpret_cast<const float *>(reinterpret_cast<const uint8_t *>(p.head_sum_bf16) + (size_t)head * kSumHeadBytes + kSumScaleAt) : 1.f;
            float ri_next = 0.f, self_next = 0.f;
            int t_next = -1;                     // the tile ri_next / self_next were fetched for
            for (int t = d.y; t < d.z; ++t, ++ccount) {
                if (ccount % kGroups != grp) continue;
                const int i = t * kTile + lrow;
                const bool row_ok = i < n;
                float ri, self;
                if (t_next == t) {
                    ri = ri_next;
                    self = self_next;
                } else {
                    ri = row_ok ? inv_norm[i] : 0.f;
                    self = row_ok ? self_dot[i] : 0.f;
                }
                if (t + (int)kGroups < d.z) {    // this group's next tile of the item: its factors arrive while this one is drained
                    const int i2 = i + (int)kGroups * kTile;
                    t_next = t + (int)kGroups;
                    ri_next = i2 < n ? inv_norm[i2] : 0.f;
                    self_next = i2 < n ? self_dot[i2] : 0.f;
                }
                if (!mbar_wait(bar(kBarAccFull + grp), (ccount / kGroups) & 1, abort_flag, sink)) {
                    ok = false;
                    break;
                }
                tc_fence_after();

                // ---- Eq. 6 before the retention rule, sum_j S[j][i]: Kbar_i . s (in parts) - Kbar_i . Kbar_i
                uint32_t sp[8];
                tmem_ld8(lane_base + 128, sp);
                tmem_wait8(sp);
                float sum = __uint_as_float(sp[kCodes ? kSumParts - 1 : 0]);
                if (kCodes) {
#pragma unroll
                    for (int part = kSumParts - 2; part >= 0; --part) sum = fmaf(sum, 0.0625f, __uint_as_float(sp[part]));
                    sum *= sum_scale;
                } else {
                    sum = (sum + __uint_as_float(sp[1])) + __uint_as_float(sp[2]);
                }
                const float total = ri * sum - self;

                // ---- the last key tile, last position first.  The accumulator holds h = k_i . k_j - T / (r_i r_j):
                // S[j][i] > T exactly when h > 0, so the screening is a sign test with nothing to load per column; a
                // partner's value is S = T + h r_i r_j, with the r_j of the tile in shared memory.
                float removed = 0.f;             // sum of h r_j over the partners found
                int nhit = 0;
                int left = row_ok ? (kOne ? 1 : p.beta) : 0;
                if (kRule) {
                    bool want = left > 0;
                    const int valid = n - jbase;                  // columns [0, valid) of the tile are candidates
                    // 32-column chunks, last first.  The TMEM load of the next chunk is issued before the current one is
                    // looked at, so its latency passes under the work (two register sets, used alternately).
                    auto chunk = [&](const uint32_t (&g)[32], int ch) {
                        const int nv = valid - ch * 32;
                        uint32_t colmask = nv >= 32 ? 0xffffffffu : (nv <= 0 ? 0u : ((1u << nv) - 1u));
                        const unsigned own = (unsigned)(i - (jbase + ch * 32));           // zero diagonal (Eq. 5)
                        if (own < 32u) colmask &= ~(1u << own);
                        // bit c of `neg` = sign bit of entry c: one funnel shift per entry, four independent chains
                        uint32_t n0 = 0u, n1 = 0u, n2 = 0u, n3 = 0u;
#pragma unroll
                        for (int c = 7; c >= 0; --c) {
                            n0 = __funnelshift_l(g[c], n0, 1);
                            n1 = __funnelshift_l(g[8 + c], n1, 1);
                            n2 = __funnelshift_l(g[16 + c], n2, 1);
                            n3 = __funnelshift_l(g[24 + c], n3, 1);
                        }
                        const uint32_t neg = (n0 | (n1 << 8)) | ((n2 << 16) | (n3 << 24));
                        // entries with a clear sign bit (h > 0, but also +0 and some NaN patterns of rows that are not
                        // candidates: confirmed one by one below), the highest first, its value picked by a select tree
                        // (with beta = 1 nearly always a single turn)
                        uint32_t pos = want ? (~neg & colmask) : 0u;
                        if (kOne) {
                            while (pos != 0u) {
                                const int top = 31 - __clz((int)pos);
                                const float hv = pick32(g, top);
                                if (hv > 0.f) {
                                    removed = hv * rj[ch * 32 + top];
                                    nhit = 1;
                                    left = 0;
                                    want = false;
                                    break;
                                }
                                pos &= ~(1u << top);
                            }
                            return;
                        }
                        // Several partners: a turn each, or, where some lane has many, one sum over the columns for all lanes (a
                        // warp takes as many turns as the lane with most).
                        const int turns = !kMany ? 0 : (int)__reduce_max_sync(0xffffffffu, pos != 0u ? (unsigned)min(__popc(pos), left) : 0u);
                        if (kMany && turns > kMostTurns) {
                            uint32_t hits = 0u;
#pragma unroll
                            for (int c = 0; c < 32; ++c) hits |= (__uint_as_float(g[c]) > 0.f) ? (1u << c) : 0u;
                            hits &= pos;
                            int taken = __popc(hits);
                            for (; taken > left; --taken) hits &= hits - 1u;                   // drop the lowest positions
                            float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll
                            for (int q = 0; q < 8; ++q) {
                                const float4 R = reinterpret_cast<const float4 *>(rj)[ch * 8 + q];
                                s0 += (hits >> (4 * q) & 1u) ? __uint_as_float(g[4 * q]) * R.x : 0.f;
                                s1 += (hits >> (4 * q + 1) & 1u) ? __uint_as_float(g[4 * q + 1]) * R.y : 0.f;
                                s2 += (hits >> (4 * q + 2) & 1u) ? __uint_as_float(g[4 * q + 2]) * R.z : 0.f;
                                s3 += (hits >> (4 * q + 3) & 1u) ? __uint_as_float(g[4 * q + 3]) * R.w : 0.f;
                            }
                            removed += (s0 + s1) + (s2 + s3);
                            nhit += taken;
                            left -= taken;
                            want = left > 0;
                            return;
                        }
                        while (pos != 0u) {
                            const int top = 31 - __clz((int)pos);
                            const float hv = pick32(g, top);
                            pos &= ~(1u << top);
                            if (hv > 0.f) {
                                removed += hv * rj[ch * 32 + top];
                                ++nhit;
                                if (--left == 0) {
                                    want = false;
                                    break;
                                }
                            }
                        }
                    };
                    if (__any_sync(0xffffffffu, want)) {
                        uint32_t ga[32], gb[32];
                        tmem_ld32(lane_base + 3 * 32, ga);
                        tmem_wait32(ga);
                        tmem_ld32(lane_base + 2 * 32, gb);
                        chunk(ga, 3);
                        tmem_wait32(gb);
                        if (__any_sync(0xffffffffu, want)) {                              // else every token of the warp is served
                            tmem_ld32(lane_base + 1 * 32, ga);
                            chunk(gb, 2);
                            tmem_wait32(ga);
                            if (__any_sync(0xffffffffu, want)) {
                                tmem_ld32(lane_base, gb);
                                chunk(ga, 1);
                                tmem_wait32(gb);
                                if (__any_sync(0xffffffffu, want)) chunk(gb, 0);
                            }
                        }
                    }
                }
                // the accumulator buffer is free again
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kBarAccEmpty + grp));

                if (row_ok) {
                    p.sbar[(size_t)head * p.cap_pad + i] = total - ((float)nhit * p.sim_threshold + removed * ri);
                    if (kRule && !kOne && p.beta > 1) p.left[(size_t)head * p.cap_pad + i] = left;
                }
                if (kRule) {                     // the tokens still short of partners, a bit each
                    const unsigned lacking = __ballot_sync(0xffffffffu, left > 0);
                    if (lane == 0) p.lacking[(size_t)head * (p.cap_pad / 32) + t * 4 + quad] = lacking;
                }
            }
            if (!ok) break;
            // the item's r_j and descriptor are no longer read by this warp
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kBarSlotEmpty + slot));
            ++k_item;
        }
    }

    // ---------------------------------------------------------------------- common exit
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        if (*abort_flag) __nanosleep(200000);      // error path only: let copies and MMAs in flight land
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemColsP1) : "memory");
    }
    if (warp == 1 && lane == 0 && !*abort_flag && tiles_done) atomicAdd(p.counters, tiles_done);
}

}  // namespace

template <int D, bool kCodes, bool kRule, bool kOne, bool kMany>
static cudaError_t launch_pass1_for(const Params &p, cudaStream_t s, const CUtensorMap &map_k, const CUtensorMap &map_hs, const CUtensorMap &map_ns,
                                    const CUtensorMap &map_ts)
{
    static PerDevice done;
    int dev = 0, sms = 0;
    cudaError_t e = device_sms(&dev, &sms);
    if (e != cudaSuccess || (e = allow_smem_once(done, dev, scores_stream_sm100_kernel<D, kCodes, kRule, kOne, kMany>, Lay<D>::kBytes)) != cudaSuccess) return e;
    const int heads = p.batch * p.hkv;
    // a head is cut into parts when there are too few heads to give every SM several items
    int splits = (4 * sms + heads - 1) / heads;
    splits = splits < 1 ? 1 : (splits > p.tiles ? p.tiles : splits);
    const unsigned long long total_items = (unsigned long long)splits * (unsigned long long)heads;
    const unsigned grid = (unsigned)(total_items < (unsigned long long)sms ? total_items : (unsigned long long)sms);
    return launch_early(scores_stream_sm100_kernel<D, kCodes, kRule, kOne, kMany>, grid, kThreadsP1, (size_t)Lay<D>::kBytes, s, 1, p, map_k, map_hs, map_ns, map_ts,
                        splits, total_items);
}

template <int D, bool kCodes>
static cudaError_t launch_pass1_form(const Params &p, cudaStream_t s, const CUtensorMap &map_k, const CUtensorMap &map_hs, const CUtensorMap &map_ns,
                                     const CUtensorMap &map_ts)
{
    if (p.beta < 1 || !(p.sim_threshold < 1.0f)) return launch_pass1_for<D, kCodes, false, false, false>(p, s, map_k, map_hs, map_ns, map_ts);
    return p.beta == 1           ? launch_pass1_for<D, kCodes, true, true, false>(p, s, map_k, map_hs, map_ns, map_ts)
           : p.beta > kMostTurns ? launch_pass1_for<D, kCodes, true, false, true>(p, s, map_k, map_hs, map_ns, map_ts)
                                 : launch_pass1_for<D, kCodes, true, false, false>(p, s, map_k, map_hs, map_ns, map_ts);
}

cudaError_t launch_scores_pass1_sm100(const Params &p, cudaStream_t s, const CUtensorMap &map_k, const CUtensorMap &map_hs,
                                      const CUtensorMap &map_ns, const CUtensorMap &map_ts)
{
    return p.codes     ? launch_pass1_form<64, true>(p, s, map_k, map_hs, map_ns, map_ts)
           : p.d == 64 ? launch_pass1_form<64, false>(p, s, map_k, map_hs, map_ns, map_ts)
                       : launch_pass1_form<128, false>(p, s, map_k, map_hs, map_ns, map_ts);
}

}  // namespace rkv
