// Stage "scores", second pass, for bf16 caches of 64 and 128 dimensions and E4M3 codes of 128: the tokens that the first pass (rkv_scores_p1_sm100.cu) left short
// of partners against the key tiles BELOW the last one, last to first.  tcgen05.mma with TMEM accumulators, fed by
// TMA, one persistent block per SM.
//
// Section 3.3's rule needs, per token i, the beta LARGEST positions j with S[j][i] > T.  S is symmetric before the
// rule, so token i's line can be read as row i, and a scan from the last position downwards turns the rule into "the
// first beta hits".  The first pass scans every token against the last key tile; where similar keys are common that
// settles most tokens.  The rest is done here, in ROUNDS:
//
//   list    The tokens still short of partners (a bit each, kept by the scans) are listed per head, ascending, in chunks of 256 (strag_compact_kernel).
//   scan    Work item = (head, chunk of 256 listed tokens, window of key tiles): the chunk's key rows are gathered
//           into two resident operand tiles by the gather warps; the window's key tiles stream through a ring, last
//           to first.  The removed entries are subtracted from what the first pass stored, `left` is updated.
//
// The first round's window is a few tiles only (kRoundTiles); the tokens that found their partners in it drop out of the next
// round's list, so the long scan down to tile 0 is paid only by the few tokens that have no partner at all (a
// single-round scan would drag every listed token of a chunk along with them).  The last round's window reaches
// tile 0.  Worst case (no pair above T): the rounds together form the whole matrix below the last tile.
//
// Every tile product carries one extra K = 16 step that folds the threshold test into the accumulator (see the
// epilogue): the screening is a maximum and a sign test with nothing to load per column.  The n x n matrix never
// leaves TMEM, and no atomics or global flags are involved in the scores.
//
// An item of 128 tokens or fewer needs one row tile: with beta = 1 its window's key tiles are then dealt out to both halves of the
// pipeline in turn (issuer, accumulators, epilogue warps), which merge their findings at the item's end -- the larger position
// counts.  With one half idle such a tile took 1400 cycles, all of it waits for the other side (8192 heads of 2168 tokens
// of 64 dimensions, 40 listed per head: the pass 745 us, 516 now).
//
// Items are handed out by a global ticket counter, longest first within a head, so neighbouring blocks work on
// the same head while its keys are in L2.
// Warp roles (512 threads): warp 15 = tickets (publishes item descriptors up to three items ahead), warps 11..14 =
// gather (fill the resident tiles of the NEXT item while the current one is scanned), warp 0 = TMA
// producer of the streamed key tiles, warp 1 = MMA issuer of row tile 0 and TMEM owner, warp 10 = MMA issuer of row
// tile 1, warps 2..9 = epilogue (warp w may touch TMEM lanes 32 (w % 4) .. +31; warps 2-5 serve row tile 0, warps 6-9
// row tile 1).
// TMEM: four 128-column fp32 accumulators, two per row tile, so the tensor pipe fills one while the epilogue
// drains the other.  Every wait on an mbarrier is bounded; on expiry the block records RKV_ERR_TIMEOUT, stops
// issuing work and leaves through the common exit that frees TMEM.  No TMA multicast and no cluster launch.
#include "rkv_sm100.cuh"

namespace rkv {

namespace {

using namespace sm100;

constexpr int kThreads = 512;                    // 16 warps: producer, 2 MMA issuers (warps 1 and 10), 8 epilogue, 4 gather, tickets
constexpr int kGatherWarp0 = 11;                 // first of the 4 gather warps
constexpr int kTicketWarp = 15;                  // draws the items and publishes their descriptors, up to three items ahead
constexpr int kItemSlots = 4;                    // ring depth of item descriptors
constexpr int kHalfBytes = kTile * 64 * 2;       // one TMA box: 128 rows x 64 bf16 (128-byte swizzled rows)
constexpr int kRowsPerItem = 2 * kTile;
constexpr uint32_t kTmemCols = 512;
constexpr int kPass1Depth = 1;                   // key tiles every token is scanned against in the first pass
constexpr int kRoundWords = 8;                   // Params::counters[kRoundWords + 2 r], [.. + 1]: items and ticket of round r

// The operand tiles of D-dimensional keys and where everything lies in shared memory (offsets from a 1024-byte aligned base).
// The streamed tiles' copies take about 2 us under load, so as many of them as fit are under way: with 128 dimensions three resident
// tiles instead of four make room for a third stage (4096 heads of 4216 tokens: 1439 us with four and two, 1384; 7168 of 2168: 973, 903;
// 4096 of 1144, beta = 4: 605, 589; with 64 dimensions six stages instead of four make no difference).  The second tile of the next
// item then waits, in registers, for the present item's end.
// The extra K = 16 slices of the operands: 128 rows x 32 bytes each (32-byte swizzle), one per resident tile and one
// per stage of the ring.
constexpr int kSliceBytes = kTile * 32;
template <int D>
struct Lay {
    static constexpr int kTileBytes = kTile * D * 2;                  // one 64-column box (16 KB) or two
    static constexpr int kResident = D == 64 ? 4 : 3;                 // resident tiles (128 gathered rows each), taken in turn
    static constexpr int kStagesB = D == 64 ? 6 : 3;                  // ring depth of streamed tiles
    static constexpr int kOffA = 0;
    static constexpr int kOffB = kOffA + kResident * kTileBytes;
    static constexpr int kOffAugA = kOffB + kStagesB * kTileBytes;
    static constexpr int kOffAugB = kOffAugA + kResident * kSliceBytes;
    // what the epilogue needs to know about a tile's tokens, left by the gather warps: position, r_i, partners lacking
    static constexpr int kOffStash = kOffAugB + kStagesB * kSliceBytes;            // kResident x 3 arrays x kTile words
    static constexpr int kOffMerge = kOffStash + kResident * 3 * kTile * 4;        // kResident x {position, accumulator value} x kTile: see kBarMerge
    static constexpr int kOffBar = kOffMerge + kResident * 2 * kTile * 4;          // mbarriers
    static constexpr int kBarQFull = 0;                          // [kItemSlots] item descriptor written
    static constexpr int kBarQEmpty = kBarQFull + kItemSlots;    // [kItemSlots] read by the producer, the 2 MMA threads, the 8 epilogue and the 4 gather warps
    static constexpr int kBarAFull = kBarQEmpty + kItemSlots;    // [kResident] resident tile, slice and stash in place (4 gather warps)
    static constexpr int kBarAEmpty = kBarAFull + kResident;     // [kResident] ... no longer read (2 MMA threads, 8 epilogue warps)
    static constexpr int kBarBFull = kBarAEmpty + kResident;     // [kStagesB]
    static constexpr int kBarBEmpty = kBarBFull + kStagesB;      // [kStagesB]
    static constexpr int kBarAccFull = kBarBEmpty + kStagesB;    // [2 buffers][2 row tiles]
    static constexpr int kBarAccEmpty = kBarAccFull + 4;         // [2][2], 4 warps each
    // [kResident] findings of the second half of an item of one row tile (its 4 epilogue warps).  As many as resident tiles: the second
    // half can be that many items ahead before it waits for a tile that the first has to give back
    static constexpr int kBarMerge = kBarAccEmpty + 4;
    static constexpr int kNumBars = kBarMerge + kResident;
    static constexpr int kOffItems = (kOffBar + kNumBars * 8 + 15) / 16 * 16;      // kItemSlots x int4
    static constexpr int kOffMisc = kOffItems + kItemSlots * 16;      // tmem base, abort flag, bail flag
    static constexpr int kSmemBytes = kOffMisc + 16 + 1024;           // + slack for the manual 1024-byte alignment
    static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");
};

struct Bars {
    uint32_t bar0;
    __device__ __forceinline__ uint32_t at(int idx) const { return bar0 + 8 * idx; }
};

// Item descriptor (int4): {head, first listed token k0, tokens in the item (1..256) | key tiles of the window << 16,
// first (highest) streamed tile}.  x < 0: no more items.  `round` selects the round's counters.
// kOne: beta = 1 (each form without the other's code: the roles share the instruction cache.  1433 -> 1401 us
// for 4096 heads of 4216 tokens, 591 -> 516 for the 64 dimensions above).
template <int D, bool kCodes, bool kOne>
__global__ void __launch_bounds__(kThreads, 1)
scores_pass2_sm100_kernel(Params p, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_ns,
                          int round)
{
    using L = Lay<D>;
    unsigned long long *const item_count = p.counters + kRoundWords + 2 * round, *const ticket = item_count + 1;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = align_smem(smem_raw);
    const uint32_t sbase = smem_u32(smem);
    int4 *items = reinterpret_cast<int4 *>(smem + L::kOffItems);
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(smem + L::kOffMisc);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + L::kOffMisc + 4);
    volatile int *bail = reinterpret_cast<volatile int *>(smem + L::kOffMisc + 8);
    const Bars bar{sbase + L::kOffBar};

    // Once a bounded wait of this call has run out, the blocks still to start return at once (a sequence with an
    // invalid length does not stop the others: it just has no candidates).  Pass 2 has nothing to do when the list
    // is empty.
    const ErrSink sink = make_sink(p);
    pdl_wait();
    if (threadIdx.x == 0) {
        int b = call_aborted(p) ? 1 : 0;
        if (*item_count == 0ull) b = 1;
        *bail = b;
    }
    __syncthreads();
    if (*bail) return;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned long long total_items = *item_count;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kItemSlots; ++s) {
            mbar_init(bar.at(L::kBarQFull + s), 1);
            mbar_init(bar.at(L::kBarQEmpty + s), 15);
        }
        for (int s = 0; s < L::kResident; ++s) {
            // the 4 gather warps fill the resident tiles; the MMA threads and the epilogue warps read them and the stash
            mbar_init(bar.at(L::kBarAFull + s), 4);
            mbar_init(bar.at(L::kBarAEmpty + s), 10);
            mbar_init(bar.at(L::kBarMerge + s), 4);
        }
        for (int s = 0; s < L::kStagesB; ++s) {
            mbar_init(bar.at(L::kBarBFull + s), 1);
            mbar_init(bar.at(L::kBarBEmpty + s), 2);              // both MMA issuers
        }
        for (int s = 0; s < 4; ++s) {
            mbar_init(bar.at(L::kBarAccFull + s), 1);
            mbar_init(bar.at(L::kBarAccEmpty + s), 4);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_holder)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_holder;
    unsigned long long tiles_done = 0ull;
    // The u-th use of a resident tile: its buffer, and the parity of its barriers' phase.  Whoever waits for these barriers meets every
    // phase in order (a parity tells two neighbouring phases apart, no more).
    auto buf_of = [](uint32_t u) -> uint32_t { return u % L::kResident; };
    auto phase_of = [](uint32_t u) -> uint32_t { return u / L::kResident & 1u; };
    auto prefetch_tile = [&](int head, int jt) {
        const int y = (int)tile_row0(p, head, jt);
#pragma unroll
        for (int x = 0; x < D; x += 64)
            asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(reinterpret_cast<uint64_t>(&map_k)), "r"(x), "r"(y) : "memory");
    };

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0) {
            uint32_t k_item = 0, bcount = 0;
            bool ok = true;
            while (ok) {
                const uint32_t qs = k_item % kItemSlots;
                if (!mbar_wait(bar.at(L::kBarQFull + qs), (k_item / kItemSlots) & 1, abort_flag, sink)) break;
                const int4 desc = items[qs];            // {head, first listed token, tokens | window, first streamed tile}
                mbar_arrive(bar.at(L::kBarQEmpty + qs));
                if (desc.x < 0) break;
                const int head = desc.x;
                const int first_tile = desc.w;             // streamed tiles: first_tile .. first_tile - n_iter + 1
                const int n_iter = desc.z >> 16;
                for (int it = 0; it < n_iter; ++it) {
                    const uint32_t s = bcount % L::kStagesB;
                    if (!mbar_wait(bar.at(L::kBarBEmpty + s), ((bcount / L::kStagesB) & 1) ^ 1, abort_flag, sink)) {
                        ok = false;
                        break;
                    }
                    const uint32_t dst = sbase + L::kOffB + s * L::kTileBytes;
                    const int jt = first_tile - it;
                    const int y = (int)tile_row0(p, head, jt);
                    mbar_expect_tx(bar.at(L::kBarBFull + s), L::kTileBytes + kSliceBytes);
                    tma_load_2d(dst, &map_k, 0, y, bar.at(L::kBarBFull + s));
                    if (D == 128) tma_load_2d(dst + kHalfBytes, &map_k, 64, y, bar.at(L::kBarBFull + s));
                    // the tile's extra slice: the norms of its keys in three bf16 parts
                    tma_load_2d(sbase + L::kOffAugB + s * kSliceBytes, &map_ns, 0, head * p.cap_pad + jt * kTile,
                                bar.at(L::kBarBFull + s));
                    ++bcount;
                }
                ++k_item;
            }
        }
        __syncwarp();
    } else if (warp == kTicketWarp) {
        // ------------------------------------------------------------------ tickets
        // Items are published as soon as a descriptor slot is free, so the gather warps learn of the next item while
        // the producer is still streaming the key tiles of the current one.
        if (lane == 0) {
            uint32_t k_item = 0;
            while (true) {
                const unsigned long long cur = atomicAdd(ticket, 1ull);
                if (cur >= total_items) break;
                const int4 desc = p.strag_items[cur];
                const uint32_t qs = k_item % kItemSlots;
                if (!mbar_wait(bar.at(L::kBarQEmpty + qs), ((k_item / kItemSlots) & 1) ^ 1, abort_flag, sink)) break;
                items[qs] = desc;
                mbar_arrive(bar.at(L::kBarQFull + qs));
                // The first tiles of the block's first two items are asked into L2 while their tokens are gathered: nothing else is
                // under way yet.  (256 heads of 1144 tokens, all of whose items these are: the pass 36 -> 32 us; for all items of a
                // large call it costs, 7168 heads of 2168 tokens 895 -> 1041, and for windows of fewer than four tiles too: 512 heads
                // of 192 tokens, two partners, 21.5 us with it, 19.5 without.)
                for (int it = 0; k_item < 2 && (desc.z >> 16) >= 4 && it < 4; ++it) prefetch_tile(desc.x, desc.w - it);
                ++k_item;
            }
            // terminator: tells the other roles that no item follows (skipped when the block is aborting)
            if (!*abort_flag) {
                const uint32_t qs = k_item % kItemSlots;
                if (mbar_wait(bar.at(L::kBarQEmpty + qs), ((k_item / kItemSlots) & 1) ^ 1, abort_flag, sink)) {
                    items[qs] = make_int4(-1, 0, 0, 0);
                    mbar_arrive(bar.at(L::kBarQFull + qs));
                }
            }
        }
        __syncwarp();
    } else if (warp == 1 || warp == 10) {
        // ------------------------------------------------------------------ MMA issuers
        // One thread per row tile of the item (warp 1: row tile 0, warp 10: row tile 1).  With a single issuer the
        // tensor pipe ran dry between tiles while the thread went through its barrier waits; two threads keep each
        // other's products queued.  Both wait for every stage and every item (which keeps either from running a
        // whole barrier phase ahead) and both release them: by a commit after products of their own, by a plain
        // arrival otherwise.
        if (lane == 0) {
            const int m = warp == 1 ? 0 : 1;
            const uint32_t idesc_s = instr_desc(kTile, kTile), idesc_k = kCodes ? instr_desc_codes(kTile, kTile) : idesc_s;
            uint32_t k_item = 0, bcount = 0, cnt = 0, use = 0;       // use: uses of resident tiles before this item
            bool ok = true;
            while (ok) {
                const uint32_t qs = k_item % kItemSlots;
                if (!mbar_wait(bar.at(L::kBarQFull + qs), (k_item / kItemSlots) & 1, abort_flag, sink)) break;
                const int4 d = items[qs];
                mbar_arrive(bar.at(L::kBarQEmpty + qs));
                if (d.x < 0) break;
                const int num_m = (d.z & 0xffff) > kTile ? 2 : 1;
                const int n_iter = d.z >> 16;
                const bool split = kOne && num_m == 1;    // one row tile, its key tiles dealt out to both issuers
                const bool mine = m < num_m || split;
                // the gathered rows are in place (of the second row tile: the first issuer asks at the item's end, to stay in step)
                const uint32_t own = use + (num_m == 2 && m == 1 ? 1u : 0u);
                if (!mbar_wait(bar.at(L::kBarAFull + buf_of(use)), phase_of(use), abort_flag, sink) ||
                    (own != use && !mbar_wait(bar.at(L::kBarAFull + buf_of(own)), phase_of(own), abort_flag, sink)))
                    break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t resident = sbase + L::kOffA + buf_of(own) * L::kTileBytes;
                const uint32_t res_slice = sbase + L::kOffAugA + buf_of(own) * kSliceBytes;
                for (int it = 0; it < n_iter; ++it) {
                    const uint32_t s = bcount % L::kStagesB;
                    if (!mbar_wait(bar.at(L::kBarBFull + s), (bcount / L::kStagesB) & 1, abort_flag, sink)) {
                        ok = false;
                        break;
                    }
                    const uint32_t stage = sbase + L::kOffB + s * L::kTileBytes;
                    if (mine && (!split || (it & 1) == m)) {
                        const uint32_t a = cnt & 1;
                        if (!mbar_wait(bar.at(L::kBarAccEmpty + a * 2 + m), ((cnt >> 1) & 1) ^ 1, abort_flag, sink)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t d_tmem = tmem_base + a * 256 + m * 128;
                        if (D == 128) umma_tile_k128(d_tmem, resident, stage, idesc_k);
                        else umma_tile_row128<kCodes>(d_tmem, resident, stage, idesc_k);
                        // ... - (T / r_i) (||k_j|| + eps): the accumulator's sign is the threshold test
                        umma_k16_sw32(d_tmem, res_slice, sbase + L::kOffAugB + s * kSliceBytes, idesc_s);
                        umma_commit(bar.at(L::kBarAccFull + a * 2 + m));
                        ++cnt;
                        ++tiles_done;
                        umma_commit(bar.at(L::kBarBEmpty + s));      // the stage may be refilled once these products have read it
                    } else {
                        mbar_arrive(bar.at(L::kBarBEmpty + s));
                    }
                    ++bcount;
                }
                if (!ok) break;
                for (int x = 0; x < num_m; ++x) {                    // so may the resident tiles
                    const uint32_t u = use + (uint32_t)x;
                    if (u > own && !mbar_wait(bar.at(L::kBarAFull + buf_of(u)), phase_of(u), abort_flag, sink)) ok = false;
                    if (mine && u == own) umma_commit(bar.at(L::kBarAEmpty + buf_of(u)));
                    else mbar_arrive(bar.at(L::kBarAEmpty + buf_of(u)));
                }
                use += (uint32_t)num_m;
                ++k_item;
            }
        }
        __syncwarp();
    } else if (warp >= kGatherWarp0) {
        // ------------------------------------------------------------------ gather warps
        // They run as far ahead of the scan as there are resident tiles that it does not use: the listed tokens' key rows go into
        // the next of them (same swizzled layout as a TMA load), each row's extra slice beside them, and what the epilogue needs
        // to know about the token into the stash.  Thread g serves rows g and g + 128 of the item.
        const int gt = (warp - kGatherWarp0) * 32 + lane;      // 0..127
        uint32_t k_item = 0, use = 0;
        bool ok = true;
        while (ok) {
            const uint32_t qs = k_item % kItemSlots;
            if (!mbar_wait(bar.at(L::kBarQFull + qs), (k_item / kItemSlots) & 1, abort_flag, sink)) break;
            const int4 d = items[qs];
            __syncwarp();
            if (lane == 0) mbar_arrive(bar.at(L::kBarQEmpty + qs));
            if (d.x < 0) break;
            const int head = d.x, k0 = d.y, rows = d.z & 0xffff;
            const int num_m = rows > kTile ? 2 : 1;
            const size_t hoff = (size_t)head * p.cap_pad;
            int pos[2];
            float rr[2];
            int lf[2];
#pragma unroll
            for (int m = 0; m < 2; ++m) pos[m] = (m * kTile + gt < rows) ? p.strag[hoff + k0 + m * kTile + gt] : -1;
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                rr[m] = pos[m] >= 0 ? __ldg(p.inv_norm + hoff + pos[m]) : 0.f;
                lf[m] = pos[m] >= 0 ? (kOne ? 1 : p.left[hoff + pos[m]]) : 0;
            }
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                if (m >= num_m || !ok) break;
                const bool row_ok = pos[m] >= 0;
                const uint4 *src = reinterpret_cast<const uint4 *>(
                    static_cast<const __nv_bfloat16 *>(p.k_cache) + (size_t)row_index(p, head, row_ok ? pos[m] : 0) * D);
                uint4 v[D / 8];                      // under way while the tile is still in use
#pragma unroll
                for (int c = 0; c < D / 8; ++c) v[c] = row_ok ? __ldg(src + c) : make_uint4(0u, 0u, 0u, 0u);
                const uint32_t ab = buf_of(use);
                if (!(ok = mbar_wait(bar.at(L::kBarAEmpty + ab), phase_of(use) ^ 1u, abort_flag, sink))) break;
                ++use;
                uint8_t *tile = smem + L::kOffA + ab * L::kTileBytes;
#pragma unroll
                for (int hb = 0; hb < D / 64; ++hb) {
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        *reinterpret_cast<uint4 *>(tile + hb * kHalfBytes + gt * 128 + ((c ^ (gt & 7)) << 4)) = v[hb * 8 + c];
                }
                // the row's extra slice: -T / r_i in three bf16 parts as (-t1, -t1, -t1, -t2, -t2, -t3, 0 ...),
                // which meets (n1, n2, n3, n1, n2, n1, 0 ...) of a key; 32-byte rows, 32-byte swizzle
                float rest = (row_ok && rr[m] > 0.f) ? -__fdiv_rn(p.sim_threshold, rr[m]) : 0.f;
                uint32_t part[3];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const __nv_bfloat16 h16 = __float2bfloat16_rn(rest);
                    part[c] = (uint32_t)__bfloat16_as_ushort(h16);
                    rest -= __bfloat162float(h16);
                }
                uint8_t *slice = smem + L::kOffAugA + ab * kSliceBytes + gt * 32;
                const int sw = (gt >> 2) & 1;
                *reinterpret_cast<uint4 *>(slice + (sw << 4)) =
                    make_uint4(part[0] | (part[0] << 16), part[0] | (part[1] << 16), part[1] | (part[2] << 16), 0u);
                *reinterpret_cast<uint4 *>(slice + ((sw ^ 1) << 4)) = make_uint4(0u, 0u, 0u, 0u);
                int32_t *stash = reinterpret_cast<int32_t *>(smem + L::kOffStash + ab * 3 * kTile * 4);
                stash[gt] = row_ok ? pos[m] : 0;
                reinterpret_cast<float *>(stash)[kTile + gt] = rr[m];
                stash[2 * kTile + gt] = lf[m];
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> tensor-core reads
                __syncwarp();
                if (lane == 0) mbar_arrive(bar.at(L::kBarAFull + ab));
            }
            ++k_item;
        }
    } else {
        // ------------------------------------------------------------------ epilogue warps
        const int ew = warp - 2;                 // 0..7
        const int m = ew >> 2;                   // row tile of the item this warp serves, or half of the key tiles of an item of one
        const int quad = warp & 3;               // TMEM lane quadrant this warp may access
        const int lrow = quad * 32 + lane;       // row within the 128-row tile
        const uint32_t lane_base = tmem_base + ((uint32_t)(quad * 32) << 16);
        uint32_t k_item = 0, cnt = 0, use = 0, merges = 0;      // merges: items of one row tile so far

        while (true) {
            const uint32_t qs = k_item % kItemSlots;
            if (!mbar_wait(bar.at(L::kBarQFull + qs), (k_item / kItemSlots) & 1, abort_flag, sink)) break;
            const int4 d = items[qs];
            __syncwarp();
            if (lane == 0) mbar_arrive(bar.at(L::kBarQEmpty + qs));
            if (d.x < 0) break;
            const int head = d.x;
            const float *inv_norm = p.inv_norm + (size_t)head * p.cap_pad;
            // ---- per item: which token this thread owns (left in the stash by the gather warps), where the scan
            // starts and ends
            const int rows = d.z & 0xffff, first_tile = d.w, last_tile = d.w - (d.z >> 16) + 1;
            const bool split = kOne && rows <= kTile;
            const bool active = (m == 0) || (rows > kTile) || split;
            const int r_item = split ? lrow : m * kTile + lrow;               // row of the item
            const bool row_ok = active && r_item < rows;
            // the resident tile (and stash) whose rows these warps look after; the other one's barrier is met at the item's end, or here
            const uint32_t num_m = rows > kTile ? 2u : 1u, own = use + (num_m == 2u && m == 1 ? 1u : 0u);
            bool item_ok = mbar_wait(bar.at(L::kBarAFull + buf_of(use)), phase_of(use), abort_flag, sink);
            if (own != use && item_ok) item_ok = mbar_wait(bar.at(L::kBarAFull + buf_of(own)), phase_of(own), abort_flag, sink);
            const int32_t *stash = reinterpret_cast<const int32_t *>(smem + L::kOffStash + buf_of(own) * 3 * kTile * 4);
            int i = 0, left = 0;
            float ri = 0.f;
            if (row_ok && item_ok) {
                i = stash[lrow];
                ri = reinterpret_cast<const float *>(stash)[kTile + lrow];
                left = stash[2 * kTile + lrow];
            }

            float removed = 0.f;
            // how many partners were found; with beta = 1 the one partner's position and accumulator value
            int nhit = 0, hit_j = -1;
            float hit_h = 0.f;
            if (active) {
                // ---- key tiles of the window, last to first
                bool ok = item_ok;
                for (int jt = first_tile - (split ? m : 0); jt >= last_tile; jt -= split ? 2 : 1) {
                    const int jbase = jt * kTile;
                    // with beta > 1 the partners' values need the tile's r_j: lane l has those of columns l, 32 + l, ..., under way
                    // while the product is
                    float rj[4] = {0.f, 0.f, 0.f, 0.f};
                    if (!kOne) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) rj[q] = __ldg(inv_norm + jbase + q * 32 + lane);
                    }
                    const uint32_t a = cnt & 1;
                    if (ok) ok = mbar_wait(bar.at(L::kBarAccFull + a * 2 + m), (cnt >> 1) & 1, abort_flag, sink);
                    ++cnt;
                    if (!ok) continue;
                    tc_fence_after();
                    const uint32_t base = lane_base + a * 256 + m * 128;
                    // a token that has its beta partners screens nothing any more
                    bool want = left > 0;
                    // The accumulator holds h = k_i . k_j - (T / r_i) (||k_j|| + eps): S[j][i] > T exactly when h > 0, so
                    // the screening is a sign test, with nothing to load per column (loads of the r_j were what this
                    // epilogue's time went into: every byte a thread receives, from TMEM or as a shared-memory
                    // broadcast, passes through the same return path).
                    auto chunk = [&](const uint32_t (&g)[32], int ch) {
                        uint32_t colmask = 0xffffffffu;
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
                        // entries with a clear sign bit (h > 0, but also +0: confirmed one by one below)
                        uint32_t pos = want ? (~neg & colmask) : 0u;
                        if (kOne) {
                            // one partner at most: the candidate at the highest set bit, its value picked by a select
                            // tree (nearly always a single turn); its r_j is fetched once, at the item's end
                            while (pos != 0u) {
                                const int top = 31 - __clz(pos);
                                const float hv = pick32(g, top);
                                if (hv > 0.f) {
                                    hit_h = hv;
                                    hit_j = jbase + ch * 32 + top;
                                    left = 0;
                                    want = false;
                                    break;
                                }
                                pos &= ~(1u << top);
                            }
                        } else {
                            // several: S = T + h r_i r_j each, a turn per partner, the warp together (4096 heads of 1068 tokens with
                            // beta = 4: the pass took 1020 us while every column of a chunk that holds a partner was compared,
                            // multiplied by an r_j loaded then and summed; 603 now)
                            while (__any_sync(0xffffffffu, pos != 0u)) {
                                const int top = 31 - __clz((int)(pos | 1u));
                                const float r = __shfl_sync(0xffffffffu, rj[ch], top);
                                const float hv = pick32(g, top);
                                if (pos != 0u && hv > 0.f) {
                                    removed += hv * r;
                                    ++nhit;
                                    --left;
                                }
                                pos = left == 0 ? 0u : pos & ~(1u << top);
                            }
                            want = left > 0;
                        }
                    };
                    // 32-column chunks, last first; the TMEM load of the next chunk is issued before the current one is looked at (two
                    // register sets, used alternately).  What this takes is integer instructions (two cycles each) and their fetch:
                    // longer loads, or a conjunction of signs first and the chunks it names loaded again, were slower with beta = 1.
                    if (__any_sync(0xffffffffu, want)) {
                        uint32_t ga[32], gb[32];
                        tmem_ld32(base + 96, ga);
                        tmem_wait32(ga);
                        tmem_ld32(base + 64, gb);
                        chunk(ga, 3);
                        tmem_wait32(gb);
                        tmem_ld32(base + 32, ga);
                        chunk(gb, 2);
                        tmem_wait32(ga);
                        tmem_ld32(base, gb);
                        chunk(ga, 1);
                        tmem_wait32(gb);
                        chunk(gb, 0);
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar.at(L::kBarAccEmpty + a * 2 + m));
                }
                item_ok = ok;
            }
            if (split && item_ok) {
                int32_t *found_j = reinterpret_cast<int32_t *>(smem + L::kOffMerge + buf_of(merges) * 2 * kTile * 4);
                float *found_h = reinterpret_cast<float *>(found_j + kTile);
                const uint32_t merge = bar.at(L::kBarMerge + (int)buf_of(merges));
                if (m == 1) {                        // the second half leaves its findings
                    found_j[lrow] = hit_j;
                    found_h[lrow] = hit_h;
                    __syncwarp();
                    if (lane == 0) mbar_arrive(merge);
                } else {
                    item_ok = mbar_wait(merge, phase_of(merges), abort_flag, sink);
                    if (item_ok && found_j[lrow] > hit_j) {
                        hit_j = found_j[lrow];
                        hit_h = found_h[lrow];
                    }
                }
            }
            if (split) ++merges;
            if (own == use && num_m == 2u && item_ok) item_ok = mbar_wait(bar.at(L::kBarAFull + buf_of(use + 1u)), phase_of(use + 1u), abort_flag, sink);
            // the item's resident tiles and stash are no longer read by this warp
            __syncwarp();
            if (lane == 0 && item_ok)
                for (uint32_t x = 0; x < num_m; ++x) mbar_arrive(bar.at(L::kBarAEmpty + buf_of(use + x)));
            use += num_m;
            if (!item_ok) break;              // (the epilogue warps meet at no barrier of their own: each may leave alone)
            if (row_ok && !(split && m == 1)) {
                // S = T + h r_i r_j for every partner found here
                if (kOne && hit_j >= 0) {
                    left = 0;
                    removed = hit_h * __ldg(inv_norm + hit_j);
                    nhit = 1;
                }
                if (nhit > 0) {
                    p.sbar[(size_t)head * p.cap_pad + i] -= (float)nhit * p.sim_threshold + removed * ri;
                    if (!kOne) p.left[(size_t)head * p.cap_pad + i] = left;
                    // the next round lists the tokens still short
                    if (left == 0) atomicAnd(p.lacking + (((size_t)head * p.cap_pad + i) >> 5), ~(1u << (i & 31)));
                }
            }
            ++k_item;
        }
    }

    // ---------------------------------------------------------------------- common exit
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        if (*abort_flag) __nanosleep(200000);      // error path only: let copies and MMAs in flight land
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
    if ((warp == 1 || warp == 10) && lane == 0 && !*abort_flag && tiles_done) atomicAdd(p.counters, tiles_done);
}

// ---- before every round: list, per head, the tokens still short of partners, and cut the list into work items ----
constexpr int kCompactWarps = 8;         // of a block; one or four per head
constexpr int kDenseMinTiles = 12;       // caches of fewer key tiles never take the symmetric route (two more launches)

// The tokens are given as one bit each, 32 to a word, so a list costs a head's 33 words per 1024 tokens and what it writes.
// (Read from a word per token by a block per head, a listing of 4096 heads of 4216 tokens took 81 us; 37 with bits.  The counters
// took part of that: three atomics per head on one line of memory.  A block adds its heads' up first: 33; 8192 heads of 2168
// tokens 35 -> 25.)  kHeadWarps: four warps share the words of a head where there are few heads -- one warp's turns over them are
// then what a call waits for (256 heads of 1144 tokens: 12 -> 8 us) --, one takes them all where blocks with more heads, and
// so fewer atomics, count for more (with two heads a block 8192 took 50 us).
// `below`: key tiles under the first pass's part that earlier rounds have covered; `width`: tiles of this round's
// window (the last round passes a width that reaches tile 0 whatever the cache size).
template <int kHeadWarps>
__global__ void __launch_bounds__(kCompactWarps * 32) strag_compact_kernel(Params p, int round, int below, int width)
{
    constexpr int kCompactHeads = kCompactWarps / kHeadWarps, kWordsPerLane = RKV_MAX_CAP / 32 / (32 * kHeadWarps);
    pdl_trigger();
    pdl_wait();
    __shared__ int warp_count[kCompactWarps], block_chunks[kCompactHeads];
    __shared__ unsigned long long block_pairs[kCompactHeads], block_slot;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int mate = warp / kHeadWarps, part = warp % kHeadWarps;        // which head of the block, which part of its words
    const int head = blockIdx.x * kCompactHeads + mate;
    const bool head_ok = head < p.batch * p.hkv;
    const int n = head_ok ? seq_candidates(p, head / p.hkv) : 0;
    int32_t *list = p.strag + (size_t)head * p.cap_pad;
    // the first pass scanned every token against the last kPass1Depth key tiles; this round starts `below` tiles
    // under that
    const int n_tiles = (n + kTile - 1) / kTile;
    const int first_tile = n_tiles - kPass1Depth - 1 - below, n_iter = min(width, first_tile + 1);
    // a head without anything left to scan, or one that went to the symmetric route, lists nothing; nor does a call that has given up
    const bool scans = head_ok && first_tile >= 0 && !call_aborted(p) && !(round > 0 && p.dense[head]);
    const int words = scans ? (n + 31) / 32 : 0, per_warp = (words + kHeadWarps - 1) / kHeadWarps, word0 = part * per_warp;
    const int my_words = min(per_warp, words - word0);
    const uint32_t *bits = p.lacking + (size_t)head * (p.cap_pad / 32) + word0;
    uint32_t word[kWordsPerLane];
    int my_count = 0;
#pragma unroll
    for (int k = 0; k < kWordsPerLane; ++k) {
        word[k] = k * 32 + lane < my_words ? bits[k * 32 + lane] : 0u;
        my_count += __popc(word[k]);
    }
    my_count = __reduce_add_sync(0xffffffffu, my_count);
    if (lane == 0) warp_count[warp] = my_count;
    __syncthreads();
    int count = 0, at = 0;                   // the head's listed tokens; those of the parts before this one
#pragma unroll
    for (int w = 0; w < kHeadWarps; ++w) {
        count += warp_count[mate * kHeadWarps + w];
        at += w < part ? warp_count[mate * kHeadWarps + w] : 0;
    }
    const bool speaks = head_ok && part == 0 && lane == 0;               // for its head
    if (speaks && !scans && round == 0) p.dense[head] = 0;
    if (scans && round == 0) {
        // Most tokens still lack a partner (few pairs exceed T): the rounds would form nearly the whole matrix for this
        // head.  It goes to the symmetric route instead, which forms each tile pair once.
        const bool dense = p.dense_ok && n_tiles >= kDenseMinTiles && 5 * count > 4 * n;
        if (speaks) p.dense[head] = dense ? 1 : 0;
        if (dense) {
            uint4 *best = reinterpret_cast<uint4 *>(p.best + (size_t)head * p.cap_pad);
            for (int i = part * 32 + lane; i < p.cap_pad / 4; i += 32 * kHeadWarps) best[i] = make_uint4(0u, 0u, 0u, 0u);
            const int pairs_of_tiles = (n_tiles + 1) / 2;
            if (part == 0) {
                unsigned long long slot = 0ull;
                if (lane == 0) {
                    slot = atomicAdd(&p.counters[kDenseWords], (unsigned long long)pairs_of_tiles);
                    // useful work: every unordered pair of the listed tokens' tiles once
                    atomicAdd(&p.counters[kPairsWord], (unsigned long long)count * (unsigned long long)(n_tiles + 1) / 2ull);
                }
                slot = __shfl_sync(0xffffffffu, slot, 0);
                for (int q = lane; q < pairs_of_tiles; q += 32) p.dense_items[slot + q] = make_int4(head, q, n, 0);   // longest first
            }
            count = 0;                       // nothing for the rounds
        }
    }
    const int chunks = (count + kRowsPerItem - 1) / kRowsPerItem;
    if (part == 0 && lane == 0) {
        block_chunks[mate] = chunks;
        block_pairs[mate] = (unsigned long long)count * (unsigned long long)n_iter;    // the work the round cannot avoid
    }
    __syncthreads();
    if (threadIdx.x == 0) {                  // the block's place in the work list, under way while the lists are written
        int total = 0;
        unsigned long long pairs = 0ull;
#pragma unroll
        for (int w = 0; w < kCompactHeads; ++w) {
            total += block_chunks[w];
            pairs += block_chunks[w] > 0 ? block_pairs[w] : 0ull;
        }
        if (total > 0) {
            block_slot = atomicAdd(&p.counters[kRoundWords + 2 * round], (unsigned long long)total);
            atomicAdd(&p.counters[2], (unsigned long long)total);
            atomicAdd(&p.counters[kPairsWord], pairs);
        }
    }
    if (count > 0) {                         // ascending positions
#pragma unroll
        for (int k = 0; k < kWordsPerLane; ++k) {
            if (k * 32 >= my_words) break;
            const int mine = __popc(word[k]);
            int incl = mine;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int o = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += o;
            }
            const int first = at + incl - mine;
            for (unsigned todo = __ballot_sync(0xffffffffu, mine > 0); todo != 0u; todo &= todo - 1u) {
                const int src = __ffs(todo) - 1;
                const uint32_t w = __shfl_sync(0xffffffffu, word[k], src);
                const int f = __shfl_sync(0xffffffffu, first, src);
                if (w >> lane & 1u) list[f + __popc(w & ((1u << lane) - 1u))] = (word0 + k * 32 + src) * 32 + lane;
            }
            at += __shfl_sync(0xffffffffu, incl, 31);
        }
    }
    __syncthreads();
    int before = 0;
    for (int w = 0; w < mate; ++w) before += block_chunks[w];
    for (int q = part * 32 + lane; q < chunks; q += 32 * kHeadWarps) {
        const int k0 = q * kRowsPerItem;
        p.strag_items[block_slot + before + q] = make_int4(head, k0, min(count - k0, kRowsPerItem) | (n_iter << 16), first_tile);
    }
}

}  // namespace

bool scores_dense_possible(int tiles, int beta) { return beta == 1 && tiles >= kDenseMinTiles; }

int scores_pass2_rounds(int tiles)
{
    const int below = tiles - kPass1Depth;      // key tiles under the first pass's part, at most
    return below <= 8 ? 1 : 2;
}

template <int D, bool kCodes, bool kOne>
static cudaError_t launch_tri_for(const Params &p, cudaStream_t s)
{
    CUtensorMap map_k, map_hs, map_ns, map_ts;
    const uint64_t sum_rows = (uint64_t)p.batch * p.hkv * (kCodes ? kSumHeadBytes / 128 : 16);
    const bool keys_ok = kCodes ? make_map_row128(&map_k, p.k_cache, key_rows_total(p), true) &&
                                      encode_map(&map_hs, MapKey{p.head_sum_bf16, sum_rows, CU_TENSOR_MAP_DATA_TYPE_UINT8, 128u, 128u, 128u, 16u, CU_TENSOR_MAP_SWIZZLE_128B})
                                : make_map_rows(&map_k, p.k_cache, key_rows_total(p), D, kTile) && make_map_rows(&map_hs, p.head_sum_bf16, sum_rows, D, 16u);
    if (!keys_ok ||
        !make_map_k16(&map_ns, p.norm_split, (uint64_t)p.batch * p.hkv * p.cap_pad) ||
        !make_map_k16(&map_ts, p.thr_split, (uint64_t)p.batch * p.hkv * kTile))
        return cudaErrorInvalidValue;
    cudaError_t e;
    static PerDevice done;
    int dev = 0, sms = 0;
    if ((e = device_sms(&dev, &sms)) != cudaSuccess || (e = allow_smem_once(done, dev, scores_pass2_sm100_kernel<D, kCodes, kOne>, Lay<D>::kSmemBytes)) != cudaSuccess)
        return e;
    const int heads = p.batch * p.hkv;
    if ((e = launch_scores_pass1_sm100(p, s, map_k, map_hs, map_ns, map_ts)) != cudaSuccess) return e;
    if ((e = mark_kernel(p, 0, s)) != cudaSuccess) return e;
    const bool rule_on = p.beta > 0 && p.sim_threshold < 1.0f;
    if (!rule_on || p.tiles < 2) return mark_kernel(p, 1, s);       // nobody can lack partners / the first pass has seen everything
    const unsigned long long max_items2 = (unsigned long long)heads * (unsigned long long)(p.cap_pad / kRowsPerItem + 1);
    const unsigned grid2 = (unsigned)(max_items2 < (unsigned long long)sms ? max_items2 : (unsigned long long)sms);
    // rounds of the second pass: short windows first, so that the tokens that find their partners soon drop out
    // before the long scan down to tile 0
    const int rounds = scores_pass2_rounds(p.tiles);
    static const int kRoundTiles[2] = {6, 1 << 20};      // (measured: 6 + rest beats 4 + 8 + rest and 8 + rest by a little)
    const bool dense_possible = p.dense_ok && p.tiles >= kDenseMinTiles;
    int below = 0;
    for (int r = 0; r < rounds; ++r) {
        const int width = r == rounds - 1 ? (1 << 20) : kRoundTiles[r];
        e = heads <= 4 * sms ? launch_early(strag_compact_kernel<4>, (unsigned)((heads + kCompactWarps / 4 - 1) / (kCompactWarps / 4)), kCompactWarps * 32, 0, s, 1, p, r, below, width)
                             : launch_early(strag_compact_kernel<1>, (unsigned)((heads + kCompactWarps - 1) / kCompactWarps), kCompactWarps * 32, 0, s, 1, p, r, below, width);
        if (e != cudaSuccess) return e;
        if (r == 0 && (e = mark_kernel(p, 1, s)) != cudaSuccess) return e;
        if ((e = launch_early(scores_pass2_sm100_kernel<D, kCodes, kOne>, grid2, kThreads, Lay<D>::kSmemBytes, s, 1, p, map_k, map_ns, r)) != cudaSuccess) return e;
        // the heads the first listing sent to the symmetric route (none on inputs where similar keys are common:
        // the kernel then returns at once)
        if (r == 0 && dense_possible && (e = launch_scores_dense_sm100(p, s, map_k, map_ns)) != cudaSuccess) return e;
        below += width;
    }
    return dense_possible ? launch_dense_finish(p, s) : cudaSuccess;
}

cudaError_t launch_scores_tri_sm100(const Params &p, cudaStream_t s)
{
    const bool one = p.beta == 1;
    if (p.codes) return one ? launch_tri_for<64, true, true>(p, s) : launch_tri_for<64, true, false>(p, s);
    if (p.d == 64) return one ? launch_tri_for<64, false, true>(p, s) : launch_tri_for<64, false, false>(p, s);
    return one ? launch_tri_for<128, false, true>(p, s) : launch_tri_for<128, false, false>(p, s);
}

}  // namespace rkv
