// Stage "prep": one streaming pass over the candidate keys.
//
// For every key row i of every head it produces r_i = 1 / (||k_i||_2 + eps), the normalisation
// factor of Eq. 5, and per 128-row tile the vector sum_i r_i * k_i.  The tile sums let the
// scoring stage obtain sum_j S[j][i] = Kbar_i . (sum_j Kbar_j) - Kbar_i . Kbar_i (Eq. 6 before the
// retention rule) without accumulating the n x n matrix element by element.
// Rows i >= n (observation tokens, unused capacity) get r_i = 0 and contribute nothing.
// The call's counters start at zero: the first block clears them (a memset in front of this kernel cost a small call 3 us).
// The abort word is among them, so no block of these kernels sets it: nothing would order that against the first block's
// store.  A block that gives up on a wait leaves kGaveUp as the first r of every tile that it has not finished instead, and
// the kernel that reads the norms next (head_sum_kernel, the CUDA-core kernel, the row-block kernel) records the abort.
// Kbar_i . Kbar_i is kept per row as well (self_dot).
//
// HBM-bound: each block brings its tile of K into shared memory with one bulk copy (cp.async.bulk, bounded wait
// on its mbarrier) and reads it from there; the row norm is reduced with warp shuffles.  Outputs are 8 bytes per
// 256-byte row.
#include <algorithm>

#include "rkv_sm100.cuh"

namespace rkv {

namespace {

__device__ __forceinline__ void clear_counters(const Params &p)
{
    if (blockIdx.x == 0 && threadIdx.x < kCounterWords) p.counters[threadIdx.x] = 0ull;
}

// Where the waits of the prep kernels record that they ran out: the caller's status, but not the abort word (see above).
__device__ __forceinline__ ErrSink prep_sink(const Params &p) { return ErrSink{p.status, nullptr, p.wait_cycles}; }

// Error path: one thread waits for what its block still has under way before the block's memory is given up, however short the
// caller's own limit is.
__device__ __forceinline__ void drain(uint32_t bar, uint32_t parity)
{
    const long long start = clock64();
    while (!sm100::mbar_try_wait_asleep(bar, parity))
        if (clock64() - start > sm100::kWaitCycles) return;
}

constexpr int kPrepThreads = 256;
constexpr int kPrepWarps = kPrepThreads / 32;

template <typename T, int D>
__global__ void __launch_bounds__(kPrepThreads, D <= 128 ? 5 : 2) prep_kernel(Params p)
{
    using namespace sm100;
    extern __shared__ __align__(128) uint8_t prep_smem[];       // the tile's candidate rows, then one mbarrier
    constexpr int kTileBytesT = kTile * D * (int)sizeof(T);
    __shared__ int abort_flag;
    const ErrSink sink = prep_sink(p);
    pdl_trigger();
    pdl_wait();
    clear_counters(p);
    constexpr int kPerVec = Elem<T>::kPerVec;            // elements per 16-byte vector
    constexpr int kVecPerLane = 2;                       // 16-byte vectors of a row held by one lane
    constexpr int kLanesPerRow = D / (kPerVec * kVecPerLane);     // 8 (bf16) or 16 (fp32)
    constexpr int kVecPerRow = D / kPerVec;
    constexpr int kRowsPerPass = 32 / kLanesPerRow;      // rows a warp covers with one load
    constexpr int kRowsPerWarp = kTile / kPrepWarps;     // 16
    constexpr int kPasses = kRowsPerWarp / kRowsPerPass;

    const int tile = blockIdx.x % p.tiles;
    const int head = blockIdx.x / p.tiles;               // head-problem index b * hkv + h
    const int b = head / p.hkv;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    int L = p.seq_lens[b];
    int budget_b = p.budgets ? p.budgets[b] : p.budget;             // Section 4.2's per-sequence (ratio) budgets
    if (L < 0 || L > p.cap || budget_b <= p.alpha || budget_b > p.budget) {
        report(p.status, RKV_ERR_INVALID_ARG);
        L = kMetaInvalid;
        budget_b = p.budget;
    }
    if (tile == 0 && head % p.hkv == 0 && threadIdx.x == 0) {
        p.meta[b] = L;
        p.meta[p.batch + b] = budget_b;
    }
    const int n = candidates_from_meta(L, budget_b, p.alpha);

    const T *K_tile = static_cast<const T *>(p.k_cache) + (size_t)tile_row0(p, head, tile) * D;      // the tile's first row
    float *inv_norm = p.inv_norm + (size_t)head * p.cap_pad;

    const int sub = lane / kLanesPerRow;                 // which of the rows of this pass
    const int lane_in_row = lane % kLanesPerRow;         // vector u of the lane = vector lane_in_row + u * kLanesPerRow
                                                         // of the row: a warp's load covers whole 128-byte lines

    // One bulk copy brings the tile's candidate rows (contiguous in memory) into shared memory: the bytes in
    // flight cost no registers, so several blocks per SM keep HBM busy.
    const int rows_here = min(max(n - tile * kTile, 0), kTile);
    const uint32_t bar = smem_u32(prep_smem + kTileBytesT);
    if (threadIdx.x == 0) {
        abort_flag = 0;
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (rows_here > 0) {
            const uint32_t bytes = (uint32_t)rows_here * D * (uint32_t)sizeof(T);
            mbar_expect_tx(bar, bytes);
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(smem_u32(prep_smem)), "l"(K_tile), "r"(bytes), "r"(bar)
                         : "memory");
        }
    }
    __syncthreads();
    const bool landed = rows_here == 0 || mbar_wait(bar, 0, &abort_flag, sink);
    if (!__syncthreads_and(landed)) {      // the block leaves as a whole, or not at all
        if (threadIdx.x == 0) {
            inv_norm[tile * kTile] = kGaveUp;
            drain(bar, 0);
        }
        return;
    }
    const uint4 *tile_s = reinterpret_cast<const uint4 *>(prep_smem);
    // packed fp32 arithmetic (two values per instruction), few lanes per row (short shuffle trees): this kernel is
    // bound by its instruction count
    constexpr int kHeld = kPerVec * kVecPerLane;         // elements of a row per lane
    float2 acc2[kHeld / 2];
#pragma unroll
    for (int e = 0; e < kHeld / 2; ++e) acc2[e] = make_float2(0.f, 0.f);

#pragma unroll
    for (int q = 0; q < kPasses; ++q) {
        const int lr = warp * kRowsPerWarp + q * kRowsPerPass + sub;       // row within the tile
        const int row = tile * kTile + lr;
        float f[kHeld];
#pragma unroll
        for (int u = 0; u < kVecPerLane; ++u) {
            uint4 vec = make_uint4(0u, 0u, 0u, 0u);
            if (lr < rows_here) vec = tile_s[lr * kVecPerRow + lane_in_row + u * kLanesPerRow];
            Elem<T>::unpack(vec, f + u * kPerVec);
        }
        float2 sq2 = make_float2(0.f, 0.f);
#pragma unroll
        for (int e = 0; e < kHeld / 2; ++e) {
            const float2 f2 = make_float2(f[2 * e], f[2 * e + 1]);
            sq2 = __ffma2_rn(f2, f2, sq2);
        }
        float sq = sq2.x + sq2.y;
#pragma unroll
        for (int off = kLanesPerRow / 2; off > 0; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
        // 1 / (sqrt(sq) + eps) from the hardware's approximate rsqrt and divide (a few ulp: far inside the score
        // tolerances, and every scoring kernel uses these same r); sq = 0 (an all-zero key) gives 1 / eps
        const float nrm = sq > 0.f ? sq * rsqrtf(sq) : 0.f;
        const float r = (row < n) ? __fdividef(1.0f, nrm + p.eps) : 0.f;
        if (lane_in_row == 0) {
            inv_norm[row] = r;                       // row < cap_pad: the grid covers exactly cap_pad rows per head
            p.self_dot[(size_t)head * p.cap_pad + row] = (r * r) * sq;     // Kbar_i . Kbar_i
        }
        const float2 r2 = make_float2(r, r);
#pragma unroll
        for (int e = 0; e < kHeld / 2; ++e) acc2[e] = __ffma2_rn(r2, make_float2(f[2 * e], f[2 * e + 1]), acc2[e]);
    }

    // fold the row groups of a warp, then the warps, in a fixed order (deterministic sums)
#pragma unroll
    for (int off = kLanesPerRow; off < 32; off <<= 1) {
#pragma unroll
        for (int e = 0; e < kHeld / 2; ++e) {
            acc2[e].x += __shfl_xor_sync(0xffffffffu, acc2[e].x, off);
            acc2[e].y += __shfl_xor_sync(0xffffffffu, acc2[e].y, off);
        }
    }
    __shared__ float part[kPrepWarps][D];
    if (sub == 0) {
#pragma unroll
        for (int u = 0; u < kVecPerLane; ++u) {
            const int col = (lane_in_row + u * kLanesPerRow) * kPerVec;
#pragma unroll
            for (int e = 0; e < kPerVec / 2; ++e) {
                part[warp][col + 2 * e] = acc2[u * kPerVec / 2 + e].x;
                part[warp][col + 2 * e + 1] = acc2[u * kPerVec / 2 + e].y;
            }
        }
    }
    __syncthreads();
    if (threadIdx.x < D) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < kPrepWarps; ++w) s += part[w][threadIdx.x];
        p.tile_sum[((size_t)head * p.tiles + tile) * D + threadIdx.x] = s;
    }
}

// ---- the same stage for bf16 caches with d = 64 or 128 (the tensor-core route): sum_i r_i k_i on the tensor cores -------
//
// The norms stay on the CUDA cores, one thread per row (the row read from shared memory once, packed fp32).  The
// weighted column sums sum_i r_i k_i[c] -- what made the kernel above instruction-bound -- are ONE small tensor-core
// product per tile: the key tile as TMA leaves it (rows of 128 d-elements, 128-byte swizzle) is used TRANSPOSED as the A
// operand (MN-major: M = d, K = the 128 rows), the B operand holds r_i in three bf16 parts (N = 16, rows 0..2), so
// D[c][0..2] sum to sum_i r_i k_i[c] to fp32 accuracy.  Eight K = 16 steps, accumulator = 16 TMEM columns.
//
// 64 dimensions: a unit of work is two tiles of a head, one behind the other in the same 32 KB.  They are the two halves of
// M, their r_i are rows 0..2 and 3..5 of the B operand, and each half of the lanes reads its own three columns.  (One tile
// per unit would leave half the bytes in flight for the same chain of waits.  8192 heads of 2168 tokens: 1276 us while the
// keys were written out once more, padded to 128 dimensions, for kernels that knew no other size; 537 now.)
//
// The threshold test of Section 3.3, S[j][i] > T, as the sign of k_i . k_j - T / (r_i r_j): the tensor-core kernels
// append one K = 16 step to a tile product whose operands are these slices.  1 / r = ||k|| + eps in three bf16
// parts (their sum has fp32 accuracy) as (n1, n2, n3, n1, n2, n1, 0 ...) for a key row; its dot product with a
// row's (-t1, -t1, -t1, -t2, -t2, -t3, 0 ...), the parts of T / r, is -T / (r_i r_j) up to terms of size 2^-24.
constexpr int kPrepTcThreads = 128;                         // one thread per row of the tile
constexpr int kPrepTcTile = kTile * kHeadDim * 2;          // a unit: 32 KB, one tile of 128 dimensions or two of 64
constexpr int kPrepTcB = 8 * 16 * 32;                      // 8 K-steps x [16 n][16 k] bf16, 32-byte rows (32-byte swizzle)
constexpr int kPrepTcBufs = 2;                             // tile buffers of a block: one in use, the others being filled
constexpr int kPrepTcBlocks = 3;                           // blocks per SM
constexpr int kPrepTcSmem = kPrepTcBufs * kPrepTcTile + kPrepTcB + 1024; // + slack for the 1024-byte alignment
constexpr uint32_t kPrepTcTmemCols = 32;

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

// bf16 caches of 64 dimensions: the lengths are recorded and the counters cleared ahead of the prep kernel.
constexpr int kLengthThreads = 256;
__global__ void __launch_bounds__(kLengthThreads) lengths_kernel(Params p)
{
    pdl_trigger();
    pdl_wait();
    clear_counters(p);
    const int b = blockIdx.x * kLengthThreads + threadIdx.x;
    if (b < p.batch) prep_unit_at<1>(p, b * p.hkv * p.tiles, true);
}

// Persistent: kPrepTcBlocks blocks per SM, block x takes tiles x, x + gridDim.x, ... of the list (head-major) and
// keeps the copies of its next kPrepTcBufs - 1 tiles in flight while it works on the present one: what bounds this
// kernel is how many bytes an SM has under way, not what it does with them.  Barriers, the TMEM columns and the tensor
// map are set up once per block.
template <int D>
__global__ void __launch_bounds__(kPrepTcThreads, kPrepTcBlocks) prep_tc_kernel(Params p, const __grid_constant__ CUtensorMap map_k, int total)
{
    using namespace sm100;
    constexpr int kSub = kHeadDim / D;                       // tiles of a unit
    constexpr int kChunks = D / 8;                           // 16-byte vectors of a row
    extern __shared__ uint8_t prep_tc_raw[];
    uint8_t *smem = align_smem(prep_tc_raw);
    uint8_t *bop = smem + kPrepTcBufs * kPrepTcTile;
    const uint32_t sbase = smem_u32(smem);
    __shared__ __align__(8) unsigned long long bars[kPrepTcBufs + 1];      // tile landed (per buffer); product done
    __shared__ uint32_t tmem_holder;
    __shared__ int abort_flag;
    const ErrSink sink = prep_sink(p);
    const int t = threadIdx.x, warp = t >> 5;
    const uint32_t bar_tile0 = smem_u32(&bars[0]), bar_mma = smem_u32(&bars[kPrepTcBufs]);

    // thread 0: the tiles of the block's k-th list entry into buffer k % kPrepTcBufs; an entry without candidates
    // completes the buffer's barrier phase without a copy, so phases and entries stay in step
    auto issue_copy = [&](int k) {
        const long long idx = (long long)blockIdx.x + (long long)k * gridDim.x;
        if (idx >= total) return;
        const PrepUnit w = prep_unit_at<kSub>(p, (int)idx, false);
        const int buf = k % kPrepTcBufs;
        const uint32_t bar = bar_tile0 + 8u * buf, dst = sbase + buf * kPrepTcTile;
        if (w.rows_here <= 0) {
            mbar_arrive(bar);
            return;
        }
        const bool both = kSub == 1 || w.rows_here > kTile;
        const int y = (int)tile_row0(p, w.head, w.tile);
        mbar_expect_tx(bar, both ? kPrepTcTile : kPrepTcTile / 2);
        tma_load_2d(dst, &map_k, 0, y, bar);
        if (kSub == 1) tma_load_2d(dst + kPrepTcTile / 2, &map_k, 64, y, bar);
        else if (both) tma_load_2d(dst + kPrepTcTile / 2, &map_k, 0, (int)tile_row0(p, w.head, w.tile + 1), bar);
    };

    if (t == 0) {
        abort_flag = 0;
        for (int q = 0; q < kPrepTcBufs; ++q) mbar_init(bar_tile0 + 8u * q, 1);
        mbar_init(bar_mma, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&tmem_holder)), "r"(kPrepTcTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // rows 3 kSub..15 of the B operand stay zero; the others are rewritten in full for every unit
    for (int x = t; x < kPrepTcB / 16; x += kPrepTcThreads) reinterpret_cast<uint4 *>(bop)[x] = make_uint4(0u, 0u, 0u, 0u);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_holder;
    uint32_t mma_parity = 0;
    pdl_trigger();
    pdl_wait();                             // the set-up above touches no global memory
    if (!p.lengths_done) clear_counters(p);
    if (t == 0)
        for (int q = 0; q < kPrepTcBufs - 1; ++q) issue_copy(q);

    int k = 0, idx = (int)blockIdx.x;
    for (; idx < total; idx += (int)gridDim.x, ++k) {
        const PrepUnit w = prep_unit_at<kSub>(p, idx, t == 0 && !p.lengths_done);
        const int head = w.head, n = w.n, rows_here = w.rows_here;
        const int buf = k % kPrepTcBufs;
        uint8_t *tile_smem = smem + buf * kPrepTcTile;
        // the buffer entry k - 1 used is free (its product was waited for, by every thread, before the last barrier)
        if (t == 0) issue_copy(k + kPrepTcBufs - 1);

        const bool landed = mbar_wait(bar_tile0 + 8u * buf, (uint32_t)(k / kPrepTcBufs) & 1u, &abort_flag, sink);
        const bool ok = __syncthreads_and(landed);           // the block goes on as a whole, or not at all

        // ---- one thread per row: norm, r, the slices; rows that are not candidates are cleared in shared memory
        // (they may hold anything, and 0 x NaN would spoil the product).  Two threads per row were measured slower:
        // the time of a tile is a chain of latencies (barrier, shared-memory loads, product, TMEM load), not of issue slots.
        const int rt = t;
        float r[kSub], sq[kSub];
#pragma unroll
        for (int u = 0; u < kSub; ++u) {
            r[u] = sq[u] = 0.f;
            if (!ok || rows_here <= 0) continue;
            // chunk c of the row: the first box, or with 128 dimensions the second as well
            uint8_t *row_smem = tile_smem + u * (kPrepTcTile / 2) + rt * 128;
            if (u * kTile + rt < rows_here) {
                float2 sq2[4];                       // four independent chains of packed multiply-adds
#pragma unroll
                for (int e = 0; e < 4; ++e) sq2[e] = make_float2(0.f, 0.f);
#pragma unroll
                for (int c = 0; c < kChunks; ++c) {
                    const uint4 vec = *reinterpret_cast<const uint4 *>(row_smem + (c >> 3) * (kPrepTcTile / 2) + (((c & 7) ^ (rt & 7)) << 4));
                    float f[8];
                    Elem<__nv_bfloat16>::unpack(vec, f);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 f2 = make_float2(f[2 * e], f[2 * e + 1]);
                        sq2[e] = __ffma2_rn(f2, f2, sq2[e]);
                    }
                }
                sq[u] = ((sq2[0].x + sq2[0].y) + (sq2[1].x + sq2[1].y)) + ((sq2[2].x + sq2[2].y) + (sq2[3].x + sq2[3].y));
                const float nrm = sq[u] > 0.f ? sq[u] * rsqrtf(sq[u]) : 0.f;
                r[u] = __fdividef(1.0f, nrm + p.eps);
            } else {
#pragma unroll
                for (int c = 0; c < kChunks; ++c)
                    *reinterpret_cast<uint4 *>(row_smem + (c >> 3) * (kPrepTcTile / 2) + ((c & 7) << 4)) = make_uint4(0u, 0u, 0u, 0u);
            }
        }
        if (ok) {
            // r in three bf16 parts: row t of the B operand's K dimension, rows 3 u..3 u + 2 of its N dimension
            const int s = rt >> 4, kk = rt & 15;
#pragma unroll
            for (int u = 0; u < kSub; ++u) {
                float rest = r[u];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const __nv_bfloat16 h16 = __float2bfloat16_rn(rest);
                    const int nn = 3 * u + c;        // (32-byte rows, 32-byte swizzle: rows 4..7 have their 16-byte halves swapped)
                    *reinterpret_cast<__nv_bfloat16 *>(bop + s * 512 + nn * 32 + (((kk >> 3) ^ (nn >> 2)) << 4) + (kk & 7) * 2) = h16;
                    rest -= __bfloat162float(h16);
                }
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");       // generic writes -> tensor-core reads
        __syncthreads();

        // ---- sum_i r_i k_i[c]: D[c][nn] = sum_i K[i][c] R[nn][i], the tile as an MN-major operand
        if (ok && rows_here > 0 && t == 0) {
            // f32 accumulate, bf16 x bf16, A MN-major (bit 15), B K-major, M = 128, N = 16
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | ((16u >> 3) << 17) | ((128u >> 4) << 24);
            tc_fence_after();
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                const uint32_t a_addr = sbase + buf * kPrepTcTile + ks * 2048;    // 16 rows of 128 bytes further
                const uint32_t b_addr = sbase + kPrepTcBufs * kPrepTcTile + ks * 512;
                // A: 64-element (128-byte) atoms along M 16 KB apart (the second TMA box), 8-row groups along K 1 KB apart
                uint64_t da = (uint64_t)((a_addr & 0x3FFFFu) >> 4) | ((uint64_t)(16384u >> 4) << 16) | ((uint64_t)(1024u >> 4) << 32) |
                              ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
                // B: 32-byte rows, 8-row groups 256 B apart, 32-byte swizzle
                uint64_t db = (uint64_t)((b_addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(256u >> 4) << 32) |
                              ((uint64_t)1 << 46) | ((uint64_t)6 << 61);
                asm volatile("{\n\t.reg .pred pp;\n\tsetp.ne.b32 pp, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, pp;\n\t}"
                             ::"r"(tmem), "l"(da), "l"(db), "r"(idesc), "r"(ks) : "memory");
            }
            umma_commit(bar_mma);
        }

        // ---- what a row leaves behind, written while the product runs
        if (ok) {
#pragma unroll
            for (int u = 0; u < kSub; ++u) {
                const int tile = w.tile + u, row = tile * kTile + rt;
                if (kSub > 1 && tile >= p.tiles) break;
                p.inv_norm[(size_t)head * p.cap_pad + row] = r[u];
                p.self_dot[(size_t)head * p.cap_pad + row] = (r[u] * r[u]) * sq[u];     // Kbar_i . Kbar_i
                if (!p.tri) continue;
                // the threshold slices of the scoring kernels (see above): 1 / r as (n1, n2, n3, n1, n2, n1, 0 ...),
                // and for the head's last key tile -T / r as (-t1, -t1, -t1, -t2, -t2, -t3, 0 ...)
                float rest = r[u] > 0.f ? __fdiv_rn(1.0f, r[u]) : 0.f;
                uint32_t part[3];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const __nv_bfloat16 h16 = __float2bfloat16_rn(rest);
                    part[c] = (uint32_t)__bfloat16_as_ushort(h16);
                    rest -= __bfloat162float(h16);
                }
                uint4 *dst = reinterpret_cast<uint4 *>(p.norm_split + ((size_t)head * p.cap_pad + row) * sm100::kSliceElems);
                dst[0] = make_uint4(part[0] | (part[1] << 16), part[2] | (part[0] << 16), part[1] | (part[0] << 16), 0u);
                if (tile == (n + kTile - 1) / kTile - 1) {
                    rest = r[u] > 0.f ? -__fdiv_rn(p.sim_threshold, r[u]) : 0.f;
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        const __nv_bfloat16 h16 = __float2bfloat16_rn(rest);
                        part[c] = (uint32_t)__bfloat16_as_ushort(h16);
                        rest -= __bfloat162float(h16);
                    }
                    uint4 *thr = reinterpret_cast<uint4 *>(p.thr_split + ((size_t)head * kTile + rt) * sm100::kSliceElems);
                    thr[0] = make_uint4(part[0] | (part[0] << 16), part[0] | (part[1] << 16), part[1] | (part[2] << 16), 0u);
                }
            }
        }

        float tsum = 0.f;
        bool done = ok;
        if (ok && rows_here > 0) {
            done = mbar_wait(bar_mma, mma_parity, &abort_flag, sink);
            mma_parity ^= 1u;
            if (done) {
                tc_fence_after();
                uint32_t acc[8];
                tmem_ld8(tmem + ((uint32_t)(warp * 32) << 16), acc);      // lane = column c of the keys (of tile c / D of the unit)
                tmem_wait8(acc);
                tsum = kSub > 1 && t >= D ? (__uint_as_float(acc[3]) + __uint_as_float(acc[4])) + __uint_as_float(acc[5])
                                          : (__uint_as_float(acc[0]) + __uint_as_float(acc[1])) + __uint_as_float(acc[2]);
            }
        }
        tc_fence_before();
        done = __syncthreads_and(done);
        if (kSub == 1 || w.tile + t / D < p.tiles) p.tile_sum[((size_t)head * p.tiles + w.tile) * D + t] = done ? tsum : 0.f;
        if (!done) break;
    }

    if (t == 0 && idx < total) {            // error path: units from this one on are given up
        for (int e = k; e < k + kPrepTcBufs; ++e)
            if ((long long)blockIdx.x + (long long)e * gridDim.x < total) drain(bar_tile0 + 8u * (e % kPrepTcBufs), (uint32_t)(e / kPrepTcBufs) & 1u);
        drain(bar_mma, mma_parity ^ 1u);
        for (; idx < total; idx += (int)gridDim.x) {
            const PrepUnit w = prep_unit_at<kSub>(p, idx, !p.lengths_done);
            for (int u = 0; u < kSub && w.tile + u < p.tiles; ++u) p.inv_norm[(size_t)w.head * p.cap_pad + (w.tile + u) * kTile] = kGaveUp;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kPrepTcTmemCols) : "memory");
    }
}

// ---- the same kernel for caches that are scored on a copy: 8-bit codes of 128 dimensions --------------------------------
//
// The tile arrives as stored (16 KB, a ring of two stages); the thread that owns a row
// widens it into the bf16 operand tile, taking the norm on the way; the tensor cores form the key sums from that
// tile as above, and the same tile is written out, by TMA, as the head's part of the scoring copy, which the later
// stages read.  The stored keys are read once and the copy is not read back here: a separate widening pass in front
// of prep_tc_kernel cost the prep stage a second sweep over keys twice the stored size.  Only for caches whose
// capacity is a whole number of tiles (a tile's store must not reach into the next head's rows).
constexpr int kFusedRaw = kTile * 128;                      // a stored tile: 16 KB
constexpr int kFusedOffRaw = kPrepTcBufs * kPrepTcTile;
constexpr int kFusedOffB = kFusedOffRaw + 2 * kFusedRaw;
constexpr int kFusedSmem = kFusedOffB + kPrepTcB + 1024;
constexpr int kFusedBlocks = 2;

__global__ void __launch_bounds__(kPrepTcThreads, kFusedBlocks)
prep_fused_kernel(Params p, const __grid_constant__ CUtensorMap map_src, const __grid_constant__ CUtensorMap map_wide,
                  const int32_t *src_table, int total)
{
    using namespace sm100;
    constexpr int D = kHeadDim;
    extern __shared__ uint8_t prep_tc_raw[];
    uint8_t *smem = align_smem(prep_tc_raw);
    uint8_t *bop = smem + kFusedOffB;
    const uint32_t sbase = smem_u32(smem);
    __shared__ __align__(8) unsigned long long bars[3];      // stored tile landed (per stage); product done
    __shared__ uint32_t tmem_holder;
    __shared__ int abort_flag;
    const ErrSink sink = prep_sink(p);
    const int t = threadIdx.x, warp = t >> 5;
    const uint32_t bar_raw0 = smem_u32(&bars[0]), bar_mma = smem_u32(&bars[2]);

    // thread 0: the stored tile of the block's k-th list entry into stage k % 2 (an entry without candidates completes
    // the stage's barrier phase without a copy)
    auto issue_copy = [&](int k) {
        const long long idx = (long long)blockIdx.x + (long long)k * gridDim.x;
        if (idx >= total) return;
        const PrepUnit w = prep_unit_at<1>(p, (int)idx, false);
        const uint32_t bar = bar_raw0 + 8u * (k & 1);
        if (w.rows_here <= 0) {
            mbar_arrive(bar);
            return;
        }
        const int y = src_table ? src_table[(size_t)w.head * (p.cap / kTile) + w.tile] * kTile : w.head * p.cap + w.tile * kTile;
        mbar_expect_tx(bar, kFusedRaw);
        tma_load_2d(sbase + kFusedOffRaw + (k & 1) * kFusedRaw, &map_src, 0, y, bar);
    };

    if (t == 0) {
        abort_flag = 0;
        mbar_init(bar_raw0, 1);
        mbar_init(bar_raw0 + 8u, 1);
        mbar_init(bar_mma, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&tmem_holder)), "r"(kPrepTcTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int x = t; x < kPrepTcB / 16; x += kPrepTcThreads) reinterpret_cast<uint4 *>(bop)[x] = make_uint4(0u, 0u, 0u, 0u);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_holder;
    uint32_t mma_parity = 0;
    pdl_trigger();
    pdl_wait();
    clear_counters(p);
    if (t == 0) issue_copy(0);

    int k = 0, idx = (int)blockIdx.x;
    for (; idx < total; idx += (int)gridDim.x, ++k) {
        const PrepUnit w = prep_unit_at<1>(p, idx, t == 0);
        const int head = w.head, tile = w.tile, n = w.n, rows_here = w.rows_here;
        const int buf = k & 1;
        uint8_t *tile_smem = smem + buf * kPrepTcTile;
        if (t == 0) {
            // the other stage was read, by every thread, before the last barrier; and the operand tile about to be
            // written was stored two entries ago: that store has to be through with shared memory
            issue_copy(k + 1);
            asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
        }
        const bool landed = mbar_wait(bar_raw0 + 8u * buf, (uint32_t)(k >> 1) & 1u, &abort_flag, sink);
        const bool ok = __syncthreads_and(landed);           // the block goes on as a whole, or not at all

        // ---- one thread per row: the stored row into the operand tile (bf16, 128 dimensions, the layout a TMA load
        // leaves), its norm on the way; rows that are not candidates become zeros
        const int rt = t;
        const int row = tile * kTile + rt;
        float r = 0.f, sq = 0.f;
        if (ok && rows_here > 0) {
            uint4 out[16];
#pragma unroll
            for (int c = 0; c < 16; ++c) out[c] = make_uint4(0u, 0u, 0u, 0u);
            if (rt < rows_here) {
                const uint8_t *raw = smem + kFusedOffRaw + buf * kFusedRaw + rt * 128;
                uint4 in[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) in[c] = *reinterpret_cast<const uint4 *>(raw + ((c ^ (rt & 7)) << 4));
                float2 sq2[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) sq2[e] = make_float2(0.f, 0.f);
#pragma unroll
                for (int c = 0; c < 8; ++c) widen16(in[c], &out[2 * c], &out[2 * c + 1]);     // 16 codes -> bf16 chunks 2 c, 2 c + 1
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    float f[8];
                    Elem<__nv_bfloat16>::unpack(out[c], f);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 f2 = make_float2(f[2 * e], f[2 * e + 1]);
                        sq2[e] = __ffma2_rn(f2, f2, sq2[e]);
                    }
                }
                sq = ((sq2[0].x + sq2[0].y) + (sq2[1].x + sq2[1].y)) + ((sq2[2].x + sq2[2].y) + (sq2[3].x + sq2[3].y));
                const float nrm = sq > 0.f ? sq * rsqrtf(sq) : 0.f;
                r = __fdividef(1.0f, nrm + p.eps);
            }
#pragma unroll
            for (int c = 0; c < 16; ++c)
                *reinterpret_cast<uint4 *>(tile_smem + (c >> 3) * (kPrepTcTile / 2) + rt * 128 + (((c & 7) ^ (rt & 7)) << 4)) = out[c];
        }
        if (ok) {
            float rest = r;
            uint32_t rp[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const __nv_bfloat16 h16 = __float2bfloat16_rn(rest);
                rp[c] = (uint32_t)__bfloat16_as_ushort(h16);
                rest -= __bfloat162float(h16);
            }
            const int s = rt >> 4, kk = rt & 15;
#pragma unroll
            for (int nn = 0; nn < 3; ++nn)
                *reinterpret_cast<unsigned short *>(bop + s * 512 + nn * 32 + ((kk >> 3) << 4) + (kk & 7) * 2) = (unsigned short)rp[nn];
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");       // generic writes -> tensor-core and TMA reads
        __syncthreads();

        if (ok && rows_here > 0 && t == 0) {
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | ((16u >> 3) << 17) | ((128u >> 4) << 24);
            tc_fence_after();
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                const uint32_t a_addr = sbase + buf * kPrepTcTile + ks * 2048;
                const uint32_t b_addr = sbase + kFusedOffB + ks * 512;
                uint64_t da = (uint64_t)((a_addr & 0x3FFFFu) >> 4) | ((uint64_t)(16384u >> 4) << 16) | ((uint64_t)(1024u >> 4) << 32) |
                              ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
                uint64_t db = (uint64_t)((b_addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(256u >> 4) << 32) |
                              ((uint64_t)1 << 46) | ((uint64_t)6 << 61);
                asm volatile("{\n\t.reg .pred pp;\n\tsetp.ne.b32 pp, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, pp;\n\t}"
                             ::"r"(tmem), "l"(da), "l"(db), "r"(idesc), "r"(ks) : "memory");
            }
            umma_commit(bar_mma);
            // the tile, as the head's rows [128 tile, 128 tile + 128) of the scoring copy (contiguous, head after head)
            const int yw = head * p.cap + tile * kTile;
            asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                         ::"l"(reinterpret_cast<uint64_t>(&map_wide)), "r"(0), "r"(yw), "r"(sbase + buf * kPrepTcTile) : "memory");
            asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                         ::"l"(reinterpret_cast<uint64_t>(&map_wide)), "r"(64), "r"(yw), "r"(sbase + buf * kPrepTcTile + kPrepTcTile / 2) : "memory");
        }
        if (t == 0) asm volatile("cp.async.bulk.commit_group;" ::: "memory");      // one group per entry, empty or not

        if (ok) {
            p.inv_norm[(size_t)head * p.cap_pad + row] = r;
            p.self_dot[(size_t)head * p.cap_pad + row] = (r * r) * sq;     // Kbar_i . Kbar_i
            if (p.tri) {
                float rest = r > 0.f ? __fdiv_rn(1.0f, r) : 0.f;
                uint32_t part[3];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const __nv_bfloat16 h16 = __float2bfloat16_rn(rest);
                    part[c] = (uint32_t)__bfloat16_as_ushort(h16);
                    rest -= __bfloat162float(h16);
                }
                uint4 *dst = reinterpret_cast<uint4 *>(p.norm_split + ((size_t)head * p.cap_pad + row) * sm100::kSliceElems);
                dst[0] = make_uint4(part[0] | (part[1] << 16), part[2] | (part[0] << 16), part[1] | (part[0] << 16), 0u);
                if (tile == (n + kTile - 1) / kTile - 1) {
                    rest = r > 0.f ? -__fdiv_rn(p.sim_threshold, r) : 0.f;
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        const __nv_bfloat16 h16 = __float2bfloat16_rn(rest);
                        part[c] = (uint32_t)__bfloat16_as_ushort(h16);
                        rest -= __bfloat162float(h16);
                    }
                    uint4 *thr = reinterpret_cast<uint4 *>(p.thr_split + ((size_t)head * kTile + rt) * sm100::kSliceElems);
                    thr[0] = make_uint4(part[0] | (part[0] << 16), part[0] | (part[1] << 16), part[1] | (part[2] << 16), 0u);
                }
            }
        }

        float tsum = 0.f;
        bool done = ok;
        if (ok && rows_here > 0) {
            done = mbar_wait(bar_mma, mma_parity, &abort_flag, sink);
            mma_parity ^= 1u;
            if (done) {
                tc_fence_after();
                uint32_t acc[8];
                tmem_ld8(tmem + ((uint32_t)(warp * 32) << 16), acc);      // lane = column c of the keys
                tmem_wait8(acc);
                tsum = (__uint_as_float(acc[0]) + __uint_as_float(acc[1])) + __uint_as_float(acc[2]);
            }
        }
        tc_fence_before();
        done = __syncthreads_and(done);
        p.tile_sum[((size_t)head * p.tiles + tile) * D + t] = done ? tsum : 0.f;
        if (!done) break;
    }

    if (t == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");      // the stores are through before the block leaves
    if (t == 0 && idx < total) {            // error path: tiles from this one on are given up
        for (int e = k; e < k + 2; ++e)
            if ((long long)blockIdx.x + (long long)e * gridDim.x < total) drain(bar_raw0 + 8u * (e & 1), (uint32_t)(e >> 1) & 1u);
        drain(bar_mma, mma_parity ^ 1u);
        for (; idx < total; idx += (int)gridDim.x) {
            const PrepUnit w = prep_unit_at<1>(p, idx, true);
            p.inv_norm[(size_t)w.head * p.cap_pad + w.tile * kTile] = kGaveUp;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kPrepTcTmemCols) : "memory");
    }
}

// The tile sums of a head added up in tile order (a launch of its own behind prep_tc_kernel: no tickets, no fences in
// the streaming kernel), also as three bf16 rows whose sum is s to fp32 accuracy (rows 3..15 of the 16-row block are
// zero): appended to the query rows, they let the tensor cores form Kbar_i . s along with the logits.
template <int D>                             // (D >= 64, the most tiles that a head can have)
__global__ void __launch_bounds__(D) head_sum_kernel(Params p)
{
    pdl_trigger();
    pdl_wait();
    const int head = blockIdx.x, t = threadIdx.x;
    const float first_r = t < p.tiles ? p.inv_norm[(size_t)head * p.cap_pad + t * kTile] : 0.f;
    const float *ts = p.tile_sum + (size_t)head * p.tiles * D + t;
    float s = 0.f;
    for (int q = 0; q < p.tiles; ++q) s += ts[(size_t)q * D];
    __nv_bfloat16 *hs = p.head_sum_bf16 + (size_t)head * 16 * D + t;
    float rest = s;
#pragma unroll
    for (int part_i = 0; part_i < 3; ++part_i) {
        const __nv_bfloat16 h16 = __float2bfloat16_rn(rest);
        hs[part_i * D] = h16;
        rest -= __bfloat162float(h16);
    }
    for (int z = 3; z < 16; ++z) hs[z * D] = __float2bfloat16_rn(0.f);
    if (prep_gave_up(first_r)) report_timeout(make_sink(p));
}

}  // namespace

template <typename T, int D>
static cudaError_t launch_prep_for(const Params &p, int dev, cudaStream_t s)
{
    static PerDevice done;
    const unsigned grid = (unsigned)p.tiles * (unsigned)(p.batch * p.hkv);
    const int smem = kTile * D * (int)sizeof(T) + 16;
    const cudaError_t e = allow_smem_once(done, dev, prep_kernel<T, D>, smem);
    if (e != cudaSuccess) return e;
    return launch_early(prep_kernel<T, D>, grid, kPrepThreads, smem, s, 1, p);
}

template <int D>
static cudaError_t launch_prep_tc_for(const Params &p, int dev, int sms, cudaStream_t s)
{
    static PerDevice done;
    CUtensorMap map_k;
    if (!sm100::make_map_rows(&map_k, p.k_cache, sm100::key_rows_total(p), D, kTile)) return cudaErrorInvalidValue;
    cudaError_t e = allow_smem_once(done, dev, prep_tc_kernel<D>, kPrepTcSmem);
    if (e != cudaSuccess) return e;
    if (p.lengths_done &&
        (e = launch_early(lengths_kernel, (unsigned)((p.batch + kLengthThreads - 1) / kLengthThreads), kLengthThreads, 0, s, 1, p)) != cudaSuccess)
        return e;
    const int total = (p.tiles + kHeadDim / D - 1) / (kHeadDim / D) * p.batch * p.hkv;
    if ((e = launch_early(prep_tc_kernel<D>, (unsigned)std::min(total, kPrepTcBlocks * sms), kPrepTcThreads, kPrepTcSmem, s, 1, p, map_k, total)) !=
        cudaSuccess)
        return e;
    return launch_early(head_sum_kernel<D>, (unsigned)(p.batch * p.hkv), D, 0, s, 1, p);
}

cudaError_t launch_prep(const Params &p, cudaStream_t s)
{
    const bool bf16 = p.dtype == RKV_BF16;
    int dev = 0, sms = 0;
    cudaError_t e = device_sms(&dev, &sms);
    if (e != cudaSuccess) return e;
    if (p.fused_codes) {                    // the tensor-core form that also writes the scoring copy
        static PerDevice done;
        const int total = p.tiles * p.batch * p.hkv;
        const uint64_t wide_rows = (uint64_t)p.batch * p.hkv * p.cap + kTile;
        const uint64_t src_rows = p.fuse_table ? (uint64_t)p.pool_pages * kTile : (uint64_t)p.batch * p.hkv * p.cap;
        CUtensorMap map_src, map_wide;
        if (!sm100::make_map_row128(&map_src, p.fuse_src, src_rows, true) || !sm100::make_map(&map_wide, p.k_cache, wide_rows, kTile))
            return cudaErrorInvalidValue;
        if ((e = allow_smem_once(done, dev, prep_fused_kernel, kFusedSmem)) != cudaSuccess) return e;
        e = launch_early(prep_fused_kernel, (unsigned)std::min(total, kFusedBlocks * sms), kPrepTcThreads, kFusedSmem, s, 1, p, map_src, map_wide,
                         p.fuse_table, total);
        if (e != cudaSuccess) return e;
        return launch_early(head_sum_kernel<kHeadDim>, (unsigned)(p.batch * p.hkv), kHeadDim, 0, s, 1, p);
    }
    if (bf16 && p.d == 128) return launch_prep_tc_for<128>(p, dev, sms, s);          // the tensor-core form
    if (bf16 && p.d == 64 && p.tri) return launch_prep_tc_for<64>(p, dev, sms, s);
    switch (p.d) {
        case 64: return bf16 ? launch_prep_for<__nv_bfloat16, 64>(p, dev, s) : launch_prep_for<float, 64>(p, dev, s);
        case 128: return launch_prep_for<float, 128>(p, dev, s);
        case 256: return bf16 ? launch_prep_for<__nv_bfloat16, 256>(p, dev, s) : launch_prep_for<float, 256>(p, dev, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace rkv
