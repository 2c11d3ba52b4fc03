// Stage "prep" on the CUDA cores (fp32 caches, 256 dimensions): one streaming pass over the candidate keys.
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

#include "rkv_prep.cuh"

namespace rkv {

namespace {

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

// The tile sums of a head added up in tile order (a launch of its own behind the streaming kernel: no tickets, no fences in
// the streaming kernel), also as three bf16 rows whose sum is s to fp32 accuracy (rows 3..15 of the 16-row block are
// zero): behind the rows of the last key tile they let the first scoring pass form Kbar_i . s in its own product.
// kCodes: as E4M3 codes, for keys that are.  A part holds what the parts before it left, 16 times as large: four more bits of the
// sum each, so that seven hold all that fp32 does of components down to 2^-17 of the largest; of smaller ones they leave 2^-42 of the largest.
template <int D, bool kCodes = false>        // (D >= 64, the most tiles that a head can have)
__global__ void __launch_bounds__(D) head_sum_kernel(Params p)
{
    pdl_trigger();
    pdl_wait();
    const int head = blockIdx.x, t = threadIdx.x;
    const float first_r = t < p.tiles ? p.inv_norm[(size_t)head * p.cap_pad + t * kTile] : 0.f;
    const float *ts = p.tile_sum + (size_t)head * p.tiles * D + t;
    float s = 0.f;
    for (int q = 0; q < p.tiles; ++q) s += ts[(size_t)q * D];
    if constexpr (kCodes) {
        __shared__ float top[D / 32];
        float m = fabsf(s);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
        if ((t & 31) == 0) top[t / 32] = m;
        __syncthreads();
        for (int w = 0; w < D / 32; ++w) m = fmaxf(m, top[w]);
        int e = 0;
        if (m > 0.f && m < 1e30f) frexpf(m, &e);                       // m < 2^e
        e = max(-100, min(100, 8 - e));                                // the largest component into [128, 256)
        uint8_t *rows = reinterpret_cast<uint8_t *>(p.head_sum_bf16) + (size_t)head * kSumHeadBytes;
        float rest = ldexpf(s, e);
        for (int part = 0; part < 16; ++part) {
            const __nv_fp8_storage_t code = part < kSumParts ? __nv_cvt_float_to_fp8(rest, __NV_SATFINITE, __NV_E4M3) : 0;
            const __half_raw h = __nv_cvt_fp8_to_halfraw(code, __NV_E4M3);
            rows[part * D + t] = code;
            rest = (rest - __half2float(*reinterpret_cast<const __half *>(&h))) * 16.f;
        }
        if (t == 0) *reinterpret_cast<float *>(rows + kSumScaleAt) = ldexpf(1.f, -e);
        if (prep_gave_up(first_r)) report_timeout(make_sink(p));
        return;
    }
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

cudaError_t launch_head_sum(const Params &p, cudaStream_t s)
{
    const unsigned heads = (unsigned)(p.batch * p.hkv);
    return p.codes     ? launch_early(head_sum_kernel<128, true>, heads, 128, 0, s, 1, p)
           : p.d == 64 ? launch_early(head_sum_kernel<64>, heads, 64, 0, s, 1, p)
                       : launch_early(head_sum_kernel<128>, heads, 128, 0, s, 1, p);
}

template <typename T, int D>
static cudaError_t launch_prep_for(const Params &p, int dev, cudaStream_t s)
{
    static PerDevice done;
    const unsigned grid = (unsigned)p.tiles * (unsigned)(p.batch * p.hkv);
    const int smem = kTile * D * (int)sizeof(T) + 16;
    const cudaError_t e = allow_smem_once(done, dev, prep_kernel<T, D>, smem);
    if (e != cudaSuccess) return e;
    return launch_early(prep_kernel<T, D>, grid, kPrepThreads, smem, s, 1, p);      // (the kernels that follow add the tile sums up)
}

cudaError_t launch_prep(const Params &p, cudaStream_t s)
{
    const bool bf16 = p.dtype == RKV_BF16;
    int dev = 0, sms = 0;
    const cudaError_t e = device_sms(&dev, &sms);
    if (e != cudaSuccess) return e;
    if (p.fused_codes || p.codes || (bf16 && (p.d == 128 || (p.d == 64 && p.tri)))) return launch_prep_sm100(p, s);          // the tensor-core form
    switch (p.d) {
        case 64: return bf16 ? launch_prep_for<__nv_bfloat16, 64>(p, dev, s) : launch_prep_for<float, 64>(p, dev, s);
        case 128: return launch_prep_for<float, 128>(p, dev, s);
        case 256: return bf16 ? launch_prep_for<__nv_bfloat16, 256>(p, dev, s) : launch_prep_for<float, 256>(p, dev, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace rkv
