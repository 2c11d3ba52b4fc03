// Stage "scores", CUDA-core version: plain fp32 arithmetic.
//
// Used for fp32 caches and, behind RKV_FLAG_SIMT_SCORES, as an independent on-GPU cross-check of the tensor-core kernels
// for bf16 caches.  It forms Eq. 5's matrix in registers and accumulates Eq. 6's sums directly (no closed form), so the
// kernels reach the same numbers along different routes.
//
// Block x of a head, x < row blocks: 64 (small problems: 16) rows of the similarity matrix: for each row i the column sum over j
// of S[j][i] (S is symmetric before the retention rule, which for token i touches line i only), minus the entries of the
// up-to-beta largest j with S[j][i] > T.
// The blocks after those: Eq. 2-3 pooled logits of the head's query group against 64 (d = 256: 32) candidate keys each.
//
// Bound by fp32 multiply-adds: a thread holds an 8 x 4 piece of a 64 x 64 product, so a 16-byte shared-memory load feeds ten
// multiply-adds (one thread per row with the whole head dimension, the earlier form, issued two loads per multiply-add:
// 256 heads of 1144 tokens took 30 ms, a single head of 88 tokens 70 us).  Rows are D + 4 floats apart: the 16 column rows
// that a half-warp reads lie in distinct banks, its own rows are broadcasts.  Packed multiply-adds over pairs of
// dimensions.  Where blocks of 64 rows would leave SMs without one, blocks of 16 rows (a 2 x 4 piece per thread): the time is
// then one block's, and a quarter of the rows is a quarter of its multiply-adds (a single head of 88 tokens: 19 us with 64
// rows per block, 9 with 16).
#include "rkv_common.cuh"

namespace rkv {

namespace {

constexpr int kSimtThreads = 128;
// kRowsT: rows that a thread holds of a block's 8 kRowsT: rg, rg + 8, ... (rg = thread / 16)
template <int D, int kRowsT> struct SimtShape {
    static constexpr int kRowsA = 8 * kRowsT;
    static constexpr int kPad = D + 4;
    static constexpr int kCols = D <= 128 ? 64 : 32;       // streamed keys per step
    static constexpr int kColsT = kCols / 16;              // ... of which a thread holds: cg, cg + 16, ... (cg = thread % 16)
    static constexpr int kChunks = (RKV_MAX_GROUP_ROWS + kRowsA - 1) / kRowsA;       // of the query rows
    static constexpr int kTiles = (kRowsA + kCols) * kPad * 4;
    static constexpr int kStage = RKV_MAX_GROUP_ROWS * (kCols + 1) * 4;              // the logits of a key block, in the tiles' room
    static constexpr int kBytes = kTiles > kStage ? kTiles : kStage;
};

// kRows rows of D elements, starting at `src` (row first_row of its head), into shared memory as fp32; rows >= valid_rows
// are zeros.
template <typename T, int D, int kRows>
__device__ __forceinline__ void load_rows(const T *src, int first_row, int valid_rows, float *dst)
{
    constexpr int kPerVec = Elem<T>::kPerVec;
    constexpr int kVecPerRow = D / kPerVec;
#pragma unroll 8
    for (int v = threadIdx.x; v < kRows * kVecPerRow; v += kSimtThreads) {
        const int r = v / kVecPerRow, c = (v % kVecPerRow) * kPerVec;
        uint4 raw = make_uint4(0u, 0u, 0u, 0u);
        if (first_row + r < valid_rows) raw = *reinterpret_cast<const uint4 *>(src + (size_t)r * D + c);
        float f[kPerVec];
        Elem<T>::unpack(raw, f);
#pragma unroll
        for (int e = 0; e < kPerVec; e += 4)
            *reinterpret_cast<float4 *>(dst + r * (D + 4) + c + e) = make_float4(f[e], f[e + 1], f[e + 2], f[e + 3]);
    }
}

// dot[i][c] = row (rg + 8 i) of A . row (cg + 16 c) of B
template <int D, int kRowsT>
__device__ __forceinline__ void tile_product(const float *A, const float *B, float (&dot)[kRowsT][SimtShape<D, kRowsT>::kColsT])
{
    constexpr int kPad = SimtShape<D, kRowsT>::kPad, kC = SimtShape<D, kRowsT>::kColsT;
    const float *a = A + (threadIdx.x >> 4) * kPad, *b = B + (threadIdx.x & 15) * kPad;
    float2 acc[kRowsT][kC];
#pragma unroll
    for (int i = 0; i < kRowsT; ++i)
#pragma unroll
        for (int c = 0; c < kC; ++c) acc[i][c] = make_float2(0.f, 0.f);
#pragma unroll 2
    for (int k = 0; k < D; k += 4) {
        float4 vb[kC];
#pragma unroll
        for (int c = 0; c < kC; ++c) vb[c] = *reinterpret_cast<const float4 *>(b + c * 16 * kPad + k);
#pragma unroll
        for (int i = 0; i < kRowsT; ++i) {
            const float4 va = *reinterpret_cast<const float4 *>(a + i * 8 * kPad + k);
#pragma unroll
            for (int c = 0; c < kC; ++c) {
                acc[i][c] = __ffma2_rn(make_float2(va.x, va.y), make_float2(vb[c].x, vb[c].y), acc[i][c]);
                acc[i][c] = __ffma2_rn(make_float2(va.z, va.w), make_float2(vb[c].z, vb[c].w), acc[i][c]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < kRowsT; ++i)
#pragma unroll
        for (int c = 0; c < kC; ++c) dot[i][c] = acc[i][c].x + acc[i][c].y;
}

template <typename T, int D, int kRowsT>
__global__ void __launch_bounds__(kSimtThreads, D <= 128 ? 3 : 2) scores_simt_kernel(Params p, int row_blocks, int key_blocks)
{
    using S = SimtShape<D, kRowsT>;
    constexpr int kC = S::kColsT, kCols = S::kCols, kRowsA = S::kRowsA;
    extern __shared__ __align__(16) float smem[];
    float *tileA = smem, *tileB = smem + kRowsA * S::kPad;
    __shared__ float rB[kCols];
    pdl_trigger();
    pdl_wait();

    const int blocks_per_head = row_blocks + key_blocks;
    const int head = blockIdx.x / blocks_per_head;
    const int x = blockIdx.x % blocks_per_head;
    const int b = head / p.hkv, h = head % p.hkv;
    const int n = seq_candidates(p, b);
    // first of the rows of the head starting at `first_row` (at most 64 of them: a piece of a page)
    auto key_rows = [&](int first_row) {
        return static_cast<const T *>(p.k_cache) + (size_t)row_index(p, head, first_row) * D;
    };
    const float *inv_norm = p.inv_norm + (size_t)head * p.cap_pad;
    const int t = threadIdx.x, rg = t >> 4, cg = t & 15;

    if (x < row_blocks) {
        // ---------------- Eq. 5-6 + retention rule for rows [kRowsA x, kRowsA x + kRowsA)
        const int i0 = x * kRowsA;
        if (i0 >= n) return;
        load_rows<T, D, kRowsA>(key_rows(i0), i0, n, tileA);
        float ri[kRowsT], total[kRowsT], removed[kRowsT];
        int left[kRowsT];
#pragma unroll
        for (int i = 0; i < kRowsT; ++i) {
            const int row = i0 + rg + 8 * i;
            ri[i] = row < n ? inv_norm[row] : 0.f;
            total[i] = removed[i] = 0.f;
            left[i] = row < n ? p.beta : 0;              // the same in the 16 threads of a row
        }
        for (int j0 = (n - 1) / kCols * kCols; j0 >= 0; j0 -= kCols) {          // descending j: "largest positions first"
            __syncthreads();
            load_rows<T, D, kCols>(key_rows(j0), j0, n, tileB);
            if (t < kCols) {
                const float r = j0 + t < n ? inv_norm[j0 + t] : 0.f;
                if (prep_gave_up(r)) report_timeout(make_sink(p));
                rB[t] = r;
            }
            __syncthreads();
            float s[kRowsT][kC];
            tile_product<D, kRowsT>(tileA, tileB, s);
            float rj[kC];
#pragma unroll
            for (int c = 0; c < kC; ++c) rj[c] = rB[cg + 16 * c];
#pragma unroll
            for (int i = 0; i < kRowsT; ++i) {
                const int own = i0 + rg + 8 * i - j0 - cg;                      // zero diagonal (Eq. 5)
                unsigned long long hits = 0ull;
#pragma unroll
                for (int c = 0; c < kC; ++c) {
                    s[i][c] = own == 16 * c ? 0.f : (s[i][c] * rj[c]) * ri[i];
                    total[i] += s[i][c];
                    const unsigned bal = __ballot_sync(0xffffffffu, s[i][c] > p.sim_threshold);
                    hits |= (unsigned long long)((bal >> (t & 16)) & 0xffffu) << (16 * c);
                }
                if (left[i] > 0 && hits != 0ull) {
                    int taken = __popcll(hits);
                    for (; taken > left[i]; --taken) hits &= hits - 1ull;       // drop the lowest positions
                    left[i] -= taken;
#pragma unroll
                    for (int c = 0; c < kC; ++c) removed[i] += (hits >> (16 * c + cg) & 1ull) ? s[i][c] : 0.f;
                }
            }
        }
#pragma unroll
        for (int i = 0; i < kRowsT; ++i) {
            float v = total[i] - removed[i];
#pragma unroll
            for (int off = 8; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);      // fixed order
            const int row = i0 + rg + 8 * i;
            if (cg == 0 && row < n) p.sbar[(size_t)head * p.cap_pad + row] = v / (float)n;
        }
    } else {
        // ---------------- Eq. 2-3: max over the group of scaled logits, per (query row, key)
        const int j0 = (x - row_blocks) * kCols;
        if (j0 >= n) return;
        const int rows = p.group * p.alpha;
        const T *Q = static_cast<const T *>(p.q_window) + ((size_t)b * p.hq + (size_t)h * p.group) * p.alpha * D;
        load_rows<T, D, kCols>(key_rows(j0), j0, n, tileB);
        float lg[S::kChunks][kRowsT][kC];                // query rows g * alpha + j, at most 112
#pragma unroll
        for (int chunk = 0; chunk < S::kChunks; ++chunk) {
            if (chunk * kRowsA >= rows) break;
            __syncthreads();
            load_rows<T, D, kRowsA>(Q + (size_t)chunk * kRowsA * D, chunk * kRowsA, rows, tileA);
            __syncthreads();
            tile_product<D, kRowsT>(tileA, tileB, lg[chunk]);
        }
        __syncthreads();                                 // the tiles are no longer read
#pragma unroll
        for (int chunk = 0; chunk < S::kChunks; ++chunk)
#pragma unroll
            for (int i = 0; i < kRowsT; ++i) {
                const int row = chunk * kRowsA + rg + 8 * i;
                if (row < rows)
#pragma unroll
                    for (int c = 0; c < kC; ++c) smem[row * (kCols + 1) + cg + 16 * c] = lg[chunk][i][c];
            }
        __syncthreads();
        const float scale = p.logit_scale;
        float *logits = p.logits + (size_t)head * p.alpha * p.cap_pad;
        for (int u = t; u < p.alpha * kCols; u += kSimtThreads) {
            const int j = u / kCols, key = u % kCols;
            if (j0 + key >= n) continue;
            float best = -INFINITY, sum = 0.f;
            for (int g = 0; g < p.group; ++g) {
                const float v = smem[(g * p.alpha + j) * (kCols + 1) + key] * scale;
                best = fmaxf(best, v);
                sum += v;
            }
            logits[(size_t)j * p.cap_pad + j0 + key] = p.gqa_mean_pool ? sum / (float)p.group : best;
        }
    }
}

template <typename T, int D, int kRowsT>
cudaError_t launch_simt_rows(const Params &p, int dev, cudaStream_t s)
{
    using S = SimtShape<D, kRowsT>;
    static PerDevice done;
    const int row_blocks = (p.cap + S::kRowsA - 1) / S::kRowsA, key_blocks = (p.cap + S::kCols - 1) / S::kCols;
    const unsigned grid = (unsigned)(row_blocks + key_blocks) * (unsigned)(p.batch * p.hkv);
    const cudaError_t e = allow_smem_once(done, dev, scores_simt_kernel<T, D, kRowsT>, S::kBytes);
    if (e != cudaSuccess) return e;
    return launch_early(scores_simt_kernel<T, D, kRowsT>, grid, kSimtThreads, S::kBytes, s, 1, p, row_blocks, key_blocks);
}

template <typename T, int D>
cudaError_t launch_simt_for(const Params &p, cudaStream_t s)
{
    int dev = 0, sms = 0;
    const cudaError_t e = device_sms(&dev, &sms);
    if (e != cudaSuccess) return e;
    const long long blocks = (long long)((p.cap + 63) / 64) * p.batch * p.hkv;       // of 64 rows
    return blocks < sms ? launch_simt_rows<T, D, 2>(p, dev, s) : launch_simt_rows<T, D, 8>(p, dev, s);
}

}  // namespace

cudaError_t launch_scores_simt(const Params &p, cudaStream_t s)
{
    const bool bf16 = p.dtype == RKV_BF16;
    switch (p.d) {
        case 64: return bf16 ? launch_simt_for<__nv_bfloat16, 64>(p, s) : launch_simt_for<float, 64>(p, s);
        case 128: return bf16 ? launch_simt_for<__nv_bfloat16, 128>(p, s) : launch_simt_for<float, 128>(p, s);
        case 256: return bf16 ? launch_simt_for<__nv_bfloat16, 256>(p, s) : launch_simt_for<float, 256>(p, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace rkv
