// Internal declarations shared by the kernels of the R-KV compression library (sm_100a).
// Nothing here is part of the public ABI (see include/rkv.h).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "rkv.h"

namespace rkv {

constexpr int kHeadDim = 128;   // columns of a full operand block of the tensor-core kernels (64 dimensions: half a block, 256: two)
constexpr int kTile = 128;      // keys per tile (rows of one tensor-core operand tile)

// meta[b] values
constexpr int kMetaInvalid = -1;

// Everything a kernel needs; passed by value.
struct Params {
    // caller tensors
    void *k_cache;
    void *v_cache;
    const void *q_window;
    int32_t *seq_lens;
    int32_t *out_idx;
    // shapes
    int batch, hkv, hq, group;      // group = G
    int d;                          // head dimension: 64, 128 or 256
    int cap, cap_pad, tiles;        // cap_pad = tiles * kTile
    int budget, buffer, alpha;
    int dtype;                      // of the keys the scoring stages read (bf16 where a widened copy of 8-bit caches is scored)
    int store_row_bytes;            // bytes of a row of the caches as stored (what the gather moves)
    float logit_scale;              // Eq. 2's 1 / sqrt(d) with the caches' own head dimension (d above may be a padded one)
    int lengths_done;               // 1: the lengths are recorded and the counters cleared when the prep kernel starts
    int form_logits;                // 1: the prep kernel forms Eq. 2-3's logits
    int codes;                      // 1: the keys are scored as they are stored, E4M3 codes of 128 dimensions
    int fused_codes;                // 1: prep writes the scoring copy itself (k_cache above) from stored rows of 128 E4M3 codes
    const void *fuse_src;           // the stored keys
    const int32_t *fuse_table;      // their block table (paged caches), else null
    // hyper-parameters
    int pool_w, beta;
    int head_mean;                  // Algorithm 1's aggregated selection: one kept set per sequence from the
                                    // head-averaged Z (Z is then left in `keys` and a second kernel selects)
    int gqa_mean_pool;              // Eq. 3 with the mean over the group's query heads instead of the max
    int mean_then_pool;             // importance in Algorithm 1's order (mean over query rows, then pooling)
    float sim_threshold, eps, lambda;
    // workspace carve-up
    float *inv_norm;     // [P][cap_pad]         r_i = 1 / (||k_i|| + eps); 0 for i >= n; kGaveUp first in a tile: not finished
    __nv_bfloat16 *norm_split;    // [P][cap_pad][8]   (n1, n2, n3, n1, n2, n1, 0, 0): 1 / r_i as three bf16 parts, laid
                                  // out (zeros up to 16 are added on the way) as the extra K = 16 slice the scoring passes append to a key row
    __nv_bfloat16 *thr_split;     // [P][128][8]       (-t1, -t1, -t1, -t2, -t2, -t3, 0, 0): -T / r_j of the keys of the
                                  // head's LAST key tile as three bf16 parts, the slice the first scoring pass appends
                                  // to that tile's rows; the dot product of the two kinds of slice is -T / (r_i r_j)
                                  // to fp32 accuracy.  Both are written by the prep stage (two-pass route only).
    float *tile_sum;     // [P][tiles][128]      sum over the tile's candidate rows of r_i * k_i
    float *logits;       // [P][alpha][cap_pad]  Eq. 2-3: group-max of scaled logits
    float *row_stat;     // [P][alpha + 1][2]    per row of logits (Eq. 3), and of the column means (Eq. 6): maximum, 1 / sum of exp(value - max)
    uint32_t *keys;      // [P][cap_pad]         Eq. 7: Z as an order-preserving integer (head_mean: Z itself)
    float *sbar;         // [P][cap_pad]         Eq. 6 column means after the retention rule.  With `tri` set the scoring
                         //                      kernels leave column SUMS minus the removed entries (the select stage
                         //                      divides by n)
    uint32_t *lacking;   // [P][cap_pad / 32]    tri: a bit per token that is still short of partners
    int32_t *left;       // [P][cap_pad]         tri, beta > 1: how many partners it still lacks
    int32_t *strag;      // [P][cap_pad]         tri: positions of the head's tokens short of partners, ascending
    int4 *strag_items;   // [P * cap_pad / 256]  tri: work list of the second scoring pass: {head, first listed
                         //                      token, tokens (1..256), first streamed tile}
    uint32_t *best;      // [P][cap_pad]         symmetric route: largest partner position + 1 found so far (0 = none)
    int32_t *dense;      // [P]                  1: the head is scored by the symmetric route of the second pass
    int4 *dense_items;   // [P * ceil(tiles/2)]  its work list: {head, pair of row tiles, n, -}
    int dense_ok;        // the symmetric route may be chosen (beta = 1, not switched off)
    float *self_dot;     // [P][cap_pad]         Kbar_i . Kbar_i (1 up to rounding and eps; 0 for a zero key)
    __nv_bfloat16 *head_sum_bf16;   // [P][16][128] the tile sums of a head added up, as three bf16 rows (hi, mid, lo), 13 zero rows
    int32_t *meta;       // [2][batch]           snapshot of seq_lens (kMetaInvalid if out of range), then each
                         //                      sequence's budget (p.budget unless the caller gave per-sequence ones)
    const int32_t *budgets;   // optional [batch]: per-sequence budgets (alpha < budgets[b] <= budget), else null
    const int32_t *block_table;   // optional [P][cap / 128]: paged caches, page (= key tile) ids into the pools, else null
    int pages_per_head;           // cap / 128 (paged caches)
    long long pool_pages;         // pages in the pools (paged caches)
    // zeroed by the prep kernel:
    unsigned long long *counters;   // [32]      [0] = similarity tiles computed by the tcgen05 kernels, [1] = item
                                    //           ticket of the first scoring pass, [2] = entries in strag_items,
                                    //           [3] = item ticket of the second pass, [4] = the call's abort word
                                    //           (non-zero once a bounded wait ran out: later kernels of the call
                                    //           then leave the caches, lengths and index lists alone),
                                    //           [5] = listed-token x key-tile pairs the second pass has to form,
                                    //           [8 + 2 r], [9 + 2 r] = work items and item ticket of its round r,
                                    //           [16], [17] = the same for the symmetric route
    int tri;                        // 1: the triangle kernels score (bf16 default); 0: another kernel does
    // optional outputs
    void *const *kernel_events;     // see rkv_desc_t
    unsigned long long *dbg_counters;
    int32_t *status;
    long long wait_cycles;          // limit of every bounded wait, in clock64() ticks
    float *dbg_I, *dbg_Sbar, *dbg_R, *dbg_Z;
};

__host__ __device__ inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Record optional event i of p.kernel_events on the stream.
inline cudaError_t mark_kernel(const Params &p, int i, cudaStream_t s)
{
    return (p.kernel_events && p.kernel_events[i]) ? cudaEventRecord(static_cast<cudaEvent_t>(p.kernel_events[i]), s)
                                                   : cudaSuccess;
}

__device__ __forceinline__ void report(int32_t *status, int code)
{
    if (status) atomicCAS(status, 0, code);
}

constexpr int kCounterWords = 32;
constexpr int kAbortWord = 4;       // index of the call's abort word in Params::counters
constexpr int kPairsWord = 5;       // index of the second pass's useful-work count
constexpr int kDenseWords = 16;     // counters[16], [17]: work items and item ticket of the symmetric route

// Where a bounded wait records that it ran out: the caller's optional status word, and the call's own abort word
// in the workspace, which the later kernels of the same call read.
struct ErrSink {
    int32_t *status;
    unsigned long long *abort_word;
    long long wait_cycles;
};
__device__ __forceinline__ ErrSink make_sink(const Params &p)
{
    return ErrSink{p.status, p.counters + kAbortWord, p.wait_cycles};
}
__device__ __forceinline__ void report_timeout(const ErrSink &sink)
{
    report(sink.status, RKV_ERR_TIMEOUT);
    if (sink.abort_word) atomicExch(sink.abort_word, 1ull);
}
// True once some kernel of this call has given up on a wait.
__device__ __forceinline__ bool call_aborted(const Params &p)
{
    return *reinterpret_cast<volatile unsigned long long *>(p.counters + kAbortWord) != 0ull;
}

// What a prep block that gave up on a wait leaves as the first r of the tiles it has not finished (an r is never negative).
constexpr float kGaveUp = -1.f;
__device__ __forceinline__ bool prep_gave_up(float r) { return r < 0.f; }

// Number of candidates of a sequence of length L with the given budget: 0 = nothing to compress.
__device__ __forceinline__ int candidates_from_meta(int L, int budget, int alpha)
{
    return (L > budget) ? (L - alpha) : 0;
}
// Where key tile `tile` (128 rows) of head-problem `head` starts, in rows of the 2-D [rows][d] view of k_cache / v_cache:
// head after head for contiguous caches, through the block table for paged ones (a page holds one key tile).
__device__ __forceinline__ long long tile_row0(const Params &p, int head, int tile)
{
    return p.block_table ? (long long)p.block_table[(size_t)head * p.pages_per_head + tile] * kTile
                         : (long long)head * p.cap + (long long)tile * kTile;
}
// ... and row r of the head.
__device__ __forceinline__ long long row_index(const Params &p, int head, int r)
{
    return tile_row0(p, head, r / kTile) + (r % kTile);
}
// The same for sequence b as every stage after prep sees it (length and budget snapshots left by the prep stage).
__device__ __forceinline__ int seq_budget(const Params &p, int b) { return p.meta[p.batch + b]; }
__device__ __forceinline__ int seq_candidates(const Params &p, int b)
{
    return candidates_from_meta(p.meta[b], p.meta[p.batch + b], p.alpha);
}

template <typename T> struct Elem;
template <> struct Elem<__nv_bfloat16> {
    static constexpr int kPerVec = 8;   // elements per 16-byte vector
    __device__ static void unpack(const uint4 &v, float *f)
    {
        const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&v);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float2 t = __bfloat1622float2(h[i]);
            f[2 * i] = t.x;
            f[2 * i + 1] = t.y;
        }
    }
};
template <> struct Elem<float> {
    static constexpr int kPerVec = 4;
    __device__ static void unpack(const uint4 &v, float *f)
    {
        f[0] = __uint_as_float(v.x);
        f[1] = __uint_as_float(v.y);
        f[2] = __uint_as_float(v.z);
        f[3] = __uint_as_float(v.w);
    }
};

// 16 E4M3 codes -> 16 bf16 values (the conversion instruction goes through f16, which holds every E4M3 value too).
// (Measured against integer / packed-bf16 decodes of the codes -- shift the low seven bits into a bf16 pattern and
// multiply by 2^120 --: those were exact too, but slower in the kernel that widens tiles on their way to the tensor
// cores.)
__device__ __forceinline__ void widen16(const uint4 &codes, uint4 *lo, uint4 *hi)
{
    const uint32_t w[4] = {codes.x, codes.y, codes.z, codes.w};
    uint32_t out[8];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const __half2_raw pair = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)((w[q] >> (16 * h)) & 0xFFFFu), __NV_E4M3);
            const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&pair));
            const __nv_bfloat162 b2 = __floats2bfloat162_rn(f.x, f.y);
            out[2 * q + h] = *reinterpret_cast<const uint32_t *>(&b2);
        }
    }
    *lo = make_uint4(out[0], out[1], out[2], out[3]);
    *hi = make_uint4(out[4], out[5], out[6], out[7]);
}

// ---- launches that overlap the end of the kernel before them (programmatic dependent launch) ----------------------------
// A kernel launched through launch_early() may become resident while its predecessor in the stream is still running: it
// lets its own successor in (pdl_trigger) and waits for the predecessor's results (pdl_wait) before it touches global
// memory.  Between the short kernels of a decode step the launch gap, 2-3 us, is most of the time.
// Such a kernel is on the GPU while its inputs are still being written, so it reads them with ordinary loads: the read-only
// path (__ldg) asks for data that nothing writes from the kernel's first block to its last.  The second pass, the symmetric
// scan and its finish may use it for keys and norms: they are launched after a listing kernel, which is launched when the
// first pass is through, and the first pass waited for all that was written before it.
// The persistent scoring kernels (both passes, the symmetric scan) let nothing in before they end.  Blocks that wait beside them take from
// them (the symmetric scan of 2048 heads of 4216 tokens, T = 0.9: 5105 us beside waiting blocks, 4764 without), and where there are few
// heads a pass runs on for long when the first blocks are out of items: a call with 32 heads of 4216 tokens 166 us when the passes let
// the next kernel in at that point, 147 so; 16 of 1700 98, 89; 32 of 4216 in 8 bits 162, 136; 256 of 1144 128.3, 126.7.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... Args>
cudaError_t launch_early(void (*kernel)(Args...), unsigned grid, unsigned block, size_t smem, cudaStream_t s, unsigned cluster, Args... args)
{
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// What a launch asks the runtime for, asked once per device (both idempotent, so threads may race).
constexpr int kDeviceSlots = 64;
inline cudaError_t device_sms(int *dev, int *sms)
{
    static std::atomic<int> known[kDeviceSlots];
    cudaError_t e = cudaGetDevice(dev);
    if (e != cudaSuccess) return e;
    const bool slot = *dev >= 0 && *dev < kDeviceSlots;
    *sms = slot ? known[*dev].load(std::memory_order_relaxed) : 0;
    if (*sms > 0) return cudaSuccess;
    e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, *dev);
    if (e == cudaSuccess && slot) known[*dev].store(*sms, std::memory_order_relaxed);
    return e;
}
// The id of the calling thread's current context, 0 where the driver cannot tell.  Ids are never used again, unlike handles: what
// belongs to a context (function attributes, streams) is kept under its id.
inline unsigned long long context_id()
{
    typedef CUresult (*GetId)(CUcontext, unsigned long long *);
    static const GetId get = []() -> GetId {
        void *sym = nullptr;
        cudaDriverEntryPointQueryResult found;
        const bool ok = cudaGetDriverEntryPoint("cuCtxGetId", &sym, cudaEnableDefault, &found) == cudaSuccess && found == cudaDriverEntryPointSuccess;
        return ok ? reinterpret_cast<GetId>(sym) : nullptr;
    }();
    unsigned long long id = 0ull;
    return get && get(nullptr, &id) == CUDA_SUCCESS ? id : 0ull;
}
// The kernel's dynamic shared memory limit (and clusters of more than 8 blocks), set once per context.  `done`: the context that the
// caller's kernel was last prepared for, per device.
struct PerDevice {
    std::atomic<unsigned long long> context[kDeviceSlots] = {};
};
template <class Kernel>
inline cudaError_t allow_smem_once(PerDevice &done, int dev, Kernel kernel, int bytes, bool wide_cluster = false)
{
    const bool slot = dev >= 0 && dev < kDeviceSlots;
    const unsigned long long context = slot ? context_id() : 0ull;
    if (context && done.context[dev].load(std::memory_order_relaxed) == context) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && wide_cluster) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess && context) done.context[dev].store(context, std::memory_order_relaxed);
    return e;
}

size_t compression_bytes(const rkv_desc_t *d, int budget, int buffer, int alpha);     // scratch of a compression alone; 0: invalid

// launchers (one per stage); each returns cudaGetLastError() of its launch
cudaError_t launch_prep(const Params &p, cudaStream_t s);
cudaError_t launch_logits_sm100(Params p, cudaStream_t s);      // two-pass route, the scores without the stage before: Eq. 2-3's logits
cudaError_t launch_widen_keys(const Params &stored, __nv_bfloat16 *wide, int wide_d, const void *q_src, void *q_dst,
                              bool keys, cudaStream_t s);
cudaError_t launch_scores_simt(const Params &p, cudaStream_t s);
cudaError_t launch_scores_sm100(const Params &p, cudaStream_t s);
cudaError_t launch_scores_tri_sm100(const Params &p, cudaStream_t s);
cudaError_t launch_select(const Params &p, cudaStream_t s);
cudaError_t launch_gather(const Params &p, cudaStream_t s);
cudaError_t launch_append(void *k_cache, void *v_cache, const void *k_new, const void *v_new, int32_t *seq_lens, int batch,
                          int hkv, int cap, int row_bytes, int32_t *status, const int32_t *block_table, cudaStream_t s);
cudaError_t launch_push_query(void *q_window, const void *q_new, int batch, int hq, int alpha, int slot, int row_bytes,
                              cudaStream_t s);
cudaError_t launch_attend(const void *k_cache, const void *v_cache, const void *q_new, const int32_t *seq_lens, float *out,
                          float *partial, int batch, int hkv, int hq, int cap, int splits, int dtype, int32_t *status,
                          long long wait_cycles, const int32_t *block_table, long long pool_pages, int head_dim, int sms, cudaStream_t s);
cudaError_t launch_attend_tc(const void *k_cache, const void *v_cache, const void *q_new, const int32_t *seq_lens, float *out,
                             float *partial, int batch, int hkv, int hq, int cap, int splits, int32_t *status, long long wait_cycles,
                             const int32_t *block_table, long long pool_pages, int src, cudaStream_t s);
int attend_tc_splits(int heads, int cap, int sms);
int attend_max_group();
int attend_splits(int heads, int cap, int sms, int G, int dtype);
bool attend_supported(int G, int dtype, int head_dim);
int attend_tc_workspace_splits(int heads, int cap, int sms);
bool attend_tc_separate(int heads, int cap, int splits, int sms, int src);
size_t attend_workspace_bytes(int heads, int cap, int sms, int G, int dtype);      // for the partial results of the splits
bool scores_sm100_available();
long long sm100_default_wait_cycles();          // default limit of the kernels' bounded waits (about two seconds)
bool scores_dense_possible(int tiles, int beta);   // the symmetric route of the second pass may be taken (two more launches)
int scores_pass2_rounds(int tiles);            // list + scan rounds of the second scoring pass for caches of `tiles` key tiles
bool select_is_fused(int cap_pad, int alpha);   // the select stage is one kernel (small caches) instead of three

}  // namespace rkv
