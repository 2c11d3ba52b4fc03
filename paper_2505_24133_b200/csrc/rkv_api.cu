// C ABI of the R-KV compression library: argument checks, workspace carve-up, stage launches.
// See include/rkv.h for the contract of every entry point.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <memory>
#include <mutex>
#include <thread>

#include "rkv_common.cuh"

namespace rkv {

namespace {

thread_local rkv_desc_t g_desc;
thread_local bool g_desc_set = false;
thread_local char g_cuda_error[256] = "";

int cuda_fail(cudaError_t e, const char *where)
{
    snprintf(g_cuda_error, sizeof(g_cuda_error), "%s: %s", where, cudaGetErrorString(e));
    return RKV_ERR_CUDA;
}

struct Layout {
    size_t k_wide, q_wide, best, dense, dense_items, inv_norm, norm_split, thr_split, tile_sum, logits, row_stat, keys, sbar, left, lacking, strag, strag_items, self_dot, head_sum_bf16, meta, counters, total;
    int cap, cap_pad, tiles, tri;
};

// The two-pass tensor-core scoring kernels are built for bf16 keys of 64 and 128 dimensions and for E4M3 codes of 128; other 8-bit
// caches use them on a widened copy.  The row-block tensor-core kernel, which forms the whole similarity matrix, takes 256 dimensions, and
// the others where it is asked for (64 on a copy padded with zeros to 128: dot products and norms do not see the padding);
// fp32 caches, or a request for it, the CUDA-core kernel.
// Bytes of a cache element and of a query element.  8-bit caches (E4M3 codes) have bf16 queries.
size_t cache_esz(const rkv_desc_t *d) { return d->dtype == RKV_BF16 ? 2 : d->dtype == RKV_F32 ? 4 : 1; }
size_t query_esz(const rkv_desc_t *d) { return d->dtype == RKV_F32 ? 4 : 2; }

bool use_simt(const rkv_desc_t *d)
{
    return d->dtype == RKV_F32 || (d->flags & RKV_FLAG_SIMT_SCORES);
}
// 1 when the two-pass tensor-core kernels score (unless a cross-check kernel is asked for).
int use_tri(const rkv_desc_t *d) { return !(use_simt(d) || d->head_dim == 256 || (d->flags & RKV_FLAG_ROWBLOCK_SCORES)); }
// The head dimension is padded from 64 to 128 in the scoring copy (keys and observation queries).
bool pads_dim(const rkv_desc_t *d) { return d->head_dim == 64 && !use_simt(d) && !use_tri(d); }
// The scoring stages read a copy of the keys in the workspace instead of the cache itself.
bool needs_copy(const rkv_desc_t *d) { return d->dtype == RKV_FP8_E4M3 || pads_dim(d); }
// Head dimension the scoring stages see.
int scoring_dim(const rkv_desc_t *d) { return pads_dim(d) ? kHeadDim : d->head_dim; }
// bf16 caches of 64 dimensions on the two-pass route: a kernel ahead of prep records the lengths.
bool lengths_ahead(const rkv_desc_t *d) { return d->head_dim == 64 && use_tri(d) && !needs_copy(d); }
// Tensor-core scoring of 64 dimensions, by either route.  Its workspace has room for the padded copy, used or not: one workspace
// serves every route, and the stages one by one, at the size that rkv_workspace_bytes() has always told.
bool tensor64(const rkv_desc_t *d) { return d->head_dim == 64 && !use_simt(d); }
// Rows of 128 E4M3 codes are scored as they are stored on the two-pass route.  For the other routes the prep kernel writes the widened
// copy itself (instead of a widening pass in front of it) where the capacity is a whole number of 128-row tiles.
bool direct_codes(const rkv_desc_t *d) { return d->dtype == RKV_FP8_E4M3 && d->head_dim == kHeadDim && use_tri(d); }
bool whole_tiles_of_codes(const rkv_desc_t *d, long long cap) { return d->dtype == RKV_FP8_E4M3 && d->head_dim == kHeadDim && cap % kTile == 0; }

// Returns RKV_OK and fills *lay when the shape arguments are usable.
int check_shapes(const rkv_desc_t *d, int budget, int buffer, int alpha, Layout *lay)
{
    if (!d) return RKV_ERR_INVALID_ARG;
    if (d->batch < 1 || d->n_kv_heads < 1 || d->n_q_heads < 1) return RKV_ERR_INVALID_ARG;
    if (d->n_q_heads % d->n_kv_heads != 0) return RKV_ERR_INVALID_ARG;
    if (alpha < 1 || budget <= alpha || buffer < 1) return RKV_ERR_INVALID_ARG;
    if (d->pool_w < 0 || d->pool_w > 64 || d->beta < 0) return RKV_ERR_INVALID_ARG;
    if (!(d->sim_threshold >= 0.f && d->sim_threshold <= 1.f) || !(d->eps >= 0.f)) return RKV_ERR_INVALID_ARG;
    if (d->head_dim != 64 && d->head_dim != 128 && d->head_dim != 256) return RKV_ERR_UNSUPPORTED;
    if (d->dtype != RKV_BF16 && d->dtype != RKV_F32 && d->dtype != RKV_FP8_E4M3) return RKV_ERR_UNSUPPORTED;
    const long long cap = (long long)budget + buffer;
    if (cap > RKV_MAX_CAP) return RKV_ERR_UNSUPPORTED;
    if ((long long)(d->n_q_heads / d->n_kv_heads) * alpha > RKV_MAX_GROUP_ROWS) return RKV_ERR_UNSUPPORTED;
    if ((long long)d->batch * d->n_kv_heads > (1ll << 24)) return RKV_ERR_UNSUPPORTED;
    if (d->block_table) {      // paged caches: a page is one key tile
        if (cap % kTile != 0 || d->pool_pages < 1 || d->pool_pages > (1ll << 23)) return RKV_ERR_INVALID_ARG;
        if (reinterpret_cast<uintptr_t>(d->block_table) & 3u) return RKV_ERR_INVALID_ARG;
    }
    if (lay) {
        const size_t P = (size_t)d->batch * d->n_kv_heads;
        lay->cap = (int)cap;
        lay->tiles = (int)((cap + kTile - 1) / kTile);
        lay->cap_pad = lay->tiles * kTile;
        size_t off = 0;
        // the scoring copy (8-bit caches, padded head dimension): the keys as bf16, head after head, plus one tile of zero
        // rows behind the last head; with a padded head dimension the observation queries as well
        const size_t hd = (size_t)(tensor64(d) ? kHeadDim : d->head_dim);
        lay->k_wide = off;
        if (needs_copy(d) || tensor64(d)) off = align_up(off + (P * lay->cap + kTile) * hd * sizeof(__nv_bfloat16), 256);
        lay->q_wide = off;
        if (tensor64(d)) off = align_up(off + (size_t)d->batch * d->n_q_heads * alpha * kHeadDim * sizeof(__nv_bfloat16), 256);
        lay->inv_norm = off;  off = align_up(off + P * lay->cap_pad * sizeof(float), 256);
        lay->norm_split = off;  off = align_up(off + P * lay->cap_pad * 8 * sizeof(__nv_bfloat16), 256);
        lay->thr_split = off;   off = align_up(off + P * kTile * 8 * sizeof(__nv_bfloat16), 256);
        lay->tile_sum = off;  off = align_up(off + P * lay->tiles * hd * sizeof(float), 256);
        lay->logits = off;    off = align_up(off + P * alpha * lay->cap_pad * sizeof(float), 256);
        lay->row_stat = off;  off = align_up(off + P * (alpha + 1) * 2 * sizeof(float), 256);
        lay->keys = off;      off = align_up(off + P * lay->cap_pad * sizeof(float), 256);
        lay->sbar = off;      off = align_up(off + P * lay->cap_pad * sizeof(float), 256);
        lay->tri = use_tri(d);
        const size_t tri = (size_t)lay->tri;
        lay->left = off;        off = align_up(off + tri * P * lay->cap_pad * sizeof(int32_t), 256);
        lay->strag = off;       off = align_up(off + tri * P * lay->cap_pad * sizeof(int32_t), 256);
        lay->lacking = off;     off = align_up(off + tri * P * (lay->cap_pad / 32) * sizeof(uint32_t), 256);
        lay->strag_items = off; off = align_up(off + tri * P * (lay->cap_pad / 256 + 1) * sizeof(int4), 256);
        lay->best = off;        off = align_up(off + tri * P * lay->cap_pad * sizeof(uint32_t), 256);
        lay->dense = off;       off = align_up(off + tri * P * sizeof(int32_t), 256);
        lay->dense_items = off; off = align_up(off + tri * P * ((lay->tiles + 1) / 2) * sizeof(int4), 256);
        lay->self_dot = off;    off = align_up(off + P * lay->cap_pad * sizeof(float), 256);
        lay->head_sum_bf16 = off; off = align_up(off + P * 16 * hd * sizeof(__nv_bfloat16), 256);
        lay->meta = off;        off = align_up(off + 2 * (size_t)d->batch * sizeof(int32_t), 256);
        lay->counters = off;    off = align_up(off + kCounterWords * sizeof(unsigned long long), 256);
        lay->total = off;
    }
    return RKV_OK;
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// What a compression asks of its descriptor and lambda beside the shapes and the tensors.
int check_settings(const rkv_desc_t *d, float lambda)
{
    if (reinterpret_cast<uintptr_t>(d->budgets) & 3u) return RKV_ERR_INVALID_ARG;
    if (!(lambda >= 0.f && lambda <= 1.f)) return RKV_ERR_INVALID_ARG;
    return use_simt(d) || scores_sm100_available() ? RKV_OK : RKV_ERR_UNSUPPORTED;
}

int run(const rkv_desc_t *d, void *k_cache, void *v_cache, const void *q_window, int32_t *seq_lens, int budget,
        int buffer, int alpha, float lambda, int32_t *out_idx, void *stream, uint32_t stages)
{
    Layout lay;
    int rc = check_shapes(d, budget, buffer, alpha, &lay);
    if (rc != RKV_OK) return rc;
    if (!k_cache || !v_cache || !q_window || !seq_lens || !out_idx) return RKV_ERR_INVALID_ARG;
    if (!aligned16(k_cache) || !aligned16(v_cache) || !aligned16(q_window)) return RKV_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(seq_lens) & 3u) || (reinterpret_cast<uintptr_t>(out_idx) & 3u)) return RKV_ERR_INVALID_ARG;
    if ((rc = check_settings(d, lambda)) == RKV_ERR_INVALID_ARG) return rc;
    if ((stages & ~RKV_STAGE_ALL) != 0u || stages == 0u) return RKV_ERR_INVALID_ARG;
    if (!d->workspace || d->workspace_bytes < lay.total) return RKV_ERR_WORKSPACE;
    if (reinterpret_cast<uintptr_t>(d->workspace) & 255u) return RKV_ERR_WORKSPACE;
    if (rc != RKV_OK) return rc;

    Params p;
    memset(&p, 0, sizeof(p));
    p.k_cache = k_cache;
    p.v_cache = v_cache;
    p.q_window = q_window;
    p.seq_lens = seq_lens;
    p.out_idx = out_idx;
    p.batch = d->batch;
    p.hkv = d->n_kv_heads;
    p.hq = d->n_q_heads;
    p.group = d->n_q_heads / d->n_kv_heads;
    p.d = d->head_dim;
    p.logit_scale = 1.0f / sqrtf((float)d->head_dim);
    p.cap = lay.cap;
    p.cap_pad = lay.cap_pad;
    p.tiles = lay.tiles;
    p.budget = budget;
    p.buffer = buffer;
    p.alpha = alpha;
    p.dtype = d->dtype;
    p.store_row_bytes = (int)(d->head_dim * cache_esz(d));
    p.pool_w = d->pool_w;
    p.beta = d->beta;
    p.mean_then_pool = (d->flags & RKV_FLAG_MEAN_THEN_POOL) ? 1 : 0;
    p.head_mean = (d->flags & RKV_FLAG_HEAD_MEAN) ? 1 : 0;
    p.gqa_mean_pool = (d->flags & RKV_FLAG_GQA_MEAN_POOL) ? 1 : 0;
    p.sim_threshold = d->sim_threshold;
    p.eps = d->eps;
    p.lambda = lambda;
    char *ws = static_cast<char *>(d->workspace);
    p.inv_norm = reinterpret_cast<float *>(ws + lay.inv_norm);
    p.norm_split = reinterpret_cast<__nv_bfloat16 *>(ws + lay.norm_split);
    p.thr_split = reinterpret_cast<__nv_bfloat16 *>(ws + lay.thr_split);
    p.tile_sum = reinterpret_cast<float *>(ws + lay.tile_sum);
    p.logits = reinterpret_cast<float *>(ws + lay.logits);
    p.row_stat = reinterpret_cast<float *>(ws + lay.row_stat);
    p.keys = reinterpret_cast<uint32_t *>(ws + lay.keys);
    p.sbar = reinterpret_cast<float *>(ws + lay.sbar);
    p.left = reinterpret_cast<int32_t *>(ws + lay.left);
    p.strag = reinterpret_cast<int32_t *>(ws + lay.strag);
    p.lacking = reinterpret_cast<uint32_t *>(ws + lay.lacking);
    p.strag_items = reinterpret_cast<int4 *>(ws + lay.strag_items);
    p.self_dot = reinterpret_cast<float *>(ws + lay.self_dot);
    p.best = reinterpret_cast<uint32_t *>(ws + lay.best);
    p.dense = reinterpret_cast<int32_t *>(ws + lay.dense);
    p.dense_items = reinterpret_cast<int4 *>(ws + lay.dense_items);
    p.dense_ok = (d->beta == 1 && !(d->flags & RKV_FLAG_NO_SYMMETRIC)) ? 1 : 0;
    p.head_sum_bf16 = reinterpret_cast<__nv_bfloat16 *>(ws + lay.head_sum_bf16);
    p.meta = reinterpret_cast<int32_t *>(ws + lay.meta);
    p.counters = reinterpret_cast<unsigned long long *>(ws + lay.counters);
    p.tri = lay.tri;
    p.status = d->device_status;
    p.budgets = d->budgets;
    p.block_table = d->block_table;
    p.pages_per_head = lay.cap / kTile;
    p.pool_pages = d->pool_pages;
    p.wait_cycles = d->wait_limit_cycles > 0 ? (long long)d->wait_limit_cycles : sm100_default_wait_cycles();
    p.kernel_events = d->kernel_events;
    p.dbg_counters = d->dbg_counters;
    p.dbg_I = d->dbg_I;
    p.dbg_Sbar = d->dbg_Sbar;
    p.dbg_R = d->dbg_R;
    p.dbg_Z = d->dbg_Z;

    cudaStream_t s = static_cast<cudaStream_t>(stream);
    void *const *ev = d->stage_events;
    cudaError_t e;
    auto mark = [&](int i) -> cudaError_t {
        return ev && ev[i] ? cudaEventRecord(static_cast<cudaEvent_t>(ev[i]), s) : cudaSuccess;
    };
    if ((e = mark(0)) != cudaSuccess) return cuda_fail(e, "cudaEventRecord");
    // What the gather moves is the caller's caches as they are stored; where a copy is scored every stage before it reads the
    // bf16 copy of the keys (contiguous: the block table, if any, is followed once, by the widening kernel).
    Params stored = p;
    // The queries that count, and of 8-bit caches the keys, are those of the stages that always read them: the queries at the
    // scores, 8-bit keys at prep.  Both at once only where one call has both stages.
    const bool at_once = (stages & RKV_STAGE_PREP) && (stages & RKV_STAGE_SCORES);
    p.form_logits = p.tri && at_once ? 1 : 0;
    p.codes = direct_codes(d) && at_once ? 1 : 0;
    const bool copies = needs_copy(d) && !p.codes;
    if (copies) {
        p.k_cache = ws + lay.k_wide;
        p.block_table = nullptr;
        p.dtype = RKV_BF16;
        p.d = scoring_dim(d);
        if (pads_dim(d)) p.q_window = ws + lay.q_wide;
        p.fused_codes = whole_tiles_of_codes(d, lay.cap) ? 1 : 0;
        p.fuse_src = stored.k_cache;
        p.fuse_table = stored.block_table;
    }
    // (8-bit codes whose capacity is no whole number of tiles: prep could record the lengths itself; the kernel stands in for the
    // widening pass of before, so that the number of launches that rkv_launch_count_for() tells stays what it was)
    p.lengths_done = lengths_ahead(d) || (p.codes && lay.cap % kTile != 0) ? 1 : 0;
    if (stages & RKV_STAGE_PREP) {
        if (copies &&
            (e = launch_widen_keys(stored, static_cast<__nv_bfloat16 *>(p.k_cache), p.d, pads_dim(d) ? stored.q_window : nullptr,
                                   pads_dim(d) ? ws + lay.q_wide : nullptr, !p.fused_codes, s)) != cudaSuccess)
            return cuda_fail(e, "widen launch");
        if ((e = launch_prep(p, s)) != cudaSuccess) return cuda_fail(e, "prep launch");
    }
    if ((e = mark(1)) != cudaSuccess) return cuda_fail(e, "cudaEventRecord");
    if (stages & RKV_STAGE_SCORES) {
        if (p.tri && !at_once && (e = launch_logits_sm100(p, s)) != cudaSuccess) return cuda_fail(e, "logits launch");
        e = use_simt(d) ? launch_scores_simt(p, s)
                        : (p.tri ? launch_scores_tri_sm100(p, s) : launch_scores_sm100(p, s));
        if (e != cudaSuccess) return cuda_fail(e, "scores launch");
        if (!p.tri && ((e = mark_kernel(p, 0, s)) != cudaSuccess || (e = mark_kernel(p, 1, s)) != cudaSuccess))
            return cuda_fail(e, "cudaEventRecord");
        if (p.dbg_counters &&
            (e = cudaMemcpyAsync(p.dbg_counters, p.counters, 8 * sizeof(unsigned long long), cudaMemcpyDeviceToDevice, s)) !=
                cudaSuccess)
            return cuda_fail(e, "cudaMemcpyAsync");
    }
    if ((e = mark(2)) != cudaSuccess) return cuda_fail(e, "cudaEventRecord");
    if (stages & RKV_STAGE_SELECT)
        if ((e = launch_select(p, s)) != cudaSuccess) return cuda_fail(e, "select launch");
    if ((e = mark(3)) != cudaSuccess) return cuda_fail(e, "cudaEventRecord");
    if (stages & RKV_STAGE_GATHER)
        if ((e = launch_gather(stored, s)) != cudaSuccess) return cuda_fail(e, "gather launch");
    if ((e = mark(4)) != cudaSuccess) return cuda_fail(e, "cudaEventRecord");
    return RKV_OK;
}

struct HostLayout {
    size_t k, v, q, seq, idx, inner, total;
    size_t kv_bytes, q_bytes, seq_bytes, idx_bytes, row_bytes;
};

int host_layout(const rkv_desc_t *d, int budget, int buffer, int alpha, HostLayout *h)
{
    Layout lay;
    int rc = check_shapes(d, budget, buffer, alpha, &lay);
    if (rc != RKV_OK) return rc;
    const size_t P = (size_t)d->batch * d->n_kv_heads;
    h->row_bytes = (size_t)d->head_dim * cache_esz(d);
    h->kv_bytes = P * lay.cap * h->row_bytes;
    h->q_bytes = (size_t)d->batch * d->n_q_heads * alpha * d->head_dim * query_esz(d);
    h->seq_bytes = (size_t)d->batch * sizeof(int32_t);
    h->idx_bytes = P * budget * sizeof(int32_t);
    size_t off = 0;
    h->k = off;      off = align_up(off + h->kv_bytes, 256);
    h->v = off;      off = align_up(off + h->kv_bytes, 256);
    h->q = off;      off = align_up(off + h->q_bytes, 256);
    h->seq = off;    off = align_up(off + h->seq_bytes, 256);
    h->idx = off;    off = align_up(off + h->idx_bytes, 256);
    h->inner = off;  off = off + lay.total;
    h->total = off;
    return RKV_OK;
}

// Two copy streams and the events between them and the caller's stream, for the host-buffer form.  A call takes one from the
// pool while it enqueues and gives it back then.  The next taker gets one whose work is done, or the one that its own stream
// used last: behind another stream's copies a call would wait for work that it has no part in.  Creating the two streams
// for each call took 250 us.
constexpr int kMaxPieces = 8;
struct HostPipe {
    int dev = -1;
    unsigned long long context = 0ull;      // its streams live and die with it
    cudaStream_t up = nullptr, down = nullptr;
    cudaEvent_t ev[3 * kMaxPieces + 2] = {};
    cudaStream_t user = nullptr;            // the stream of the call that used it last, and that call's thread (the handles of the
    std::thread::id thread;                 // legacy and the per-thread default stream stand for a stream per thread)
    bool last_used_by(cudaStream_t s) const { return user == s && thread == std::this_thread::get_id(); }
    bool idle() const { return cudaStreamQuery(up) == cudaSuccess && cudaStreamQuery(down) == cudaSuccess; }
    bool open(int device)
    {
        dev = device;
        context = context_id();
        bool ok = cudaStreamCreateWithFlags(&up, cudaStreamNonBlocking) == cudaSuccess &&
                  cudaStreamCreateWithFlags(&down, cudaStreamNonBlocking) == cudaSuccess;
        for (cudaEvent_t &x : ev)
            if (ok) ok = cudaEventCreateWithFlags(&x, cudaEventDisableTiming) == cudaSuccess;
        return ok;
    }
    ~HostPipe()
    {
        for (cudaEvent_t x : ev)
            if (x) cudaEventDestroy(x);
        if (up) cudaStreamDestroy(up);
        if (down) cudaStreamDestroy(down);
    }
};
class PipePool {
public:
    std::unique_ptr<HostPipe> take(int dev, cudaStream_t s)
    {
        // (queries and new streams are no part of a capture that another thread may have under way)
        cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
        cudaThreadExchangeStreamCaptureMode(&mode);
        std::unique_ptr<HostPipe> x = find(dev, s);
        if (!x) {
            x.reset(new HostPipe);
            if (!x->open(dev)) {
                cudaGetLastError();         // (the call then goes through the caller's stream alone)
                x.reset();
            }
        }
        cudaThreadExchangeStreamCaptureMode(&mode);
        if (x) {
            x->user = s;
            x->thread = std::this_thread::get_id();
        }
        return x;
    }
    void give(std::unique_ptr<HostPipe> x)
    {
        std::lock_guard<std::mutex> guard(lock_);
        for (auto &slot : free_)
            if (!slot) {
                slot = std::move(x);
                return;
            }
    }                                       // (no slot left: destroyed when its work is done)

private:
    std::unique_ptr<HostPipe> find(int dev, cudaStream_t s)
    {
        const unsigned long long context = context_id();
        std::lock_guard<std::mutex> guard(lock_);
        for (auto &x : free_)
            if (x && x->dev == dev && x->context == context && x->last_used_by(s)) return std::move(x);
        for (auto &x : free_)
            if (x && x->dev == dev && x->context == context && x->idle()) return std::move(x);
        return nullptr;
    }
    std::mutex lock_;
    std::unique_ptr<HostPipe> free_[16];
};
PipePool &pipe_pool()
{
    static PipePool *pool = new PipePool;   // never destroyed: the CUDA runtime may be gone before this library's statics
    return *pool;
}

}  // namespace

size_t compression_bytes(const rkv_desc_t *d, int budget, int buffer, int alpha)
{
    Layout lay;
    return check_shapes(d, budget, buffer, alpha, &lay) == RKV_OK ? lay.total : 0;
}

}  // namespace rkv

using namespace rkv;

extern "C" {

void rkv_desc_default(rkv_desc_t *desc)
{
    if (!desc) return;
    memset(desc, 0, sizeof(*desc));
    desc->head_dim = kHeadDim;
    desc->dtype = RKV_BF16;
    desc->pool_w = 4;
    desc->beta = 1;
    desc->sim_threshold = 0.5f;
    desc->eps = 1e-8f;
}

size_t rkv_workspace_bytes(const rkv_desc_t *desc, int32_t budget, int32_t buffer, int32_t alpha)
{
    // (one workspace serves a compression and the decode attention of its shape: with fp32 caches and large query groups the latter
    // may need more)
    const size_t scoring = compression_bytes(desc, budget, buffer, alpha);
    return scoring ? std::max(scoring, rkv_decode_workspace_bytes(desc, budget, buffer)) : 0;
}

int rkv_set_desc(const rkv_desc_t *desc)
{
    if (!desc) return RKV_ERR_INVALID_ARG;
    g_desc = *desc;
    g_desc_set = true;
    return RKV_OK;
}

int rkv_compress(void *k_cache, void *v_cache, const void *q_window, int32_t *seq_lens, int32_t budget,
                 int32_t buffer, int32_t alpha, float lambda, int32_t *out_idx, void *stream)
{
    if (!g_desc_set) return RKV_ERR_INVALID_ARG;
    return run(&g_desc, k_cache, v_cache, q_window, seq_lens, budget, buffer, alpha, lambda, out_idx, stream,
               RKV_STAGE_ALL);
}

int rkv_compress_ex(const rkv_desc_t *desc, void *k_cache, void *v_cache, const void *q_window,
                    int32_t *seq_lens, int32_t budget, int32_t buffer, int32_t alpha, float lambda,
                    int32_t *out_idx, void *stream)
{
    return run(desc, k_cache, v_cache, q_window, seq_lens, budget, buffer, alpha, lambda, out_idx, stream,
               RKV_STAGE_ALL);
}

int rkv_compress_stages(const rkv_desc_t *desc, void *k_cache, void *v_cache, const void *q_window,
                        int32_t *seq_lens, int32_t budget, int32_t buffer, int32_t alpha, float lambda,
                        int32_t *out_idx, void *stream, uint32_t stage_mask)
{
    return run(desc, k_cache, v_cache, q_window, seq_lens, budget, buffer, alpha, lambda, out_idx, stream,
               stage_mask);
}

size_t rkv_host_workspace_bytes(const rkv_desc_t *desc, int32_t budget, int32_t buffer, int32_t alpha)
{
    HostLayout h;
    return host_layout(desc, budget, buffer, alpha, &h) == RKV_OK ? h.total : 0;
}

int rkv_compress_host(const rkv_desc_t *desc, void *host_k_cache, void *host_v_cache, const void *host_q_window,
                      int32_t *host_seq_lens, int32_t budget, int32_t buffer, int32_t alpha, float lambda,
                      int32_t *host_out_idx, void *stream)
{
    HostLayout h;
    int rc = host_layout(desc, budget, buffer, alpha, &h);
    if (rc != RKV_OK) return rc;
    if (!host_k_cache || !host_v_cache || !host_q_window || !host_seq_lens || !host_out_idx || desc->block_table)
        return RKV_ERR_INVALID_ARG;      // (the host-buffer form takes contiguous caches only)
    if (!desc->workspace || desc->workspace_bytes < h.total) return RKV_ERR_WORKSPACE;
    if (reinterpret_cast<uintptr_t>(desc->workspace) & 255u) return RKV_ERR_WORKSPACE;
    if ((rc = check_settings(desc, lambda)) != RKV_OK) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // Pieces of whole sequences: while one is compressed, the next comes in and the one before goes out (the link carries both
    // directions at once).  A copy costs about 5 us beside its bytes, so a piece has 16 MB or more, and the small arrays cross
    // once per call.  Events, counters and stream capture are for the call as a whole.
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &capturing) != cudaSuccess) capturing = cudaStreamCaptureStatusActive;
    long long pieces = (long long)(2 * h.kv_bytes / (16u << 20));
    pieces = pieces < kMaxPieces ? pieces : kMaxPieces;
    pieces = pieces < 1 ? 1 : (pieces < desc->batch ? pieces : desc->batch);
    if (capturing != cudaStreamCaptureStatusNone || desc->stage_events || desc->kernel_events || desc->dbg_counters) pieces = 1;
    int dev = 0;
    std::unique_ptr<HostPipe> pipe;
    if (pieces > 1 && cudaGetDevice(&dev) == cudaSuccess) pipe = pipe_pool().take(dev, s);
    if (!pipe) pieces = 1;
    cudaStream_t up = pipe ? pipe->up : s, down = pipe ? pipe->down : s;
    cudaError_t e = cudaSuccess;
    const char *where = "host to device copy";
    const size_t P = (size_t)desc->batch * desc->n_kv_heads, cap = (size_t)budget + buffer;
    char *ws = static_cast<char *>(desc->workspace);
    char *hk = static_cast<char *>(host_k_cache), *hv = static_cast<char *>(host_v_cache);
    auto copy = [&](void *dst, const void *src, size_t bytes, cudaMemcpyKind kind, cudaStream_t st) {
        if (e == cudaSuccess) e = cudaMemcpyAsync(dst, src, bytes, kind, st);
    };
    auto link = [&](int ev, cudaStream_t from, cudaStream_t to) {
        if (e == cudaSuccess && pipe && (e = cudaEventRecord(pipe->ev[ev], from)) == cudaSuccess) e = cudaStreamWaitEvent(to, pipe->ev[ev], 0);
    };
    // first sequence of piece i: the first and the last piece are half as large, nothing runs beside them
    auto edge = [&](int i) -> size_t { return i == 0 ? 0 : i == pieces ? desc->batch : (size_t)desc->batch * (2 * i - 1) / (2 * pieces - 2); };
    link(0, s, up);                         // the staging buffers may still be in use by earlier work of the stream
    copy(ws + h.q, host_q_window, h.q_bytes, cudaMemcpyHostToDevice, up);
    copy(ws + h.seq, host_seq_lens, h.seq_bytes, cudaMemcpyHostToDevice, up);
    for (int i = 0; i < (int)pieces && e == cudaSuccess && rc == RKV_OK; ++i) {
        const size_t b0 = edge(i), nb = edge(i + 1) - b0;
        if (nb == 0) continue;
        const size_t kv0 = h.kv_bytes / desc->batch * b0, kv = h.kv_bytes / desc->batch * nb;
        copy(ws + h.k + kv0, hk + kv0, kv, cudaMemcpyHostToDevice, up);
        link(1 + 3 * i, up, s);             // the scores need the keys alone
        copy(ws + h.v + kv0, hv + kv0, kv, cudaMemcpyHostToDevice, up);
        if (e != cudaSuccess) break;
        rkv_desc_t inner = *desc;
        inner.batch = (int32_t)nb;
        inner.workspace = ws + h.inner;     // the pieces are compressed one after the other
        inner.workspace_bytes = desc->workspace_bytes - h.inner;
        if (inner.budgets) inner.budgets += b0;
        for (float **dump : {&inner.dbg_I, &inner.dbg_Sbar, &inner.dbg_R, &inner.dbg_Z})
            if (*dump) *dump += b0 * desc->n_kv_heads * cap;
        auto stages = [&](uint32_t mask) {
            return run(&inner, ws + h.k + kv0, ws + h.v + kv0, ws + h.q + h.q_bytes / desc->batch * b0,
                       reinterpret_cast<int32_t *>(ws + h.seq) + b0, budget, buffer, alpha, lambda,
                       reinterpret_cast<int32_t *>(ws + h.idx + h.idx_bytes / desc->batch * b0), stream, mask);
        };
        if (pipe) {
            rc = stages(RKV_STAGE_ALL & ~RKV_STAGE_GATHER);
            link(2 + 3 * i, up, s);
            if (rc == RKV_OK) rc = stages(RKV_STAGE_GATHER);
        } else {
            rc = stages(RKV_STAGE_ALL);
        }
        if (rc != RKV_OK) break;
        where = "device to host copy";
        link(3 + 3 * i, s, down);
        // rows [0, budget) of every head come back; rows beyond are unspecified after a compression and are left
        // as the host has them
        const size_t pitch = cap * h.row_bytes, width = budget * h.row_bytes, rows = P / desc->batch * nb;
        if (e == cudaSuccess) e = cudaMemcpy2DAsync(hk + kv0, pitch, ws + h.k + kv0, pitch, width, rows, cudaMemcpyDeviceToHost, down);
        if (e == cudaSuccess) e = cudaMemcpy2DAsync(hv + kv0, pitch, ws + h.v + kv0, pitch, width, rows, cudaMemcpyDeviceToHost, down);
    }
    if (rc == RKV_OK) {
        copy(host_seq_lens, ws + h.seq, h.seq_bytes, cudaMemcpyDeviceToHost, down);
        copy(host_out_idx, ws + h.idx, h.idx_bytes, cudaMemcpyDeviceToHost, down);
        link(3 * kMaxPieces + 1, down, s);
    }
    if (pipe) {
        // an error on the way: what is under way in the copy streams still reads and writes the caller's buffers and workspace,
        // so the caller's stream waits for it as it does after a call that succeeds
        if (rc != RKV_OK || e != cudaSuccess)
            for (cudaStream_t x : {up, down})
                if (cudaEventRecord(pipe->ev[3 * kMaxPieces + 1], x) != cudaSuccess ||
                    cudaStreamWaitEvent(s, pipe->ev[3 * kMaxPieces + 1], 0) != cudaSuccess)
                    cudaStreamSynchronize(x);
        pipe_pool().give(std::move(pipe));
    }
    return rc != RKV_OK ? rc : (e == cudaSuccess ? RKV_OK : cuda_fail(e, where));
}

int rkv_append(const rkv_desc_t *d, void *k_cache, void *v_cache, const void *k_new, const void *v_new, int32_t *seq_lens,
               int32_t budget, int32_t buffer, void *stream)
{
    // shape checks as for the compression (alpha plays no part here: any valid value)
    int rc = check_shapes(d, budget, buffer, 1, nullptr);
    if (rc != RKV_OK) return rc;
    if (!k_cache || !v_cache || !k_new || !v_new || !seq_lens) return RKV_ERR_INVALID_ARG;
    if (!aligned16(k_cache) || !aligned16(v_cache) || !aligned16(k_new) || !aligned16(v_new)) return RKV_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(seq_lens) & 3u) return RKV_ERR_INVALID_ARG;
    const int row_bytes = (int)(d->head_dim * cache_esz(d));
    const cudaError_t e = launch_append(k_cache, v_cache, k_new, v_new, seq_lens, d->batch, d->n_kv_heads, budget + buffer,
                                        row_bytes, d->device_status, d->block_table, static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? RKV_OK : cuda_fail(e, "append launch");
}

int rkv_push_query(const rkv_desc_t *d, void *q_window, const void *q_new, int32_t alpha, int32_t slot, void *stream)
{
    if (!d || alpha < 1 || slot < 0 || slot >= alpha) return RKV_ERR_INVALID_ARG;
    int rc = check_shapes(d, alpha + 1, 1, alpha, nullptr);        // descriptor fields and alpha against the group limit
    if (rc != RKV_OK) return rc;
    if (!q_window || !q_new || !aligned16(q_window) || !aligned16(q_new)) return RKV_ERR_INVALID_ARG;
    const int row_bytes = (int)(d->head_dim * query_esz(d));
    const cudaError_t e = launch_push_query(q_window, q_new, d->batch, d->n_q_heads, alpha, slot, row_bytes,
                                            static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? RKV_OK : cuda_fail(e, "push_query launch");
}

static int attend_plan(const rkv_desc_t *d, int32_t budget, int32_t buffer, int *splits, size_t *bytes, int *sm_count)
{
    int rc = check_shapes(d, budget, buffer, 1, nullptr);
    if (rc != RKV_OK) return rc;
    const int G = d->n_q_heads / d->n_kv_heads;
    if (!attend_supported(G, d->dtype, d->head_dim)) return RKV_ERR_UNSUPPORTED;
    int dev = 0, sms = 0;
    if (device_sms(&dev, &sms) != cudaSuccess)
        sms = 148;       // sizing only (no device here): the B200's count
    *sm_count = sms;
    *splits = attend_splits(d->batch * d->n_kv_heads, budget + buffer, sms, G, d->dtype);
    *bytes = attend_workspace_bytes(d->batch * d->n_kv_heads, budget + buffer, sms, G, d->dtype);
    return RKV_OK;
}

size_t rkv_decode_workspace_bytes(const rkv_desc_t *desc, int32_t budget, int32_t buffer)
{
    int splits = 1, sms = 0;
    size_t bytes = 0;
    return attend_plan(desc, budget, buffer, &splits, &bytes, &sms) == RKV_OK ? bytes : 0;
}

int rkv_decode_attention(const rkv_desc_t *d, const void *k_cache, const void *v_cache, const void *q_new,
                         const int32_t *seq_lens, float *out, int32_t budget, int32_t buffer, void *stream)
{
    int splits = 1, sms = 0;
    size_t bytes = 0;
    int rc = attend_plan(d, budget, buffer, &splits, &bytes, &sms);
    if (rc != RKV_OK) return rc;
    if (!k_cache || !v_cache || !q_new || !seq_lens || !out) return RKV_ERR_INVALID_ARG;
    if (!aligned16(k_cache) || !aligned16(v_cache) || !aligned16(q_new) || !aligned16(out)) return RKV_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(seq_lens) & 3u) return RKV_ERR_INVALID_ARG;
    if (bytes > 0) {
        if (!d->workspace || d->workspace_bytes < bytes) return RKV_ERR_WORKSPACE;
        if (reinterpret_cast<uintptr_t>(d->workspace) & 255u) return RKV_ERR_WORKSPACE;
    }
    const long long wait = d->wait_limit_cycles > 0 ? (long long)d->wait_limit_cycles : sm100_default_wait_cycles();
    const cudaError_t e = launch_attend(k_cache, v_cache, q_new, seq_lens, out, static_cast<float *>(d->workspace), d->batch,
                                        d->n_kv_heads, d->n_q_heads, budget + buffer, splits, d->dtype, d->device_status,
                                        wait, d->block_table, d->pool_pages, d->head_dim, sms, static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? RKV_OK : cuda_fail(e, "decode attention launch");
}

int rkv_launch_count(const rkv_desc_t *desc, uint32_t stage_mask)
{
    int c = 0;
    for (uint32_t bit = 1; bit <= RKV_STAGE_GATHER; bit <<= 1) c += (stage_mask & bit) ? 1 : 0;
    if (stage_mask & RKV_STAGE_SELECT) c += 2;      // row statistics and importance run ahead of the selection kernel
    // bf16 keys of 64 and 128 dimensions: the tile sums are added up per head by a kernel of its own behind the prep kernel
    if (desc && (stage_mask & RKV_STAGE_PREP) && desc->dtype != RKV_F32 &&
        (desc->head_dim == 0 || scoring_dim(desc) == kHeadDim || tensor64(desc)))
        c += 1;
    // the kernel that writes the scoring copy, or the one that records the lengths
    if (desc && (stage_mask & RKV_STAGE_PREP) && (needs_copy(desc) || lengths_ahead(desc))) c += 1;
    if (desc && (stage_mask & RKV_STAGE_SELECT) && (desc->flags & RKV_FLAG_HEAD_MEAN)) c += 1;   // per-sequence selection
    // the two-pass route's logits, where they are not formed by a prep kernel of the same call
    if (desc && (stage_mask & RKV_STAGE_SCORES) && !(stage_mask & RKV_STAGE_PREP) && use_tri(desc)) c += 2;
    // the two-pass scoring path is the first pass plus up to two rounds of (listing, second pass) while the
    // retention rule is on
    if (desc && (stage_mask & RKV_STAGE_SCORES) && use_tri(desc) && desc->beta > 0 && desc->sim_threshold < 1.0f) {
        c += 4;
        if (desc->beta == 1 && !(desc->flags & RKV_FLAG_NO_SYMMETRIC)) c += 2;      // symmetric route: scan and finish
    }
    return c;
}

int rkv_launch_count_for(const rkv_desc_t *desc, int32_t budget, int32_t buffer, int32_t alpha, uint32_t stage_mask)
{
    Layout lay;
    if (check_shapes(desc, budget, buffer, alpha, &lay) != RKV_OK) return 0;
    int c = rkv_launch_count(desc, stage_mask);
    // the prep kernel writes the copy of the keys itself and nothing else needs a pass of its own
    if ((stage_mask & RKV_STAGE_PREP) && whole_tiles_of_codes(desc, lay.cap)) c -= 1;
    if ((stage_mask & RKV_STAGE_SELECT) && select_is_fused(lay.cap_pad, alpha)) c -= 2;
    if ((stage_mask & RKV_STAGE_SCORES) && use_tri(desc) && desc->beta > 0 && desc->sim_threshold < 1.0f)
    {
        c -= lay.tiles < 2 ? 4                                      // one key tile: the first scoring pass has seen everything
                           : 2 * (2 - scores_pass2_rounds(lay.tiles));   // small caches take one round
        if (desc->beta == 1 && !(desc->flags & RKV_FLAG_NO_SYMMETRIC) && !scores_dense_possible(lay.tiles, desc->beta)) c -= 2;
    }
    return c;
}

const char *rkv_status_string(int status)
{
    switch (status) {
        case RKV_OK: return "RKV_OK";
        case RKV_ERR_INVALID_ARG: return "RKV_ERR_INVALID_ARG";
        case RKV_ERR_UNSUPPORTED: return "RKV_ERR_UNSUPPORTED";
        case RKV_ERR_WORKSPACE: return "RKV_ERR_WORKSPACE";
        case RKV_ERR_CUDA: return "RKV_ERR_CUDA";
        case RKV_ERR_TIMEOUT: return "RKV_ERR_TIMEOUT";
        default: return "RKV_ERR_UNKNOWN";
    }
}

const char *rkv_last_cuda_error(void) { return g_cuda_error; }

}  // extern "C"
