// Stage "select": finishes the scores and picks the kept tokens.  Larger caches, three kernels:
//
//   row_stats   one warp per (head, row): the maximum and the sum of exponentials of the row's n values, i.e. a softmax in
//               two numbers -- the alpha rows of pooled logits (Eq. 3) and the row of column means (Eq. 6)
//   importance  eight consecutive tokens per thread (other windows than the default: a block per 1024 tokens of a head): Eq. 4's sliding max over {i-W .. i+W-1} per row (taken on the
//               logits: exp is monotone, so the max of the weights is the weight of the max), the softmax weight of
//               that maximum, mean over the alpha rows  -> I;  R of Eq. 6;  Eq. 7  Z = lambda I - (1 - lambda) R, left as
//               an order-preserving integer key
//   select      one block per head: exact k-th largest key by a radix select in shared memory; among equal scores the later
//               position is kept; the kept candidate positions are written in ascending order, then the alpha
//               observation positions.
//
// Small caches: one kernel, a block per head, with the pooled logits in shared memory.
// All of them read scratch that the stage before has just written (L2-resident for small batches).  The first two are bound
// by that memory, the selection by the latency of its barriers: many threads per block and as many blocks as fit.
// (4096 heads of 4216 tokens: 144 + 156 + 80 us; 147 + 129 + 199 while the selection did Eq. 6 and 7 itself and each of its
// threads walked and wrote a run of tokens one by one.  256 heads of 1144 tokens, the single kernel: 31 -> 20 us.)
#include "rkv_common.cuh"

namespace rkv {

namespace {

constexpr int kSelThreads = 512;

__device__ __forceinline__ uint32_t order_key(float z)
{
    // monotone map float -> uint32: larger float <=> larger key (-0 and +0 differ; harmless)
    uint32_t u = __float_as_uint(z);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float warp_max(float v)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, off));
    return v;
}
__device__ __forceinline__ float warp_sum(float v)
{
    // fixed reduction tree: the result does not depend on scheduling
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}
// The same over a block; scratch: a float per warp, free to be overwritten when the call before has returned everywhere.
template <int kThreads>
__device__ __forceinline__ float block_max(float v, float *scratch)
{
    v = warp_max(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = v;
    __syncthreads();
    return warp_max((threadIdx.x & 31) < kThreads / 32 ? scratch[threadIdx.x & 31] : -INFINITY);
}
template <int kThreads>
__device__ __forceinline__ float block_sum(float v, float *scratch)
{
    v = warp_sum(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = v;
    __syncthreads();
    return warp_sum((threadIdx.x & 31) < kThreads / 32 ? scratch[threadIdx.x & 31] : 0.f);
}

// What a lane takes its exponentials relative to: its running maximum, unless it has met nothing above -inf yet (a logit may be
// that low: it weighs nothing, where -inf - -inf would make the row's sum NaN).
__device__ __forceinline__ float finite_ref(float m) { return m == -INFINITY ? 0.f : m; }

// Eq. 6's column mean of a token: the two-pass scoring kernels leave the column sum minus the removed entries.
__device__ __forceinline__ float column_mean(const Params &p, float v, int n) { return p.tri ? v / (float)n : v; }

constexpr size_t kFusedSmemLimit = 64 * 1024;   // largest shared-memory footprint for the single-kernel form
constexpr int kStatThreads = 256;
constexpr int kImpThreads = 256;
constexpr int kImpTokens = 1024;     // tokens per importance block

// row_stat[head][j][0] = max of row j, [1] = 1 / sum exp(value - max); row alpha: the column means.  A warp per row, 1024
// values in flight, the sum kept relative to the running maximum of each lane (a block per row and its barriers: 184 us for
// 4096 heads of 4216 tokens; 157, and 144 since a last step no longer works on 128-value pieces that lie behind the row).
__global__ void __launch_bounds__(kStatThreads) row_stats_kernel(Params p)
{
    pdl_trigger();
    pdl_wait();
    const int rows = p.alpha + 1, lane = threadIdx.x & 31;
    const int unit = blockIdx.x * (kStatThreads / 32) + (threadIdx.x >> 5);
    const int head = unit / rows, j = unit % rows;
    if (head >= p.batch * p.hkv) return;
    const int n = seq_candidates(p, head / p.hkv);
    if (n == 0) return;
    const bool means = j == p.alpha;
    const float *row = means ? p.sbar + (size_t)head * p.cap_pad : p.logits + ((size_t)head * p.alpha + j) * p.cap_pad;
    const float scale = means && p.tri ? (float)n : 1.0f;          // (x / 1 is x)
    float m = -INFINITY, s = 0.f;
    for (int at = 0; at < n; at += 1024) {
        const int i0 = at + lane * 4;
        float4 v[8];
        float top = -INFINITY;
#pragma unroll
        for (int u = 0; u < 8; ++u)
            v[u] = i0 + u * 128 < n ? *reinterpret_cast<const float4 *>(row + i0 + u * 128) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = i0 + u * 128;
            if (at + u * 128 >= n) break;                          // (the warp as a whole: the rest of a last step is not worked on)
            if (means) v[u] = make_float4(v[u].x / scale, v[u].y / scale, v[u].z / scale, v[u].w / scale);
            if (i + 3 >= n) {
                if (i >= n) v[u].x = -INFINITY;
                if (i + 1 >= n) v[u].y = -INFINITY;
                if (i + 2 >= n) v[u].z = -INFINITY;
                v[u].w = -INFINITY;
            }
            top = fmaxf(fmaxf(top, v[u].x), fmaxf(fmaxf(v[u].y, v[u].z), v[u].w));
        }
        if (top > m) {
            s *= expf(m - top);
            m = top;
        }
        const float ref = finite_ref(m);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (at + u * 128 >= n) break;
            if (i0 + u * 128 < n) s += (expf(v[u].x - ref) + expf(v[u].y - ref)) + (expf(v[u].z - ref) + expf(v[u].w - ref));
        }
    }
    const float mw = warp_max(m);
    s = warp_sum(s == 0.f ? 0.f : s * expf(m - mw));               // (a lane without values: 0)
    if (lane == 0) {
        float *out = p.row_stat + ((size_t)head * rows + j) * 2;
        out[0] = mw;
        out[1] = 1.0f / s;
    }
}

// Eq. 6-7 of token i from its importance I and column mean sb (max m, inverse sum inv of their softmax): the integer key of
// Z, or Z itself where the heads of a sequence are averaged first.
__device__ __forceinline__ uint32_t joint_key(const Params &p, bool dump, int head, int i, float I, float sb, float m, float inv)
{
    const float R = expf(sb - m) * inv;
    const float Z = p.lambda * I - (1.0f - p.lambda) * R;
    if (dump) {
        const size_t dbg = (size_t)head * p.cap + i;
        if (p.dbg_I) p.dbg_I[dbg] = I;
        if (p.dbg_Sbar) p.dbg_Sbar[dbg] = sb;
        if (p.dbg_R) p.dbg_R[dbg] = R;
        if (p.dbg_Z) p.dbg_Z[dbg] = Z;
    }
    return p.head_mean ? __float_as_uint(Z) : order_key(Z);
}
__device__ __forceinline__ bool dumps(const Params &p) { return p.dbg_I || p.dbg_Sbar || p.dbg_R || p.dbg_Z; }

// Eq. 4, 6 and 7 for kImpTokens tokens of one head.
__global__ void __launch_bounds__(kImpThreads) importance_kernel(Params p)
{
    pdl_trigger();
    pdl_wait();
    const int chunks = (p.cap + kImpTokens - 1) / kImpTokens;
    const int head = blockIdx.x / chunks, i0 = (blockIdx.x % chunks) * kImpTokens;
    const int n = seq_candidates(p, head / p.hkv);
    if (i0 >= n) return;
    const int W = p.pool_w;
    const float *logits = p.logits + (size_t)head * p.alpha * p.cap_pad;
    const float *stat = p.row_stat + (size_t)head * (p.alpha + 1) * 2;
    const float *sbar = p.sbar + (size_t)head * p.cap_pad;
    uint32_t *keys = p.keys + (size_t)head * p.cap_pad;
    const float inv_alpha = 1.0f / (float)p.alpha;
    for (int i = i0 + threadIdx.x; i < min(i0 + kImpTokens, n); i += kImpThreads) {
        const int lo = max(i - W, 0), hi = min(i + W - 1, n - 1);
        float I = 0.f;
        if (p.mean_then_pool) {
            // Algorithm 1's order: the mean of the alpha softmax weights at each position of the window, then the max
            for (int u = min(lo, i); u <= max(hi, i); ++u) {
                float mean = 0.f;
                for (int j = 0; j < p.alpha; ++j)
                    mean += expf(logits[(size_t)j * p.cap_pad + u] - stat[2 * j]) * stat[2 * j + 1];
                I = fmaxf(I, mean * inv_alpha);
            }
        } else {
            for (int j = 0; j < p.alpha; ++j) {
                const float *row = logits + (size_t)j * p.cap_pad;
                float best = row[i];
                for (int u = lo; u <= hi; ++u) best = fmaxf(best, row[u]);
                I += expf(best - stat[2 * j]) * stat[2 * j + 1];
            }
            I *= inv_alpha;
        }
        keys[i] = joint_key(p, dumps(p), head, i, I, column_mean(p, sbar[i], n), stat[2 * p.alpha], stat[2 * p.alpha + 1]);
    }
}

// The eight maxima of Eq. 4 with the default window W = 4 (positions i-4 .. i+3) for tokens i0 .. i0+7 from the 16 logits at
// i0-4 .. i0+11, by a doubling scheme; positions that are no candidates hold -inf.
__device__ __forceinline__ void window_max8(const float (&x)[16], float (&best)[8])
{
    float m2[15], m4[13];
#pragma unroll
    for (int u = 0; u < 15; ++u) m2[u] = fmaxf(x[u], x[u + 1]);
#pragma unroll
    for (int u = 0; u < 13; ++u) m4[u] = fmaxf(m2[u], m2[u + 2]);
#pragma unroll
    for (int t = 0; t < 8; ++t) best[t] = fmaxf(m4[t], m4[t + 4]);        // x[t .. t+7]
}
// the 16 logits around i0 (a multiple of 8) of a row, -inf beyond the candidates [0, n)
__device__ __forceinline__ void window_load(const float *row, int i0, int n, int cap_pad, float (&x)[16])
{
    const float4 none = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    const float4 *r4 = reinterpret_cast<const float4 *>(row + i0);
    const float4 a = i0 >= 4 ? r4[-1] : none, b = r4[0], c = r4[1];          // i0 + 7 < cap_pad (a multiple of 128)
    const float4 d = i0 + 8 < cap_pad ? r4[2] : none;
    x[0] = a.x, x[1] = a.y, x[2] = a.z, x[3] = a.w, x[4] = b.x, x[5] = b.y, x[6] = b.z, x[7] = b.w;
    x[8] = c.x, x[9] = c.y, x[10] = c.z, x[11] = c.w, x[12] = d.x, x[13] = d.y, x[14] = d.z, x[15] = d.w;
    if (i0 < 4 || i0 + 11 >= n) {
#pragma unroll
        for (int u = 0; u < 16; ++u) {
            const int pos = i0 - 4 + u;
            if (pos < 0 || pos >= n) x[u] = -INFINITY;
        }
    }
}

// The default window: eight consecutive tokens per thread, per query row four 16-byte loads for the 16 logits their windows
// cover (the general kernel above reads each logit nine times).
constexpr int kImp8Threads = 256;

// Threads go over the groups of eight tokens of all heads in a row (a block per 2048 tokens of a head left every second or third
// block almost empty: 177 us for 8192 heads of 2168 tokens, 162 now).
__global__ void __launch_bounds__(kImp8Threads) importance_w4_kernel(Params p)
{
    pdl_trigger();
    pdl_wait();
    const int groups = (p.cap + 7) / 8;
    const long long unit = (long long)blockIdx.x * kImp8Threads + threadIdx.x;
    if (unit >= (long long)p.batch * p.hkv * groups) return;
    const int head = (int)(unit / groups);
    const int i0 = (int)(unit % groups) * 8;     // first token of this thread
    const int n = seq_candidates(p, head / p.hkv);
    if (i0 >= n) return;
    const float *logits = p.logits + (size_t)head * p.alpha * p.cap_pad;
    const float *stat = p.row_stat + (size_t)head * (p.alpha + 1) * 2;
    float acc[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) acc[t] = 0.f;
#pragma unroll 2
    for (int j = 0; j < p.alpha; ++j) {
        float x[16], best[8];
        window_load(logits + (size_t)j * p.cap_pad, i0, n, p.cap_pad, x);
        window_max8(x, best);
        const float mj = stat[2 * j], inv = stat[2 * j + 1];
#pragma unroll
        for (int t = 0; t < 8; ++t) acc[t] += expf(best[t] - mj) * inv;
    }
    const float inv_alpha = 1.0f / (float)p.alpha, m = stat[2 * p.alpha], inv_r = stat[2 * p.alpha + 1];
    const bool dump = dumps(p);
    const float4 *s4 = reinterpret_cast<const float4 *>(p.sbar + (size_t)head * p.cap_pad + i0);
    const float4 sa = s4[0], sc = s4[1];
    const float sb[8] = {sa.x, sa.y, sa.z, sa.w, sc.x, sc.y, sc.z, sc.w};
    uint32_t key[8];
#pragma unroll
    for (int t = 0; t < 8; ++t)
        key[t] = i0 + t < n ? joint_key(p, dump, head, i0 + t, acc[t] * inv_alpha, column_mean(p, sb[t], n), m, inv_r) : 0u;
    uint4 *out = reinterpret_cast<uint4 *>(p.keys + (size_t)head * p.cap_pad + i0);
    out[0] = make_uint4(key[0], key[1], key[2], key[3]);
    out[1] = make_uint4(key[4], key[5], key[6], key[7]);
}

// Exact top-k over n order-preserving keys in shared memory (written by the caller, one owner per slot; no barrier
// needed before the call; lo, hi: bounds of this thread's keys), later position first among equal keys.  Writes the k kept
// positions in ascending order and then the alpha observation positions n .. n+alpha-1 into `copies` index lists of
// `budget` entries, `budget` apart.
// The digits are taken from the distance to the smallest key, from its highest bit that occurs: scores of one head lie close
// together, and their common leading bits would be passes without an effect.
template <int kThreads>
__device__ __forceinline__ void radix_select_emit(const uint32_t *keys, uint32_t lo, uint32_t hi, int n, int k, int alpha, int budget,
                                                  int32_t *out, int copies)
{
    constexpr int kWarps = kThreads / 32;
    __shared__ uint32_t hist[4][256];
    __shared__ uint32_t bound[2][kWarps];
    __shared__ uint32_t sel_prefix, sel_want;
    __shared__ uint32_t warp_tot[kWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int t = tid; t < 4 * 256; t += kThreads) (&hist[0][0])[t] = 0u;
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) {
        bound[0][warp] = lo;
        bound[1][warp] = hi;
    }
    if (tid == 0) {
        sel_prefix = 0u;
        sel_want = (uint32_t)k;
    }
    __syncthreads();
    lo = __reduce_min_sync(0xffffffffu, bound[0][lane % kWarps]);
    hi = __reduce_max_sync(0xffffffffu, bound[1][lane % kWarps]);

    // ---- radix select: the k-th largest distance, 8 bits at a time from the top
    const int bits = 32 - __clz(hi - lo);
    int pass = 0;
    for (int top = bits; top > 0; top -= 8, ++pass) {
        const int shift = max(top - 8, 0);
        const uint32_t prefix = sel_prefix;
        const uint32_t high_mask = top >= 32 ? 0u : 0xffffffffu << top;
        for (int i = tid; i < n; i += kThreads) {
            const uint32_t key = keys[i] - lo;
            if ((key & high_mask) == prefix) atomicAdd(&hist[pass][(key & ~high_mask) >> shift], 1u);
        }
        __syncthreads();
        if (tid < 32) {
            // lane l owns digits 255-8l .. 248-8l (descending); find the digit holding the want-th key
            const uint32_t want = sel_want;        // read before any lane may overwrite it below
            uint32_t local[8], sum = 0u;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                local[e] = hist[pass][255 - (tid * 8 + e)];
                sum += local[e];
            }
            uint32_t incl = sum;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t o = __shfl_up_sync(0xffffffffu, incl, off);
                if (tid >= off) incl += o;
            }
            uint32_t run = incl - sum;             // keys in larger digits, owned by earlier lanes
            __syncwarp();
#pragma unroll
            for (int e = 0; e < 8; ++e) {          // exactly one (lane, e) holds the want-th key
                if (run < want && want <= run + local[e]) {
                    sel_prefix = prefix | ((uint32_t)(255 - (tid * 8 + e)) << shift);
                    sel_want = want - run;
                }
                run += local[e];
            }
        }
        __syncthreads();
    }
    const uint32_t theta = lo + sel_prefix;   // key of the k-th largest score
    const uint32_t need_eq = sel_want;        // how many tokens equal to theta are kept (the latest ones)

    // ---- emit the kept positions in ascending order: a contiguous piece per warp, 32 tokens at a time
    const int piece = ((n + kThreads - 1) / kThreads) * 32;
    const int first = warp * piece, last = min(first + piece, n);
    uint32_t gt = 0u, eq = 0u;
    for (int i = first; i < last; i += 32) {
        const uint32_t key = i + lane < last ? keys[i + lane] : 0u;
        gt += __popc(__ballot_sync(0xffffffffu, i + lane < last && key > theta));
        eq += __popc(__ballot_sync(0xffffffffu, i + lane < last && key == theta));
    }
    if (lane == 0) warp_tot[warp] = (gt << 16) | eq;     // n <= 8192: both counts fit 16 bits, sums never carry across
    __syncthreads();
    const uint32_t wsum = lane < kWarps ? warp_tot[lane] : 0u;
    const uint32_t excl = __reduce_add_sync(0xffffffffu, lane < warp ? wsum : 0u);
    const uint32_t skip_eq = (__reduce_add_sync(0xffffffffu, wsum) & 0xffffu) - need_eq;    // the earliest ties are the ones dropped
    uint32_t g = excl >> 16, q = excl & 0xffffu;
    const uint32_t below = (1u << lane) - 1u;
    for (int i = first; i < last; i += 32) {
        const uint32_t key = i + lane < last ? keys[i + lane] : 0u;
        const bool over = i + lane < last && key > theta, tie = i + lane < last && key == theta;
        const uint32_t over_mask = __ballot_sync(0xffffffffu, over), tie_mask = __ballot_sync(0xffffffffu, tie);
        const uint32_t ties = q + __popc(tie_mask & below);
        if (over || (tie && ties >= skip_eq)) {
            const uint32_t at = g + __popc(over_mask & below) + (ties > skip_eq ? ties - skip_eq : 0u);
            for (int c = 0; c < copies; ++c) out[(size_t)c * budget + at] = i + lane;
        }
        g += __popc(over_mask);
        q += __popc(tie_mask);
    }
    for (int j = tid; j < alpha; j += kThreads)
        for (int c = 0; c < copies; ++c) out[(size_t)c * budget + k + j] = n + j;   // observation tokens
    for (int j = k + alpha + tid; j < budget; j += kThreads)                     // a sequence with a smaller budget of its own
        for (int c = 0; c < copies; ++c) out[(size_t)c * budget + j] = -1;
}

// What a block writes for a head that is not selected from (true): -1 after a wait that ran out in an earlier stage (the
// scores are incomplete), the identity list under Algorithm 1's guard, and -1 for an invalid length.
template <int kThreads>
__device__ __forceinline__ bool settled(const Params &p, int head, int32_t *out)
{
    const int b = head / p.hkv, L = p.meta[b];
    const bool aborted = call_aborted(p);
    if (!aborted && L > seq_budget(p, b)) return false;
    for (int j = threadIdx.x; j < p.budget; j += kThreads) out[j] = (!aborted && j < L) ? j : -1;
    return true;
}

// (what a block waits for is its own barriers: with half the threads twice the blocks are under way.  8192 heads of 2168
// tokens: 136 us with 512, 98; 4096 heads of 4216: 104, 80.)
constexpr int kPickThreads = 256;
__global__ void __launch_bounds__(kPickThreads, 8) select_kernel(Params p)
{
    extern __shared__ uint4 sel_smem[];            // [cap_pad] keys
    pdl_trigger();
    pdl_wait();
    const int head = blockIdx.x, b = head / p.hkv;
    int32_t *out = p.out_idx + (size_t)head * p.budget;
    if (settled<kPickThreads>(p, head, out)) return;
    if (p.head_mean) return;                       // select_mean_kernel picks the sequence's positions
    const int budget_b = seq_budget(p, b), n = p.meta[b] - p.alpha;
    const uint4 *src = reinterpret_cast<const uint4 *>(p.keys + (size_t)head * p.cap_pad);
    uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll 4
    for (int v = threadIdx.x; v * 4 < n; v += kPickThreads) {
        const uint4 k4 = src[v];
        sel_smem[v] = k4;
        lo = min(lo, k4.x);
        hi = max(hi, k4.x);
        if (v * 4 + 1 < n) lo = min(lo, k4.y), hi = max(hi, k4.y);
        if (v * 4 + 2 < n) lo = min(lo, k4.z), hi = max(hi, k4.z);
        if (v * 4 + 3 < n) lo = min(lo, k4.w), hi = max(hi, k4.w);
    }
    radix_select_emit<kPickThreads>(reinterpret_cast<const uint32_t *>(sel_smem), lo, hi, n, budget_b - p.alpha, p.alpha, p.budget, out, 1);
}

// Small caches: the three steps in one block per head, the pooled logits in shared memory.
// 512 threads where the heads do not fill the chip (the fastest for one head), 256 where blocks queue up: what they wait for is
// mostly their own barriers and loads, and twice as many are under way.
template <int kThreads>
__global__ void __launch_bounds__(kThreads, 1024 / kThreads) select_fused_kernel(Params p)
{
    constexpr int kWarps = kThreads / 32;
    extern __shared__ uint4 sel_smem[];            // [cap_pad] column means, then keys; [cap_pad] means of weights; [alpha][cap_pad] logits
    __shared__ float part[4 * RKV_MAX_GROUP_ROWS];          // a row's two halves: maximum, sum of exponentials
    __shared__ float stat[2 * RKV_MAX_GROUP_ROWS];
    __shared__ float scratch[kWarps];
    pdl_trigger();
    pdl_wait();
    const int head = blockIdx.x, b = head / p.hkv;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int32_t *out = p.out_idx + (size_t)head * p.budget;
    if (settled<kThreads>(p, head, out)) return;
    const int budget_b = seq_budget(p, b), n = p.meta[b] - p.alpha;
    float *row = reinterpret_cast<float *>(sel_smem), *weight = row + p.cap_pad, *lg = row + 2 * p.cap_pad;
    const float *logits = p.logits + (size_t)head * p.alpha * p.cap_pad;
    const float *sbar = p.sbar + (size_t)head * p.cap_pad;

    // ---- Eq. 6: the column means and their maximum
    float m = -INFINITY;
    for (int i = tid; i < n; i += kThreads) {
        const float v = column_mean(p, sbar[i], n);
        row[i] = v;
        m = fmaxf(m, v);
    }
    // ---- Eq. 3: two warps per query row, half of it each, 512 values in flight
    const int half_n = ((n + 255) / 256) * 128;
    for (int q = warp; q < 2 * p.alpha; q += kWarps) {
        const float *src = logits + (size_t)(q >> 1) * p.cap_pad;
        float *dst = lg + (size_t)(q >> 1) * p.cap_pad;
        const int end = (q & 1) ? n : min(half_n, n);
        float mj = -INFINITY, sj = 0.f;
        for (int i0 = (q & 1) * half_n + lane * 4; i0 < end; i0 += 512) {
            float4 v[4];
            float top = -INFINITY;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (i0 + u * 128 < end) v[u] = *reinterpret_cast<const float4 *>(src + i0 + u * 128);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = i0 + u * 128;
                if (i >= end) break;
                if (i + 1 >= n) v[u].y = -INFINITY;
                if (i + 2 >= n) v[u].z = -INFINITY;
                if (i + 3 >= n) v[u].w = -INFINITY;
                *reinterpret_cast<float4 *>(dst + i) = v[u];
                top = fmaxf(fmaxf(top, v[u].x), fmaxf(fmaxf(v[u].y, v[u].z), v[u].w));
            }
            if (top > mj) {
                sj *= expf(mj - top);
                mj = top;
            }
            const float ref = finite_ref(mj);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (i0 + u * 128 >= end) break;
                sj += (expf(v[u].x - ref) + expf(v[u].y - ref)) + (expf(v[u].z - ref) + expf(v[u].w - ref));
            }
        }
        const float mw = warp_max(mj);
        const float sw = warp_sum(sj == 0.f ? 0.f : sj * expf(mj - mw));        // (a lane without values: 0)
        if (lane == 0) {
            part[2 * q] = mw;
            part[2 * q + 1] = sw;
        }
    }
    m = block_max<kThreads>(m, scratch);        // (its barriers also close the loops above)
    for (int j = tid; j < p.alpha; j += kThreads) {
        const float m0 = part[4 * j], m1 = part[4 * j + 2], mj = fmaxf(m0, m1);
        const float s0 = part[4 * j + 1], s1 = part[4 * j + 3];
        stat[2 * j] = mj;
        stat[2 * j + 1] = 1.0f / ((s0 == 0.f ? 0.f : s0 * expf(m0 - mj)) + (s1 == 0.f ? 0.f : s1 * expf(m1 - mj)));
    }
    float s = 0.f;
    for (int i = tid; i < n; i += kThreads) s += expf(row[i] - m);
    s = block_sum<kThreads>(s, scratch);
    const float inv = 1.0f / s;

    // ---- Eq. 4 and 7; the key of a token takes the place of its column mean
    uint32_t *keys = reinterpret_cast<uint32_t *>(row);
    const float inv_alpha = 1.0f / (float)p.alpha;
    const int W = p.pool_w;
    const bool dump = dumps(p);
    uint32_t lo = 0xffffffffu, hi = 0u;
    auto finish = [&](int i, float I) {
        const uint32_t key = joint_key(p, dump, head, i, I, row[i], m, inv);
        if (p.head_mean) p.keys[(size_t)head * p.cap_pad + i] = key;
        keys[i] = key;
        lo = min(lo, key);
        hi = max(hi, key);
    };
    if (p.mean_then_pool) {
        // Algorithm 1's order: the mean of the alpha softmax weights per position, then the max over the window
        for (int i = tid; i < n; i += kThreads) {
            float mean = 0.f;
            for (int j = 0; j < p.alpha; ++j) mean += expf(lg[j * p.cap_pad + i] - stat[2 * j]) * stat[2 * j + 1];
            weight[i] = mean * inv_alpha;
        }
        __syncthreads();
        for (int i = tid; i < n; i += kThreads) {
            float best = weight[i];
            for (int u = max(i - W, 0); u <= min(i + W - 1, n - 1); ++u) best = fmaxf(best, weight[u]);
            finish(i, best);
        }
    } else if (W == 4) {
        // eight tokens and half of the query rows per thread; the pair of threads adds its halves up
        for (int t0 = 0; t0 < n; t0 += kThreads * 4) {
            const int i0 = t0 + (tid >> 1) * 8;
            float acc[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) acc[t] = 0.f;
            if (i0 < n)
                for (int j = tid & 1; j < p.alpha; j += 2) {
                    float x[16], best[8];
                    window_load(lg + (size_t)j * p.cap_pad, i0, n, p.cap_pad, x);
                    window_max8(x, best);
                    const float mj = stat[2 * j], invj = stat[2 * j + 1];
#pragma unroll
                    for (int t = 0; t < 8; ++t) acc[t] += expf(best[t] - mj) * invj;
                }
#pragma unroll
            for (int t = 0; t < 8; ++t) acc[t] += __shfl_xor_sync(0xffffffffu, acc[t], 1);
#pragma unroll
            for (int t = 0; t < 8; ++t)
                if ((t & 1) == (tid & 1) && i0 + t < n) finish(i0 + t, acc[t] * inv_alpha);
        }
    } else {
        for (int i = tid; i < n; i += kThreads) {
            const int first = max(i - W, 0), last = min(i + W - 1, n - 1);
            float acc = 0.f;
            for (int j = 0; j < p.alpha; ++j) {
                const float *r = lg + j * p.cap_pad;
                float best = r[i];
                for (int u = first; u <= last; ++u) best = fmaxf(best, r[u]);
                acc += expf(best - stat[2 * j]) * stat[2 * j + 1];
            }
            finish(i, acc * inv_alpha);
        }
    }
    if (p.head_mean) return;      // Z of this head is in p.keys; select_mean_kernel picks the sequence's positions
    radix_select_emit<kThreads>(keys, lo, hi, n, budget_b - p.alpha, p.alpha, p.budget, out, 1);
}

// Algorithm 1's aggregated selection, one block per sequence: AggScore_i = mean over the KV heads of Z_i^h (left in
// p.keys by the kernels above), exact top-k on it, the same index list written for every head of the sequence.
__global__ void __launch_bounds__(kSelThreads, 4) select_mean_kernel(Params p)
{
    extern __shared__ uint4 sel_smem[];
    pdl_trigger();
    pdl_wait();
    const int b = blockIdx.x, tid = threadIdx.x;
    const int L = p.meta[b];
    if (call_aborted(p)) return;    // the selection before has written -1 everywhere
    if (L <= seq_budget(p, b)) return;      // ... or the identity lists
    const int n = L - p.alpha;
    uint32_t *keys = reinterpret_cast<uint32_t *>(sel_smem);
    const float *z = reinterpret_cast<const float *>(p.keys) + (size_t)b * p.hkv * p.cap_pad;
    const float hkv = (float)p.hkv;
    uint32_t lo = 0xffffffffu, hi = 0u;
    for (int i = tid; i < n; i += kSelThreads) {
        float acc = 0.f;
        for (int h = 0; h < p.hkv; ++h) acc += z[(size_t)h * p.cap_pad + i];      // fixed head order
        keys[i] = order_key(acc / hkv);
        lo = min(lo, keys[i]);
        hi = max(hi, keys[i]);
    }
    radix_select_emit<kSelThreads>(keys, lo, hi, n, seq_budget(p, b) - p.alpha, p.alpha, p.budget, p.out_idx + (size_t)b * p.hkv * p.budget, p.hkv);
}

}  // namespace

bool select_is_fused(int cap_pad, int alpha) { return (size_t)(alpha + 2) * cap_pad * sizeof(float) <= kFusedSmemLimit; }

static cudaError_t launch_select_mean(const Params &p, cudaStream_t s)
{
    // (up to 32 KB of shared memory: RKV_MAX_CAP words)
    return launch_early(select_mean_kernel, (unsigned)p.batch, kSelThreads, (size_t)p.cap_pad * sizeof(float), s, 1, p);
}

template <int kThreads>
static cudaError_t launch_fused(const Params &p, unsigned heads, int dev, cudaStream_t s)
{
    static PerDevice done;
    const cudaError_t e = allow_smem_once(done, dev, select_fused_kernel<kThreads>, (int)kFusedSmemLimit);
    if (e != cudaSuccess) return e;
    return launch_early(select_fused_kernel<kThreads>, heads, kThreads, (size_t)(p.alpha + 2) * p.cap_pad * sizeof(float), s, 1, p);
}

cudaError_t launch_select(const Params &p, cudaStream_t s)
{
    const unsigned heads = (unsigned)(p.batch * p.hkv);
    int dev = 0, sms = 0;
    cudaError_t e = device_sms(&dev, &sms);
    if (e != cudaSuccess) return e;
    if (select_is_fused(p.cap_pad, p.alpha)) {
        if ((e = mark_kernel(p, 2, s)) != cudaSuccess || (e = mark_kernel(p, 3, s)) != cudaSuccess) return e;
        e = heads > 2u * (unsigned)sms ? launch_fused<256>(p, heads, dev, s) : launch_fused<kSelThreads>(p, heads, dev, s);
        if (e != cudaSuccess) return e;
        return p.head_mean ? launch_select_mean(p, s) : cudaSuccess;
    }
    if ((e = launch_early(row_stats_kernel, (heads * (unsigned)(p.alpha + 1) + kStatThreads / 32 - 1) / (kStatThreads / 32), kStatThreads, 0, s, 1, p)) != cudaSuccess) return e;
    if ((e = mark_kernel(p, 2, s)) != cudaSuccess) return e;
    if (p.pool_w == 4 && !p.mean_then_pool)
        e = launch_early(importance_w4_kernel, (unsigned)(((unsigned long long)heads * ((p.cap + 7) / 8) + kImp8Threads - 1) / kImp8Threads), kImp8Threads, 0,
                         s, 1, p);
    else
        e = launch_early(importance_kernel, heads * (unsigned)((p.cap + kImpTokens - 1) / kImpTokens), kImpThreads, 0, s, 1, p);
    if (e != cudaSuccess) return e;
    if ((e = mark_kernel(p, 3, s)) != cudaSuccess) return e;
    if ((e = launch_early(select_kernel, heads, kPickThreads, (size_t)p.cap_pad * sizeof(float), s, 1, p)) != cudaSuccess) return e;
    return p.head_mean ? launch_select_mean(p, s) : cudaSuccess;
}

}  // namespace rkv
