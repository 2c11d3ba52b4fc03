// The two cache updates of a decode step that surround the compression (Section 3.1: newly generated tokens enter the
// buffer part of the cache; Algorithm 1's observation buffer M_alpha holds the last alpha queries).  Plain byte
// movement, one 16-byte vector per thread.
#include "rkv_common.cuh"

namespace rkv {

namespace {

constexpr int kDecThreads = 256;
constexpr int kOneBlockVecs = 8192;     // 16-byte vectors of a sequence's new rows, for K and for V

// k_new / v_new [batch][hkv][row_vecs] -> row seq_lens[b] of every head of sequence b, then seq_lens[b] += 1.  One block per
// sequence: the length changes behind the block's own barrier, when every copy has read it (as two launches, copies and
// lengths, the call took 2.5 us more).  Where a sequence has more rows than a block moves in that time (kOneBlockVecs: one
// sequence of 512 heads of 256 bytes 8.6 us, of 1024 11.5 instead of 10), several blocks share them and bump_kernel follows.
template <bool kShared>                    // several blocks per sequence
__global__ void __launch_bounds__(kDecThreads) append_kernel(uint4 *k_cache, uint4 *v_cache, const uint4 *k_new,
                                                             const uint4 *v_new, int32_t *seq_lens, int hkv, int cap,
                                                             int row_vecs, int parts, int32_t *status, const int32_t *block_table)
{
    pdl_trigger();
    pdl_wait();
    const int b = kShared ? blockIdx.x / parts : blockIdx.x, part = kShared ? blockIdx.x % parts : 0;
    const int L = seq_lens[b];
    const int vecs = hkv * row_vecs, x0 = part * kDecThreads + threadIdx.x;
    uint4 k0, v0;                           // the first vectors are under way together with the length (8 heads: 1.47 -> 1.14 us a call in a graph)
    if (x0 < vecs) {
        k0 = k_new[(size_t)b * vecs + x0];
        v0 = v_new[(size_t)b * vecs + x0];
    }
    if (L < 0 || L >= cap) {
        if (threadIdx.x == 0 && part == 0) report(status, RKV_ERR_INVALID_ARG);        // the cache of this sequence is full (or its length invalid)
        return;
    }
    for (int x = x0; x < vecs; x += (kShared ? parts : 1) * kDecThreads) {
        const int head = b * hkv + x / row_vecs, vec = x % row_vecs;
        // row L of the head: head after head, or through the block table (pages of kTile rows) for paged caches
        const size_t row = block_table ? (size_t)block_table[(size_t)head * (cap / kTile) + L / kTile] * kTile + L % kTile
                                       : (size_t)head * cap + L;
        const size_t src = (size_t)b * vecs + x, dst = row * row_vecs + vec;
        k_cache[dst] = x == x0 ? k0 : k_new[src];
        v_cache[dst] = x == x0 ? v0 : v_new[src];
    }
    if (kShared) return;
    __syncthreads();
    if (threadIdx.x == 0) seq_lens[b] = L + 1;
}

// seq_lens[b] += 1 for the sequences that took the new token, when the blocks that share a sequence are through
__global__ void __launch_bounds__(kDecThreads) bump_kernel(int32_t *seq_lens, int batch, int cap)
{
    pdl_trigger();
    pdl_wait();
    const int b = blockIdx.x * kDecThreads + threadIdx.x;
    if (b >= batch) return;
    const int L = seq_lens[b];
    if (L >= 0 && L < cap) seq_lens[b] = L + 1;
}

// q_new [batch][hq][row_vecs] -> row `slot` of every query head's window [batch][hq][alpha][row_vecs]
__global__ void __launch_bounds__(kDecThreads) push_query_kernel(uint4 *q_window, const uint4 *q_new, long long total,
                                                                 int alpha, int slot, int row_vecs)
{
    pdl_trigger();
    pdl_wait();
    const long long t = (long long)blockIdx.x * kDecThreads + threadIdx.x;
    if (t >= total) return;
    const int vec = (int)(t % row_vecs);
    const long long qh = t / row_vecs;                  // b * hq + query head
    q_window[((size_t)qh * alpha + slot) * row_vecs + vec] = q_new[t];
}

}  // namespace

cudaError_t launch_append(void *k_cache, void *v_cache, const void *k_new, const void *v_new, int32_t *seq_lens, int batch,
                          int hkv, int cap, int row_bytes, int32_t *status, const int32_t *block_table, cudaStream_t s)
{
    const int row_vecs = row_bytes / 16, vecs = hkv * row_vecs;
    const int parts = vecs <= kOneBlockVecs ? 1 : (vecs + kDecThreads - 1) / kDecThreads;
    cudaError_t e = launch_early(parts > 1 ? append_kernel<true> : append_kernel<false>, (unsigned)batch * (unsigned)parts, kDecThreads, 0, s, 1, static_cast<uint4 *>(k_cache),
                                 static_cast<uint4 *>(v_cache), static_cast<const uint4 *>(k_new), static_cast<const uint4 *>(v_new),
                                 seq_lens, hkv, cap, row_vecs, parts, status, block_table);
    if (e != cudaSuccess || parts == 1) return e;
    return launch_early(bump_kernel, (unsigned)((batch + kDecThreads - 1) / kDecThreads), kDecThreads, 0, s, 1, seq_lens, batch, cap);
}

cudaError_t launch_push_query(void *q_window, const void *q_new, int batch, int hq, int alpha, int slot, int row_bytes,
                              cudaStream_t s)
{
    const int row_vecs = row_bytes / 16;
    const long long total = (long long)batch * hq * row_vecs;
    const unsigned grid = (unsigned)((total + kDecThreads - 1) / kDecThreads);
    return launch_early(push_query_kernel, grid, kDecThreads, 0, s, 1, static_cast<uint4 *>(q_window),
                        static_cast<const uint4 *>(q_new), total, alpha, slot, row_vecs);
}

}  // namespace rkv
