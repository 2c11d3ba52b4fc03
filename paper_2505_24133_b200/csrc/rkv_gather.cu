// Stage "gather": Algorithm 1's gather + concatenate, done in place.
//
// For every head, row j of K and of V becomes row idx[j] (j < budget).  idx is strictly ascending, so
// idx[j] >= j: rows only move towards lower positions and the untouched prefix (idx[j] == j) is free.  A stream is one of
// the caches of one head; rows go through it in chunks, in ascending order: a chunk's stores only touch rows that no later
// chunk reads, so a chunk may be stored once it and the chunks before it have been read.  No scratch copy, no
// reallocation.  HBM-bound: kept rows read and written once.
// The stream of (KV head 0, K) also stores the new length, seq_lens[b] = budget.
//
// Two kernels.  gather_bulk_kernel: bulk copies through shared memory, eight streams per block, a loading and a storing warp
// each, a block per SM.  What is kept comes in runs (a few per cent of the rows are dropped), so a chunk is one to three copies in
// and one copy out, and the bytes in flight cost neither registers nor issue slots.  gather_kernel: 16-byte loads and stores by
// threads, a block per stream, or four that take a column slice of its rows each.  Which one a call takes is a matter of how
// many streams there are and how long a row is (launch_gather_for; us for 1024 to 4096 rows per stream, in the call):
//   streams x rows of bytes    160 x 2048 x 256   160 x 2048 x 128   512 x 4096 x 256   4096 x 2048 x 256   8192 x 4096 x 256
//   bulk                              45                 33               168                 694               2800
//   threads, four slices              35                 25               207                 837               3486
//   threads, a block per stream       72                 39               213                 698               2768
//                            24576 x 4096 x 256   8192 x 4096 x 128  16384 x 2048 x 128   8192 x 1024 x 512
//   bulk                            8490               1400                1408                1386
//   threads, a block per stream     8090               1563                1519                1792
// The bulk kernel on fewer SMs is no rule to go by: somewhere between 100 and 122 blocks, differently on different GPUs of the type,
// lies a step of 10 % (8192 streams of 256-byte rows with 120 blocks: 2620, 2760, 2875 and 2940 us on four of them, with 111 blocks 2725 on
// one and 2940 on another; by threads 2768-2772 on all).
#include <algorithm>

#include "rkv_sm100.cuh"

namespace rkv {

namespace {

using namespace sm100;

// ---- bulk copies -------------------------------------------------------------------------------------------------------
constexpr int kBulkStreams = 8;                              // streams of a block at a time
constexpr int kBulkThreads = 2 * kBulkStreams * 32;
constexpr int kBulkBytes = 24 * 1024;                        // buffers of a stream
constexpr int kBulkSmem = kBulkStreams * kBulkBytes;

template <int kRowBytes>
__global__ void __launch_bounds__(kBulkThreads, 1) gather_bulk_kernel(Params p, int streams)
{
    constexpr int kRows = 8192 / kRowBytes < 32 ? 8192 / kRowBytes : 32;        // rows of a chunk: a lane each, 8 KB at most
    constexpr int kChunk = kRows * kRowBytes;
    constexpr int kBufs = kBulkBytes / kChunk;
    static_assert(kTile % kRows == 0, "a chunk never crosses a page");
    extern __shared__ __align__(128) uint8_t bulk_smem[];
    __shared__ __align__(8) unsigned long long bars[kBulkStreams][2][kBufs];    // chunk landed; chunk read out
    __shared__ int abort_flag;
    // (no wait here is cut short by a caller's limit: a stream that is given up half-way is lost)
    const ErrSink sink{p.status, p.counters + kAbortWord, kWaitCycles};
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int w = warp % kBulkStreams;
    const bool loads = warp < kBulkStreams;
    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int i = 0; i < kBulkStreams; ++i)
            for (int b = 0; b < kBufs; ++b) {
                mbar_init(smem_u32(&bars[i][0][b]), 1);
                mbar_init(smem_u32(&bars[i][1][b]), 1);
            }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    pdl_trigger();
    pdl_wait();
    if (call_aborted(p)) return;                    // a bounded wait ran out earlier in this call: caches and lengths stay as they are
    const uint32_t base = smem_u32(bulk_smem) + w * kBulkBytes;
    const uint32_t full = smem_u32(&bars[w][0][0]), empty = smem_u32(&bars[w][1][0]);
    uint32_t count = 0;                             // chunks of this warp so far
    bool ok = true;
    for (int stream = blockIdx.x + w * gridDim.x; stream < streams && ok; stream += gridDim.x * kBulkStreams) {
        const int head = stream >> 1, which = stream & 1, b = head / p.hkv;
        const int budget = seq_budget(p, b);
        if (p.meta[b] <= budget) continue;          // nothing was selected for this sequence
        uint8_t *cache = static_cast<uint8_t *>(which ? p.v_cache : p.k_cache);
        const int32_t *idx = p.out_idx + (size_t)head * p.budget;
        const int chunks = (budget + kRows - 1) / kRows;
        // the chunks that are in place already are a prefix (idx[j] - j never decreases)
        int c0 = 0;
        for (;; c0 += 32) {
            const int last = min((c0 + lane + 1) * kRows, budget) - 1;
            const unsigned moved = __ballot_sync(0xffffffffu, c0 + lane >= chunks || idx[last] != last);
            if (moved) {
                c0 += __ffs(moved) - 1;
                break;
            }
        }
        if (loads) {
            auto fetch = [&](int c) -> int {        // the chunk's source rows, a lane each; fetched two chunks ahead
                const int j = c * kRows + lane;
                return lane < kRows && j < budget ? idx[j] : -1;
            };
            int next = fetch(c0), next2 = fetch(c0 + 1);
            for (int c = c0; c < chunks; ++c, ++count) {
                const int rows = min(kRows, budget - c * kRows);
                const int cur = next;
                next = next2;
                next2 = fetch(c + 2);
                // a copy per run of consecutive rows (a run also ends with a page)
                const int prev = __shfl_up_sync(0xffffffffu, cur, 1);
                const bool start = lane < rows && (lane == 0 || cur != prev + 1 || (p.block_table && cur % kTile == 0));
                const unsigned starts = __ballot_sync(0xffffffffu, start);
                const unsigned above = lane < 31 ? starts >> (lane + 1) : 0u;
                const int len = above ? __ffs(above) : rows - lane;
                const long long row = start ? row_index(p, head, cur) : 0;
                const uint32_t buf = count % kBufs;
                ok = __all_sync(0xffffffffu, mbar_wait(empty + 8u * buf, ((count / kBufs) & 1u) ^ 1u, &abort_flag, sink));
                if (!ok) break;
                if (lane == 0) mbar_expect_tx(full + 8u * buf, (uint32_t)(rows * kRowBytes));
                __syncwarp();
                if (start)
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 ::"r"(base + buf * kChunk + lane * kRowBytes), "l"(cache + row * kRowBytes), "r"(len * kRowBytes), "r"(full + 8u * buf)
                                 : "memory");
            }
        } else if (lane == 0) {
            if (which == 0 && head % p.hkv == 0) p.seq_lens[b] = budget;
            int old = -1;                           // the buffer whose store may still be reading it
            for (int c = c0; c < chunks; ++c, ++count) {
                const int rows = min(kRows, budget - c * kRows);
                const long long row = row_index(p, head, c * kRows);
                const uint32_t buf = count % kBufs;
                if (!(ok = mbar_wait(full + 8u * buf, (count / kBufs) & 1u, &abort_flag, sink))) break;
                asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                             ::"l"(cache + row * kRowBytes), "r"(base + buf * kChunk), "r"(rows * kRowBytes) : "memory");
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                if (old >= 0) mbar_arrive(empty + 8u * old);
                old = (int)buf;
            }
            asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
            if (old >= 0) mbar_arrive(empty + 8u * old);
        }
        ok = __all_sync(0xffffffffu, ok);
    }
    if (abort_flag) __nanosleep(200000);            // error path only: let the copies in flight land
}

// ---- threads -----------------------------------------------------------------------------------------------------------
constexpr int kGatherThreads = 256;

// kVecPerRow: 16-byte vectors per row: 4 (8-bit, d = 64) .. 64 (fp32, d = 256).  kSplit: column slices of a row (disjoint bytes: no
// ordering among them).
template <int kVecPerRow, int kSplit>
__global__ void __launch_bounds__(kGatherThreads) gather_kernel(Params p)
{
    constexpr int kChunkRows = 64 * kSplit;             // of 256 bytes: 16 KB in flight per block
    constexpr int kVecPerSlice = kVecPerRow / kSplit;
    constexpr int kVecPerThread = kChunkRows * kVecPerSlice / kGatherThreads;
    constexpr int kRowsPerStep = kGatherThreads / kVecPerSlice;
    pdl_trigger();
    pdl_wait();
    const int slice = blockIdx.x % kSplit;
    const int stream = blockIdx.x / kSplit;
    const int head = stream >> 1;
    const int which = stream & 1;
    const int b = head / p.hkv;
    const int budget_b = seq_budget(p, b);
    if (p.meta[b] <= budget_b) return;
    if (call_aborted(p)) return;
    if (which == 0 && slice == 0 && head % p.hkv == 0 && threadIdx.x == 0) p.seq_lens[b] = budget_b;

    // rows are addressed through row_index(): head after head, or page by page for paged caches
    uint4 *base = reinterpret_cast<uint4 *>(which ? p.v_cache : p.k_cache) + slice * kVecPerSlice;
    const int32_t *idx = p.out_idx + (size_t)head * p.budget;
    const int lane_vec = threadIdx.x % kVecPerSlice;
    const int lane_row = threadIdx.x / kVecPerSlice;

    for (int j0 = 0; j0 < budget_b; j0 += kChunkRows) {
        const int j_end = min(j0 + kChunkRows, budget_b);
        if (idx[j_end - 1] == j_end - 1) continue;   // ascending and idx[j] >= j: the whole chunk is in place
        uint4 held[kVecPerThread];
        int src[kVecPerThread];
#pragma unroll
        for (int q = 0; q < kVecPerThread; ++q) {
            const int j = j0 + q * kRowsPerStep + lane_row;
            src[q] = (j < j_end) ? idx[j] : -1;
            if (src[q] >= 0 && src[q] != j) held[q] = base[(size_t)row_index(p, head, src[q]) * kVecPerRow + lane_vec];
        }
        __syncthreads();                             // every source row of the chunk is in registers
#pragma unroll
        for (int q = 0; q < kVecPerThread; ++q) {
            const int j = j0 + q * kRowsPerStep + lane_row;
            if (src[q] >= 0 && src[q] != j) base[(size_t)row_index(p, head, j) * kVecPerRow + lane_vec] = held[q];
        }
    }
}

template <int kVecPerRow>
cudaError_t launch_gather_for(const Params &p, cudaStream_t s)
{
    const unsigned streams = 2u * (unsigned)(p.batch * p.hkv);
    int dev = 0, sms = 0;
    cudaError_t e = device_sms(&dev, &sms);
    if (e != cudaSuccess) return e;
    // Few streams: what a block of either kernel keeps in flight does not fill the chip, so a row is cut into slices (wide rows fill
    // a slice's chunk by themselves: from a stream per SM on they are the bulk kernel's).
    if (streams <= (unsigned)(kVecPerRow <= 16 ? sms * 3 / 2 : sms))
        return launch_early(gather_kernel<kVecPerRow, 4>, streams * 4, kGatherThreads, 0, s, 1, p);
    // Rows of 256 bytes in many streams: the thread kernel keeps as much in flight as the bulk kernel, and turns between reading and
    // writing less often.
    if constexpr (kVecPerRow == 16)
        if (streams >= 4096u) return launch_early(gather_kernel<kVecPerRow, 1>, streams, kGatherThreads, 0, s, 1, p);
    static PerDevice done;
    if ((e = allow_smem_once(done, dev, gather_bulk_kernel<kVecPerRow * 16>, kBulkSmem)) != cudaSuccess) return e;
    return launch_early(gather_bulk_kernel<kVecPerRow * 16>, std::min(streams, (unsigned)sms), kBulkThreads, (size_t)kBulkSmem, s, 1, p,
                        (int)streams);
}

}  // namespace

cudaError_t launch_gather(const Params &p, cudaStream_t s)
{
    switch (p.store_row_bytes / 16) {
        case 4: return launch_gather_for<4>(p, s);
        case 8: return launch_gather_for<8>(p, s);
        case 16: return launch_gather_for<16>(p, s);
        case 32: return launch_gather_for<32>(p, s);
        case 64: return launch_gather_for<64>(p, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace rkv
