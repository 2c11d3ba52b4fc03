// What the forms of the prep stage share (rkv_prep.cu: CUDA cores; rkv_prep_sm100.cu: tensor cores).
#pragma once

#include "rkv_sm100.cuh"

namespace rkv {

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

cudaError_t launch_head_sum(const Params &p, cudaStream_t s);
cudaError_t launch_prep_sm100(const Params &p, cudaStream_t s);       // bf16 keys of 64 and 128 dimensions, E4M3 codes of 128

}  // namespace rkv
