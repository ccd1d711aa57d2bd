// finish.cuh -- the final sum over task results, in a kernel of its own
// (generic.cu) or at the end of an eliminated walk (handed to NVRTC with core.cuh).
#pragma once

#include "core.cuh"

namespace pk {

// The sum of the threads' accumulators, in every thread, in a fixed order.
template <class A>
__device__ __forceinline__ typename A::Acc block_sum(typename A::Acc acc, u64 *sh) {
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) acc = A::acc_add(acc, A::shfl_down(acc, d));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
    if (lane == 0) A::acc_store(sh + warp * A::ACC_WORDS, acc);
    __syncthreads();
    acc = A::acc_load(sh);
    for (int w = 1; w < nw; ++w) acc = A::acc_add(acc, A::acc_load(sh + w * A::ACC_WORDS));
    return acc;
}

// An accumulator that another block stored during this launch.
template <class A>
__device__ __forceinline__ typename A::Acc acc_load_l2(const u64 *src) {
    u64 w[A::ACC_WORDS];
#pragma unroll
    for (int i = 0; i < A::ACC_WORDS; ++i) w[i] = __ldcg(src + i);
    return A::acc_load(w);
}

// Whether this block is the last of the launch to get here (what the blocks
// stored before is then visible to it).  Nothing waits.
__device__ __forceinline__ bool last_block(u64 *done_blocks) {
    __shared__ int last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(done_blocks, 1ull) == gridDim.x - 1;
        __threadfence();
    }
    __syncthreads();
    return last != 0;
}

// The end of a plan's walk in the walk's own launch: the last block sums the
// task results, writes the result words where the host reads them (pinned
// memory: skipped blocks, result, abort flag at their workspace places) and
// clears the workspace counters for the next launch.  A compute is then one
// launch: no reset, no second kernel, no copy back (n=24 0/1, 2^14 outer steps:
// 51 -> 38 us a call).
template <class A>
__device__ __forceinline__ void finish_walk(const FinishArgs &f) {
    if (!f.host) return;
    __shared__ u64 sh[32 * A::ACC_WORDS];
    if (!last_block(f.ws + 7)) return;
    typename A::Acc acc = A::acc_zero();
    constexpr int kAhead = 8;   // results under way per thread: a load from L2 takes as long as dozens of additions
    for (u64 t0 = threadIdx.x; t0 < f.ntasks; t0 += (u64)kAhead * blockDim.x) {
        typename A::Acc a[kAhead];
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            const u64 t = t0 + (u64)i * blockDim.x;
            a[i] = t < f.ntasks ? acc_load_l2<A>(f.task_out + t * (u64)A::ACC_WORDS) : A::acc_zero();
        }
#pragma unroll
        for (int i = 0; i < kAhead; ++i) acc = A::acc_add(acc, a[i]);
    }
    acc = block_sum<A>(acc, sh);
    if (threadIdx.x == 0) {   // (the end of the launch makes these visible to the host)
        f.host[1] = 0;
        f.host[6] = 0;
        A::acc_store(f.host + 2, A::acc_norm(acc));
        f.ws[0] = 0;
        f.ws[7] = 0;
    }
}

}  // namespace pk
