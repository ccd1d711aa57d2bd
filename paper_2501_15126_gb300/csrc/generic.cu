// generic.cu -- dispatch to the precompiled generic kernels, and the final
// reduction kernels.
#include <algorithm>

#include <cuda_runtime.h>

#include "finish.cuh"
#include "kernels.hpp"
#include "vm.hpp"

namespace pk {

// ------------------------------------------------------------------ final reduction
// Task results summed in a fixed order (deterministic): block b takes tasks
// [b per, (b + 1) per), and the last block to finish adds the blocks' sums in
// block order.  A block's sum takes the place of its first task's result.
// (FP64 runs at 2 lanes per clock and SM, so one block of 1024 threads spent
// 25-38 us in its shuffle trees; blocks of 128 threads over the whole GPU
// spend a few.)
template <class A>
__device__ __forceinline__ void reduce_tasks(u64 *task_out, u64 ntasks, u64 per, u64 *result, u64 *done_blocks) {
    __shared__ u64 sh[32 * 6];
    typename A::Acc acc = A::acc_zero();
    const u64 b = blockIdx.x * per, e = b + per < ntasks ? b + per : ntasks;
    for (u64 t = b + threadIdx.x; t < e; t += blockDim.x)
        acc = A::acc_add(acc, A::acc_load(task_out + t * (u64)A::ACC_WORDS));
    acc = block_sum<A>(acc, sh);
    if (gridDim.x == 1) {
        if (threadIdx.x == 0) A::acc_store(result, A::acc_norm(acc));
        return;
    }
    if (threadIdx.x == 0) A::acc_store(task_out + b * (u64)A::ACC_WORDS, acc);
    if (!last_block(done_blocks)) return;
    acc = A::acc_zero();
    for (u64 k = threadIdx.x; k < gridDim.x; k += blockDim.x)
        acc = A::acc_add(acc, acc_load_l2<A>(task_out + k * per * (u64)A::ACC_WORDS));
    acc = block_sum<A>(acc, sh);
    if (threadIdx.x == 0) A::acc_store(result, A::acc_norm(acc));
}

template <class A>
__global__ void __launch_bounds__(128) k_reduce(u64 *task_out, u64 ntasks, u64 per, u64 *result, u64 *done_blocks) {
    reduce_tasks<A>(task_out, ntasks, per, result, done_blocks);
}

// One warp per matrix, lane-strided then a fixed shuffle tree: deterministic.
template <class A>
__global__ void __launch_bounds__(256) k_batch_reduce(const BatchMat *mats, int nmat, u64 ntasks,
                                                      const u64 *task_out, u64 *result) {
    const int m = (int)((blockIdx.x * (u64)blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (m >= nmat) return;
    const u64 b = mats[m].task_begin;
    const u64 e = (m + 1 < nmat) ? mats[m + 1].task_begin : ntasks;
    typename A::Acc acc = A::acc_zero();
    for (u64 t = b + lane; t < e; t += 32) acc = A::acc_add(acc, A::acc_load(task_out + t * (u64)A::ACC_WORDS));
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) acc = A::acc_add(acc, A::shfl_down(acc, d));
    if (lane == 0) A::acc_store(result + (u64)m * A::ACC_WORDS, A::acc_norm(acc));
}

// Serving: segment m sums pool[seg[2m] .. seg[2m] + seg[2m+1]) (task units),
// one warp per segment, fixed order.
template <class A>
__global__ void __launch_bounds__(256) k_segment_reduce(const u64 *seg, int nseg, const u64 *pool, u64 *result) {
    const int m = (int)((blockIdx.x * (u64)blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (m >= nseg) return;
    const u64 b = seg[2 * m], e = b + seg[2 * m + 1];
    typename A::Acc acc = A::acc_zero();
    for (u64 t = b + lane; t < e; t += 32) acc = A::acc_add(acc, A::acc_load(pool + t * (u64)A::ACC_WORDS));
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) acc = A::acc_add(acc, A::shfl_down(acc, d));
    if (lane == 0) A::acc_store(result + (u64)m * 4, A::acc_norm(acc));
}

}  // namespace pk

namespace perm {

cudaError_t segment_reduce_launch(int arith, const uint64_t *seg, int nseg, const uint64_t *pool, uint64_t *result,
                                  cudaStream_t st) {
    const unsigned long long *sg = reinterpret_cast<const unsigned long long *>(seg);
    const unsigned long long *in = reinterpret_cast<const unsigned long long *>(pool);
    unsigned long long *out = reinterpret_cast<unsigned long long *>(result);
    const int grid = (nseg * 32 + 255) / 256;
    if (nseg <= 0) return cudaSuccess;
    switch (arith) {
    case 0: pk::k_segment_reduce<pk::ArithF64><<<grid, 256, 0, st>>>(sg, nseg, in, out); break;
    case 1: pk::k_segment_reduce<pk::ArithExact<2>><<<grid, 256, 0, st>>>(sg, nseg, in, out); break;
    case 2: pk::k_segment_reduce<pk::ArithExact<4>><<<grid, 256, 0, st>>>(sg, nseg, in, out); break;
    case 3: pk::k_segment_reduce<pk::ArithExact<6>><<<grid, 256, 0, st>>>(sg, nseg, in, out); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t batch_reduce_launch(int arith, const pk::BatchMat *mats, int nmat, uint64_t ntasks,
                                const uint64_t *task_out, uint64_t *result, cudaStream_t st) {
    const unsigned long long *in = reinterpret_cast<const unsigned long long *>(task_out);
    unsigned long long *out = reinterpret_cast<unsigned long long *>(result);
    const int grid = (nmat * 32 + 255) / 256;
    if (nmat <= 0) return cudaSuccess;
    switch (arith) {
    case 0: pk::k_batch_reduce<pk::ArithF64><<<grid, 256, 0, st>>>(mats, nmat, ntasks, in, out); break;
    case 1: pk::k_batch_reduce<pk::ArithExact<2>><<<grid, 256, 0, st>>>(mats, nmat, ntasks, in, out); break;
    case 2: pk::k_batch_reduce<pk::ArithExact<4>><<<grid, 256, 0, st>>>(mats, nmat, ntasks, in, out); break;
    case 3: pk::k_batch_reduce<pk::ArithExact<6>><<<grid, 256, 0, st>>>(mats, nmat, ntasks, in, out); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

GenericFns generic_fns_f64(int nmax);
GenericFns generic_fns_dd(int nmax);
GenericFns generic_fns_r64(int nmax, int fold);
GenericFns generic_fns_r96(int nmax, int fold);
GenericFns generic_fns_r128(int nmax, int fold);
GenericFns generic_fns_r160(int nmax, int fold);
GenericFns generic_fns_r192(int nmax, int fold);

GenericFns generic_fns(int nmax, int kind) {
    if (nmax < 16) return vm_fns(kind);   // shared-memory classes of the eliminated walk
    const int limbs = kind >> 1, fold = kind & 1;
    switch (limbs) {
    case 0: return fold ? generic_fns_dd(nmax) : generic_fns_f64(nmax);
    case 2: return generic_fns_r64(nmax, fold);
    case 3: return generic_fns_r96(nmax, fold);
    case 4: return generic_fns_r128(nmax, fold);
    case 5: return generic_fns_r160(nmax, fold);
    case 6: return generic_fns_r192(nmax, fold);
    default: return GenericFns();
    }
}

cudaError_t reduce_launch(int arith, uint64_t *task_out, uint64_t ntasks, uint64_t *result, uint64_t *done_blocks,
                          cudaStream_t st) {
    unsigned long long *in = reinterpret_cast<unsigned long long *>(task_out);
    unsigned long long *out = reinterpret_cast<unsigned long long *>(result);
    unsigned long long *dn = reinterpret_cast<unsigned long long *>(done_blocks);
    // 512 tasks a block (four additions a thread) until the GPU is full
    const unsigned long long per = std::max<unsigned long long>(512, (ntasks + 151) / 152);
    const unsigned grid = (unsigned)std::max<unsigned long long>(1, (ntasks + per - 1) / per);
    switch (arith) {
    case 0: pk::k_reduce<pk::ArithF64><<<grid, 128, 0, st>>>(in, ntasks, per, out, dn); break;
    case 1: pk::k_reduce<pk::ArithExact<2>><<<grid, 128, 0, st>>>(in, ntasks, per, out, dn); break;
    case 2: pk::k_reduce<pk::ArithExact<4>><<<grid, 128, 0, st>>>(in, ntasks, per, out, dn); break;
    case 3: pk::k_reduce<pk::ArithExact<6>><<<grid, 128, 0, st>>>(in, ntasks, per, out, dn); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace perm
