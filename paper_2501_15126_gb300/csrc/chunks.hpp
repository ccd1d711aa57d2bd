// chunks.hpp -- chunk lengths (log2 of Gray indices) of the matrices of a batch.
// A task is 32 chunks and leaves up to 24 bytes of result, so the chunk length of
// a long walk bounds the memory of a call.
#pragma once

#include <algorithm>

namespace perm {

// Chained walks of families that are not autotuned (tune.cpp): 2^9 steps spread
// small matrices over the SMs (2^12 against 2^9 steps, p = 0.35: one n=22 FP64
// matrix 3.84 and 0.77 ms, 60 of them 10.6 and 8.7 ms).  From n = 28 on chunks grow
// with the walk, which keeps the 2^12 tasks that fill the GPU (eight n=28 FP64:
// 27.5 ms at 2^9, 27.1 at 2^10), up to the 2^12 steps of every longer walk.
inline int batch_default_chunk_log2(int n) { return std::min(12, std::max(9, n - 18)); }

// Eliminated walks that share a launch, h outer columns: 2^3 outer steps a lane, and
// full warps first; beyond 2^max_tasks_log2 tasks the chunks grow.
inline int shared_chunk_log2(int h, int max_tasks_log2) {
    return std::max(std::max(0, std::min(3, h - 5)), h - 5 - max_tasks_log2);
}
// A matrix of a batch: up to 1.5 MB of results, dozens of tasks for every warp that
// the GPU holds (one n=36 p=0.2 FP64: 45.5 ms with 2^17 tasks, 44.2 with 2^16).
constexpr int kBatchTasksLog2 = 16;

}  // namespace perm
