// plan_res.hpp -- the CUDA resources of a plan, kept between plans.
//
// A plan needs one device buffer (its image, workspace words and task results),
// a few pinned words, pinned staging for the image and two timing events.
// Creating and freeing them takes some 450 us, forty times a small walk.  A
// released set goes to a free list of its device and size class and the next
// plan takes it from there; each list keeps at most kKeep sets (about 10 MB of
// device memory per device in all), and what does not fit is freed.  A plan holds
// its set alone from create to destroy, and every compute, a failed one too, ends
// with its stream synchronised, so a released set has no work in flight; a set
// whose stream could not be waited for is freed instead (size_class = -1).  The
// sets of a context that cudaDeviceReset ended are gone with it: a listed set is
// handed out only in the context it was made in, while the driver still knows its
// buffer by the id it had.
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

namespace perm {

struct PlanRes {
    int device = -1;
    int size_class = -1;             // -1: a device buffer of its own size, never kept
    unsigned char *dev = nullptr;
    uint64_t *host = nullptr;        // 8 pinned words, then the staging area
    unsigned char *stage() const { return reinterpret_cast<unsigned char *>(host + 8); }
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    void *context = nullptr;            // the CUDA context it was made in
    unsigned long long buffer_id = 0;   // the driver's, unique in the process: dev's allocation
};

constexpr size_t kStageBytes = 32 * 1024;

// A set with at least `bytes` of device memory on the current device.
cudaError_t plan_res_take(size_t bytes, PlanRes *out);
void plan_res_give(PlanRes &r);

}  // namespace perm
