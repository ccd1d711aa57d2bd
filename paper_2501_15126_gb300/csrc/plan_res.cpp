// plan_res.cpp -- free lists of plan resources (plan_res.hpp).
#include "plan_res.hpp"

#include <map>
#include <mutex>

#include <cuda.h>

namespace perm {

namespace {

constexpr size_t kClassBytes[] = {64 * 1024, 512 * 1024};   // walks of up to 2^11 and 2^14 FP64 tasks
constexpr int kClasses = 2;
constexpr size_t kKeep = 16;

struct FreeList {
    size_t count = 0;
    PlanRes set[kKeep];
};

std::mutex g_mu;
std::map<std::pair<int, int>, FreeList> &lists() {
    // never destroyed: the CUDA runtime may be gone before static destructors run
    static auto *l = new std::map<std::pair<int, int>, FreeList>();
    return *l;
}

template <class F>
F driver_entry(const char *name) {
    void *f = nullptr;
    cudaDriverEntryPointQueryResult q;
    const cudaError_t e = cudaGetDriverEntryPointByVersion(name, &f, 12000, cudaEnableDefault, &q);
    return e == cudaSuccess && q == cudaDriverEntryPointSuccess ? reinterpret_cast<F>(f) : nullptr;
}

// The id of the allocation at p, 0 if there is none (a context is bound to the thread).
unsigned long long buffer_id(const void *p) {
    static const auto fn = driver_entry<CUresult (*)(void *, CUpointer_attribute, CUdeviceptr)>("cuPointerGetAttribute");
    unsigned long long id = 0;
    if (!fn || fn(&id, CU_POINTER_ATTRIBUTE_BUFFER_ID, reinterpret_cast<CUdeviceptr>(p)) != CUDA_SUCCESS) return 0;
    return id;
}

// The thread's context; the device's primary one is bound first where it has none.
cudaError_t current_context(void **out) {
    static const auto fn = driver_entry<CUresult (*)(CUcontext *)>("cuCtxGetCurrent");
    CUcontext c = nullptr;
    *out = nullptr;
    if (!fn || fn(&c) != CUDA_SUCCESS) return cudaSuccess;   // unknown: nothing is kept
    if (!c) {
        const cudaError_t e = cudaFree(nullptr);
        if (e != cudaSuccess) return e;
        fn(&c);
    }
    *out = c;
    return cudaSuccess;
}

void release(PlanRes &r) {
    if (r.dev) cudaFree(r.dev);
    if (r.host) cudaFreeHost(r.host);
    if (r.ev0) cudaEventDestroy(r.ev0);
    if (r.ev1) cudaEventDestroy(r.ev1);
    r = PlanRes();
}

}  // namespace

cudaError_t plan_res_take(size_t bytes, PlanRes *out) {
    PlanRes r;
    cudaError_t e = cudaGetDevice(&r.device);
    if (e != cudaSuccess) return e;
    for (int c = 0; c < kClasses && r.size_class < 0; ++c)
        if (bytes <= kClassBytes[c]) r.size_class = c;
    if (r.size_class >= 0) {
        if ((e = current_context(&r.context)) != cudaSuccess) return e;
        std::lock_guard<std::mutex> lk(g_mu);
        FreeList &l = lists()[{r.device, r.size_class}];
        for (size_t i = l.count; i-- > 0;) {
            const PlanRes s = l.set[i];
            const bool alive = buffer_id(s.dev) == s.buffer_id;
            if (alive && s.context != r.context) continue;   // another context's
            l.set[i] = l.set[--l.count];                     // taken, or gone with its context
            if (!alive) continue;
            *out = s;
            return cudaSuccess;
        }
    }
    e = cudaMalloc(&r.dev, r.size_class >= 0 ? kClassBytes[r.size_class] : bytes);
    if (e == cudaSuccess) e = cudaMallocHost(&r.host, 64 + kStageBytes);
    if (e == cudaSuccess) e = cudaEventCreate(&r.ev0);
    if (e == cudaSuccess) e = cudaEventCreate(&r.ev1);
    if (e != cudaSuccess) {
        release(r);
        return e;
    }
    r.buffer_id = buffer_id(r.dev);
    if (!r.buffer_id || !r.context) r.size_class = -1;   // cannot be told from a dead one: not kept
    *out = r;
    return cudaSuccess;
}

void plan_res_give(PlanRes &r) {
    if (!r.dev) return;
    if (r.size_class >= 0) {
        std::lock_guard<std::mutex> lk(g_mu);
        FreeList &l = lists()[{r.device, r.size_class}];
        if (l.count < kKeep) {
            l.set[l.count++] = r;
            r = PlanRes();
            return;
        }
    }
    release(r);
}

}  // namespace perm
