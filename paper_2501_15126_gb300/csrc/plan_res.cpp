// plan_res.cpp -- free lists of plan resources (plan_res.hpp).
#include "plan_res.hpp"

#include <map>
#include <mutex>
#include <vector>

namespace perm {

namespace {

constexpr size_t kClassBytes[] = {64 * 1024, 512 * 1024};   // walks of up to 2^11 and 2^14 FP64 tasks
constexpr int kClasses = 2;
constexpr size_t kKeep = 16;

std::mutex g_mu;
std::map<std::pair<int, int>, std::vector<PlanRes>> &lists() {
    // never destroyed: the CUDA runtime may be gone before static destructors run
    static auto *l = new std::map<std::pair<int, int>, std::vector<PlanRes>>();
    return *l;
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
        std::lock_guard<std::mutex> lk(g_mu);
        std::vector<PlanRes> &l = lists()[{r.device, r.size_class}];
        if (!l.empty()) {
            *out = l.back();
            l.pop_back();
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
    *out = r;
    return cudaSuccess;
}

void plan_res_give(PlanRes &r) {
    if (!r.dev) return;
    if (r.size_class >= 0) {
        std::lock_guard<std::mutex> lk(g_mu);
        std::vector<PlanRes> &l = lists()[{r.device, r.size_class}];
        if (l.size() < kKeep) {
            l.push_back(r);
            r = PlanRes();
            return;
        }
    }
    release(r);
}

}  // namespace perm
