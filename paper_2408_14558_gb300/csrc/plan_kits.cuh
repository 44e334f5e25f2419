// Page-locked words and events of plans, kept from one plan for the next
// (host code only).
#pragma once

#include <cuda_runtime_api.h>

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <mutex>
#include <vector>

namespace spg {

// The id of the calling thread's CUDA context (0 if there is none to be had).
// No two contexts of a process share one, so what was made in a context that a
// cudaDeviceReset has ended is told from what belongs to the next (0.5 us).
inline unsigned long long context_id() {
    using GetId = int (*)(void *, unsigned long long *);  // cuCtxGetId
    static const GetId get = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &found) != cudaSuccess ||
            found != cudaDriverEntryPointSuccess)
            f = nullptr;
        return (GetId)f;
    }();
    unsigned long long id = 0;
    if (!get) return 0;
    if (get(nullptr, &id) == 0) return id;
    cudaFree(nullptr);  // no context yet, or none since the reset: makes one
    if (get(nullptr, &id) == 0) return id;
    cudaGetLastError();
    return 0;
}

// What one plan holds: `words` page-locked words and 18 events of one context.
struct PlanKit {
    unsigned long long ctx = 0;
    int64_t *pinned = nullptr;
    size_t words = 0;
    cudaEvent_t ev[8] = {}, kev[10] = {};
};

// Making and destroying a kit takes about 80 us, a fifth of a small multiply.  A
// kit is handed out to one plan at a time, under a lock, and comes back once that
// plan's stream is known to be idle; at most kMost wait (about 9 KB each), for the
// life of the process, the others are destroyed.  Only kits of the usual number
// of words are kept.
class PlanKits {
  public:
    static constexpr size_t kMost = 16;
    explicit PlanKits(size_t usual_words) : usual_(usual_words) {}

    // A kit of at least `words` words for context `ctx`, a kept one or a new one.
    cudaError_t take(unsigned long long ctx, size_t words, PlanKit *out) {
        {
            std::lock_guard<std::mutex> hold(lock_);
            for (size_t i = 0; i < kept_.size(); i++)
                if (ctx != 0 && kept_[i].ctx == ctx && kept_[i].words >= words) {
                    *out = kept_[i];
                    kept_[i] = kept_.back();
                    kept_.pop_back();
                    return cudaSuccess;
                }
        }
        PlanKit k;
        k.ctx = ctx;
        k.words = std::max(words, usual_);
        cudaError_t e = cudaMallocHost((void **)&k.pinned, sizeof(int64_t) * k.words);
        for (auto &x : k.ev)
            if (e == cudaSuccess) e = cudaEventCreate(&x);
        for (auto &x : k.kev)
            if (e == cudaSuccess) e = cudaEventCreate(&x);
        if (e != cudaSuccess) {
            destroy(k);
            return e;
        }
        *out = k;
        return cudaSuccess;
    }

    // Back from a plan.  idle: everything queued with the kit has ended (else a
    // copy may still land in its words); ctx: the calling thread's context now.
    void give(const PlanKit &k, bool idle, unsigned long long ctx) {
        if (!k.pinned) return;
        if (ctx != k.ctx && !alive(k)) return;  // gone with its context
        if (idle && ctx != 0 && ctx == k.ctx && k.words == usual_) {
            std::lock_guard<std::mutex> hold(lock_);
            if (kept_.size() >= kMost)  // room taken by kits that a reset has ended
                kept_.erase(std::remove_if(kept_.begin(), kept_.end(),
                                           [&](const PlanKit &o) { return o.ctx != ctx && !alive(o); }),
                            kept_.end());
            if (kept_.size() < kMost) {
                kept_.push_back(k);
                return;
            }
        }
        destroy(k);
    }

  private:
    // its page-locked words are still known to CUDA
    static bool alive(const PlanKit &k) {
        cudaPointerAttributes a{};
        const bool known = cudaPointerGetAttributes(&a, k.pinned) == cudaSuccess && a.type == cudaMemoryTypeHost;
        cudaGetLastError();
        return known;
    }
    static void destroy(const PlanKit &k) {
        for (cudaEvent_t e : k.ev)
            if (e) cudaEventDestroy(e);
        for (cudaEvent_t e : k.kev)
            if (e) cudaEventDestroy(e);
        if (k.pinned) cudaFreeHost(k.pinned);
    }
    const size_t usual_;
    std::mutex lock_;
    std::vector<PlanKit> kept_;
};

}  // namespace spg
