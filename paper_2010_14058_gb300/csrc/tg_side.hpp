// tg_side.hpp -- streams beside the caller's for one count call.
#pragma once

#include <cstddef>
#include <memory>
#include <mutex>
#include <utility>
#include <vector>
#include <cuda_runtime.h>

#include "tg_error.hpp"

namespace tg {

// Side streams of one count call: the wedge forms and the triangle kernels do
// not depend on each other and run beside each other, since on a small graph
// none of them fills the GPU and on a large one each ends in a tail.  A set
// is taken for the call and given back once the joins are enqueued (what a
// later call enqueues on it comes after).  Its streams have the priority of
// the caller's, so that the caller's choice governs the whole count.  The
// process keeps at most kKeep sets per device and priority, more exist only
// while that many calls run at once.
class SideStreams {
public:
    static constexpr int kSides = 3;
    explicit SideStreams(cudaStream_t main) : main_(main) {
        TG_CK(cudaGetDevice(&dev_));
        const cudaError_t e = cudaStreamGetPriority(main, &priority_);
        forget(e);
        if (e != cudaSuccess) priority_ = 0;
        {
            std::lock_guard<std::mutex> lock(mutex());
            auto &pool = free_sets();
            for (size_t k = 0; k < pool.size() && !set_; ++k)
                if (mine(*pool[k])) {
                    set_ = std::move(pool[k]);
                    pool.erase(pool.begin() + (std::ptrdiff_t)k);
                }
        }
        if (!set_) {
            set_ = std::make_unique<Set>();
            set_->dev = dev_;
            set_->priority = priority_;
            for (auto &x : set_->s) TG_CK(cudaStreamCreateWithPriority(&x, cudaStreamNonBlocking, priority_));
            for (auto &x : set_->ev) TG_CK(cudaEventCreateWithFlags(&x, cudaEventDisableTiming));
        }
    }
    ~SideStreams() {
        if (forked_) {                                      // an error between fork and join: nothing may still run
            for (cudaStream_t x : set_->s) forget(cudaStreamSynchronize(x));   // when the caller gives its buffers back
            return;
        }
        std::lock_guard<std::mutex> lock(mutex());
        size_t kept = 0;
        for (const auto &x : free_sets()) kept += mine(*x) ? 1 : 0;
        if (kept >= kKeep) return;
        try {
            free_sets().push_back(std::move(set_));
        } catch (...) {                                     // (no host memory: the set goes)
        }
    }
    cudaStream_t side(int k) const { return set_->s[k]; }
    // the sides start after what the main stream has so far
    void fork() {
        forked_ = true;
        TG_CK(cudaEventRecord(set_->ev[0], main_));
        for (cudaStream_t x : set_->s) TG_CK(cudaStreamWaitEvent(x, set_->ev[0], 0));
    }
    // side k goes on after what the main stream has so far
    void after_main(int k) {
        TG_CK(cudaEventRecord(set_->ev[1], main_));
        TG_CK(cudaStreamWaitEvent(set_->s[k], set_->ev[1], 0));
    }
    // the main stream goes on after the sides
    void join() {
        for (int k = 0; k < kSides; ++k) {
            TG_CK(cudaEventRecord(set_->ev[2 + k], set_->s[k]));
            TG_CK(cudaStreamWaitEvent(main_, set_->ev[2 + k], 0));
        }
        forked_ = false;
    }

private:
    struct Set {
        int dev = 0, priority = 0;
        cudaStream_t s[kSides] = {};
        cudaEvent_t ev[2 + kSides] = {};
        ~Set() {                                            // (work enqueued on them completes all the same)
            for (cudaStream_t x : s)
                if (x) forget(cudaStreamDestroy(x));
            for (cudaEvent_t x : ev)
                if (x) forget(cudaEventDestroy(x));
        }
    };
    static constexpr size_t kKeep = 8;
    static std::mutex &mutex() {
        static std::mutex *m = new std::mutex();
        return *m;
    }
    static std::vector<std::unique_ptr<Set>> &free_sets() {   // never destroyed: the CUDA context may go first
        static auto *v = new std::vector<std::unique_ptr<Set>>();
        return *v;
    }
    bool mine(const Set &x) const { return x.dev == dev_ && x.priority == priority_; }
    cudaStream_t main_;
    int dev_ = 0, priority_ = 0;
    bool forked_ = false;
    std::unique_ptr<Set> set_;
};

}  // namespace tg
