// plan_store.h -- the device copies of a mesh's patch plans, shared by the
// states of the mesh.
//
// A copy is made by the first state that needs it, shared by those that
// follow, and kept when the last one goes, so that a state made later on the
// mesh finds it (on the level-7 sphere a copy costs 42 ms to make, mixed, and
// a state 8 without).  The idle copies are given back by trim(), which the
// autotuner calls behind its rejected candidates, the request runtime where
// they stand in the way of its budget and state creation where memory has run
// out, and with the store.  Nothing here synchronises the device: a copy is
// complete before any second state can see it, and is freed in stream order
// behind the work of every state that held it.
#pragma once

#include <cstddef>

#include <algorithm>
#include <array>
#include <map>
#include <memory>
#include <mutex>
#include <vector>

#include <cuda_runtime.h>

namespace sse {

// The arrays of one copy, uploaded in stream order; in counting mode only
// their sizes are summed.  Whatever is not handed over is freed.
class PlanUpload {
public:
    PlanUpload(cudaStream_t st, bool count_only) : stream_(st), count_(count_only) {}
    PlanUpload(const PlanUpload &) = delete;
    PlanUpload &operator=(const PlanUpload &) = delete;
    ~PlanUpload() {
        for (void *p : ptrs_) cudaFreeAsync(p, stream_);
    }
    template <class T> T *put(const std::vector<T> &v) {
        const size_t nb = std::max<size_t>(v.size(), 1) * sizeof(T);
        bytes += (nb + 255) / 256 * 256;
        if (count_ || failed) return nullptr;
        ptrs_.reserve(ptrs_.size() + 1);
        void *p = nullptr;
        if (cudaMallocAsync(&p, nb, stream_) != cudaSuccess) {
            failed = true;
            cudaGetLastError();
            return nullptr;
        }
        ptrs_.push_back(p);
        if (!v.empty() && cudaMemcpyAsync(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice,
                                          stream_) != cudaSuccess) {
            failed = true;
            cudaGetLastError();
        }
        return (T *)p;
    }
    std::vector<void *> hand_over() {
        std::vector<void *> out;
        out.swap(ptrs_);
        return out;
    }
    bool failed = false;
    size_t bytes = 0;

private:
    cudaStream_t stream_;
    bool count_;
    std::vector<void *> ptrs_;
};

class PlanStore {
public:
    using Key = std::array<int, 4>;   // kind, bytes of a real, and the plan's own two
    explicit PlanStore(int device) : device_(device) {}
    PlanStore(const PlanStore &) = delete;
    PlanStore &operator=(const PlanStore &) = delete;

    // The copy `key` for a state on `st`: the one there is, or one that
    // fill(PlanUpload &, View &) makes; nothing is kept of one that failed.
    // Every acquire that succeeds has its release.
    template <class View, class Fill>
    cudaError_t acquire(const Key &key, cudaStream_t st, View &out, Fill &&fill) {
        std::lock_guard<std::mutex> lk(mu_);
        auto it = live_.find(key);
        if (it == live_.end()) {
            PlanUpload up(st, false);
            auto view = std::make_shared<View>();
            fill(up, *view);
            if (up.failed) return cudaErrorMemoryAllocation;
            // complete before another stream may read it
            const cudaError_t e = cudaStreamSynchronize(st);
            if (e != cudaSuccess) return e;
            sizes_[key] = up.bytes;
            it = live_.emplace(key, Copy{}).first;
            it->second.view = view;
            it->second.bytes = up.bytes;
            it->second.ptrs = up.hand_over();
            resident_ += up.bytes;
        }
        it->second.holders++;
        out = *static_cast<const View *>(it->second.view.get());
        return cudaSuccess;
    }

    // Bytes of the copy `key`, made or not.
    template <class View, class Fill> size_t size(const Key &key, Fill &&fill) {
        std::lock_guard<std::mutex> lk(mu_);
        auto it = sizes_.find(key);
        if (it != sizes_.end()) return it->second;
        PlanUpload up(nullptr, true);
        View view{};
        fill(up, view);
        return sizes_[key] = up.bytes;
    }

    // A state whose work is all queued on `st` gives its hold back.
    void release(const Key &key, cudaStream_t st) {
        std::lock_guard<std::mutex> lk(mu_);
        auto it = live_.find(key);
        if (it == live_.end()) return;
        it->second.holders--;
        leave(it->second, st);
    }

    // Free the copies that no state holds, but for those in `keep`.  Returns
    // their bytes.
    size_t trim(const std::vector<Key> &keep = {}) {
        std::lock_guard<std::mutex> lk(mu_);
        OnDevice dev(device_);
        size_t freed = 0;
        for (auto it = live_.begin(); it != live_.end();) {
            Copy &c = it->second;
            if (c.holders > 0 || std::find(keep.begin(), keep.end(), it->first) != keep.end()) {
                ++it;
                continue;
            }
            for (cudaEvent_t e : c.left) {
                cudaStreamWaitEvent(cudaStreamPerThread, e, 0);
                cudaEventDestroy(e);
            }
            for (void *p : c.ptrs) cudaFreeAsync(p, cudaStreamPerThread);
            freed += c.bytes;
            it = live_.erase(it);
        }
        resident_ -= freed;
        return freed;
    }
    ~PlanStore() { trim(); }

    std::vector<Key> keys() {
        std::lock_guard<std::mutex> lk(mu_);
        std::vector<Key> out;
        for (const auto &kv : live_) out.push_back(kv.first);
        return out;
    }
    // bytes of all copies, and of those that no state holds
    size_t resident() {
        std::lock_guard<std::mutex> lk(mu_);
        return resident_;
    }
    size_t idle() {
        std::lock_guard<std::mutex> lk(mu_);
        size_t n = 0;
        for (const auto &kv : live_) n += kv.second.holders > 0 ? 0 : kv.second.bytes;
        return n;
    }

private:
    // events and the per-thread stream belong to the current device
    struct OnDevice {
        int was = -1;
        explicit OnDevice(int dev) {
            if (cudaGetDevice(&was) != cudaSuccess || was == dev ||
                cudaSetDevice(dev) != cudaSuccess)
                was = -1;
        }
        ~OnDevice() {
            if (was >= 0) cudaSetDevice(was);
        }
    };
    struct Copy {
        std::shared_ptr<const void> view;
        std::vector<void *> ptrs;
        size_t bytes = 0;
        int holders = 0;
        std::vector<cudaEvent_t> left;   // behind the work of the holders that left
    };
    // Remember where the leaving state's stream stands; those that have been
    // passed are dropped.  Where no event is to be had, wait.
    void leave(Copy &c, cudaStream_t st) {
        size_t n = 0;
        for (cudaEvent_t e : c.left) {
            if (cudaEventQuery(e) == cudaErrorNotReady) c.left[n++] = e;
            else cudaEventDestroy(e);
        }
        c.left.resize(n);
        OnDevice dev(device_);
        cudaEvent_t e = nullptr;
        bool kept = false;
        if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess) {
            kept = cudaEventRecord(e, st) == cudaSuccess;
            if (kept) {
                try {
                    c.left.push_back(e);
                } catch (...) {
                    kept = false;
                }
            }
            if (!kept) cudaEventDestroy(e);
        }
        if (!kept) {
            cudaGetLastError();
            cudaStreamSynchronize(st);
        }
    }

    const int device_;
    std::mutex mu_;
    std::map<Key, Copy> live_;
    std::map<Key, size_t> sizes_;
    size_t resident_ = 0;
};

}  // namespace sse
