// Pinned memory that fields are read back through, two halves of kHalf bytes
// per device, made on first use and kept: a copy into it runs at the link's
// rate and beside the conversion of the half before, and neither pages of a
// fresh buffer nor the driver's own staging cost anything.  One read uses it at
// a time, from the copy it queues behind its domain's steps to the last value;
// a read that finds it taken goes through a buffer of its own and waits for
// nothing but its own domain.  lbm_release_cached_memory gives it back.
//
// A stage belongs to the device of the stream that is read through (an event
// can be recorded only on a stream of its own device), whatever device is
// current at the call.
#pragma once

#include <cstddef>
#include <map>
#include <mutex>
#include <vector>

#include <cuda_runtime_api.h>

namespace lbmgpu {

struct ReadStage {
    static constexpr size_t kHalf = (size_t)4 << 20;
    std::mutex use;                    // held by the read that uses the rest
    char* half[2] = {nullptr, nullptr};
    cudaEvent_t landed[2] = {nullptr, nullptr};

    // The stage of the stream's device (the current device for the default stream).
    static ReadStage& of(cudaStream_t stream) {
        int dev = 0;
        if (cudaStreamGetDevice(stream, &dev) != cudaSuccess) {
            cudaGetLastError();
            cudaGetDevice(&dev);
        }
        std::lock_guard<std::mutex> lk(table_mutex());
        ReadStage*& s = table()[dev];
        if (!s) s = new ReadStage(dev);
        return *s;
    }

    // Memory and events exist, or are made now; false where they cannot be.
    bool ready() {
        if (half[0]) return true;
        int cur = device;
        cudaGetDevice(&cur);
        if (cur != device) cudaSetDevice(device);
        void* p = nullptr;
        bool ok = cudaHostAlloc(&p, 2 * kHalf, cudaHostAllocPortable) == cudaSuccess;
        for (auto& e : landed) ok = ok && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess;
        if (cur != device) cudaSetDevice(cur);
        if (!ok) {
            cudaGetLastError();
            release_events();
            if (p) cudaFreeHost(p);
            return false;
        }
        half[0] = (char*)p;
        half[1] = half[0] + kHalf;
        return true;
    }

    // Gives the memory of every stage back.  A stage in use is waited for, with no
    // lock held that a read elsewhere takes.
    static void release_all() {
        std::vector<ReadStage*> stages;
        {
            std::lock_guard<std::mutex> lk(table_mutex());
            for (auto& kv : table()) stages.push_back(kv.second);
        }
        for (ReadStage* s : stages) {
            std::lock_guard<std::mutex> lk(s->use);
            if (!s->half[0]) continue;
            s->release_events();
            cudaFreeHost(s->half[0]);
            s->half[0] = s->half[1] = nullptr;
        }
    }

private:
    explicit ReadStage(int dev) : device(dev) {}
    void release_events() {
        for (auto& e : landed) {
            if (e) cudaEventDestroy(e);
            e = nullptr;
        }
    }
    // stages live as long as the process: a read may still run when statics go
    static std::mutex& table_mutex() {
        static std::mutex* m = new std::mutex();
        return *m;
    }
    static std::map<int, ReadStage*>& table() {
        static auto* t = new std::map<int, ReadStage*>();
        return *t;
    }
    const int device;
};

}  // namespace lbmgpu
