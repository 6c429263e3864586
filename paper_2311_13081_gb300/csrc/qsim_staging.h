// qsim_staging.h -- pinned host staging for uploads that must not wait for earlier work of the
// stream.
#pragma once
#include <cuda_runtime_api.h>

#include <cstddef>

namespace qsim {

// The calling thread's pinned staging on one device for the batched launch's descriptors.  From
// pageable memory the upload waited for everything before it on the stream (the previous
// launch), so consecutive calls left the GPU idle for the whole of their host work.  Two
// slots in turn: a call waits only if the copy of the call before the last has not run yet.
// At most two buffers of the largest call's descriptors (~1 KB a run) a device, freed when
// the thread ends.
struct Staging {
    void* p[2] = {nullptr, nullptr};
    size_t cap[2] = {0, 0};
    cudaEvent_t ev[2] = {nullptr, nullptr};
    int turn = 0;
    ~Staging() {
        for (int i = 0; i < 2; ++i) {
            if (ev[i]) {
                cudaEventSynchronize(ev[i]);
                cudaEventDestroy(ev[i]);
            }
            if (p[i]) cudaFreeHost(p[i]);
        }
        cudaGetLastError();
    }
    // Space for `bytes`, or null (the caller then copies from pageable memory).
    void* take(size_t bytes) {
        const int i = turn;
        bool ok = ev[i] || cudaEventCreateWithFlags(&ev[i], cudaEventDisableTiming) == cudaSuccess;
        ok = ok && cudaEventSynchronize(ev[i]) == cudaSuccess;
        if (ok && cap[i] < bytes) {
            if (p[i]) cudaFreeHost(p[i]);
            p[i] = nullptr;
            cap[i] = 0;
            ok = cudaHostAlloc(&p[i], bytes, cudaHostAllocDefault) == cudaSuccess;
            if (ok) cap[i] = bytes;
            else p[i] = nullptr;
        }
        if (!ok) {
            cudaGetLastError();
            return nullptr;
        }
        return p[i];
    }
    // The space taken last is read by the work submitted to st so far.
    void used(cudaStream_t st) {
        if (cudaEventRecord(ev[turn], st) != cudaSuccess) {
            cudaGetLastError();
            if (cudaStreamSynchronize(st) != cudaSuccess) {
                // nothing says when the copy has run: the buffer is given up, never written again
                cudaGetLastError();
                p[turn] = nullptr;
                cap[turn] = 0;
            }
        }
        turn ^= 1;
    }
};

// The staging of the current device (events and waits belong to one), or null.
inline Staging* staging_slot() {
    constexpr int kMaxDev = 16;
    static thread_local Staging slots[kMaxDev];
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) {
        cudaGetLastError();
        return nullptr;
    }
    return &slots[dev];
}

}  // namespace qsim
