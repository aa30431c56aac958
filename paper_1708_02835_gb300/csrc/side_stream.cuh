// A stream beside the one a call was given.  Whatever way the call ends, the given stream waits for
// the work on this one before anything that follows there (the workspace's release, a caller's
// next use of its buffers): an early return leaves kernels in flight on it.
#pragma once
#include <cuda_runtime.h>

namespace egs {

struct SideStream {
    cudaStream_t st = nullptr;
    cudaStream_t owner = nullptr;  // the stream that waits
    cudaEvent_t done = nullptr;
    bool open = false;  // has work that owner does not wait for yet

    cudaError_t create(cudaStream_t owner_stream, bool high_priority)
    {
        owner = owner_stream;
        int least = 0, greatest = 0;
        cudaError_t e = cudaDeviceGetStreamPriorityRange(&least, &greatest);
        if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&st, cudaStreamNonBlocking, high_priority ? greatest : least);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&done, cudaEventDisableTiming);
        return e;
    }

    // owner waits for everything enqueued so far; if that cannot be arranged, the host does.
    cudaError_t join()
    {
        if (!open) return cudaSuccess;
        open = false;
        cudaError_t e = cudaEventRecord(done, st);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(owner, done, 0);
        if (e != cudaSuccess) cudaStreamSynchronize(st);
        return e;
    }

    SideStream() = default;
    SideStream(const SideStream &) = delete;
    SideStream &operator=(const SideStream &) = delete;
    // a stream or event with work pending is released once that work completes
    ~SideStream()
    {
        join();
        if (st) cudaStreamDestroy(st);
        if (done) cudaEventDestroy(done);
    }
};

}  // namespace egs
