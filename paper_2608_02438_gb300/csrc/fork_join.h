// fork_join.h -- a side stream that takes part of a call's work beside the
// caller's stream, and is always joined into it again.
#ifndef XPRESS_FORK_JOIN_H
#define XPRESS_FORK_JOIN_H

#include <cuda_runtime_api.h>

namespace xp {

// The caller may free or reuse its buffers once its own stream has reached the
// call's end, also when the call returned an error halfway: whatever was put on
// the side stream is joined when the object goes out of scope, by events (so that
// a capture sees it too), or by waiting for the stream if even that fails.
class StreamFork {
public:
    StreamFork(cudaStream_t main, cudaStream_t side, cudaEvent_t join_event)
        : main_(main), side_(side), join_event_(join_event)
    {
    }
    StreamFork(const StreamFork &) = delete;
    StreamFork &operator=(const StreamFork &) = delete;
    ~StreamFork()
    {
        if (open_ && join() != cudaSuccess) (void)cudaStreamSynchronize(side_);
    }
    // The side stream goes on from here: what follows on it sees the main stream's work so far.
    cudaError_t fork(cudaEvent_t event)
    {
        cudaError_t e = cudaEventRecord(event, main_);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(side_, event, 0);
        open_ = open_ || e == cudaSuccess;
        return e;
    }
    cudaError_t join()
    {
        cudaError_t e = cudaEventRecord(join_event_, side_);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(main_, join_event_, 0);
        open_ = e != cudaSuccess;
        return e;
    }
    cudaStream_t stream() const { return side_; }

private:
    cudaStream_t main_, side_;
    cudaEvent_t join_event_;
    bool open_ = false;
};

}  // namespace xp

#endif
