// side_streams.h -- work of several groups on streams of their own, forked from one
// stream and joined back into it (host code).
#pragma once
#include <vector>

#include <cuda_runtime.h>

#include "qsg.h"

namespace qsg {

class SideStreams {
public:
    SideStreams() = default;
    SideStreams(const SideStreams &) = delete;
    SideStreams &operator=(const SideStreams &) = delete;
    ~SideStreams() {
        for (cudaStream_t t : side_) cudaStreamDestroy(t);
        for (cudaEvent_t e : joins_) cudaEventDestroy(e);
        if (fork_) cudaEventDestroy(fork_);
    }

    // Run work(i, stream) for i = 0 .. n - 1: those with side(i) each on a stream of
    // its own, forked from st, the others one after another on st; st continues after
    // all of them.  On an error no further work is started, but st is still ordered
    // after everything that was: what the caller queues or frees next must not meet
    // it.  fail(e) turns a CUDA error into a status; the first error is returned.
    template <class Side, class Work, class Fail>
    qsg_status run(size_t n, cudaStream_t st, Side side, Work work, Fail fail) {
        if (cudaError_t e = grow(n)) return fail(e);
        if (cudaError_t e = cudaEventRecord(fork_, st)) return fail(e);
        qsg_status status = QSG_OK;
        size_t forked = 0;  // groups below it with side(i) are forked
        for (; forked < n && status == QSG_OK; ++forked) {
            if (!side(forked)) continue;
            if (cudaError_t e = cudaStreamWaitEvent(side_[forked], fork_, 0)) {
                status = fail(e);
                break;
            }
            status = work(forked, side_[forked]);
        }
        for (size_t i = 0; i < n && status == QSG_OK; ++i)
            if (!side(i)) status = work(i, st);
        for (size_t i = 0; i < forked; ++i) {
            if (!side(i)) continue;
            cudaError_t e = cudaEventRecord(joins_[i], side_[i]);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(st, joins_[i], 0);
            if (e == cudaSuccess) continue;
            cudaStreamSynchronize(side_[i]);  // the host waits where the streams cannot
            if (status == QSG_OK) status = fail(e);
        }
        return status;
    }

private:
    cudaError_t grow(size_t n) {
        if (!fork_)
            if (cudaError_t e = cudaEventCreateWithFlags(&fork_, cudaEventDisableTiming)) return e;
        while (side_.size() < n) {
            cudaStream_t t = nullptr;
            if (cudaError_t e = cudaStreamCreateWithFlags(&t, cudaStreamNonBlocking)) return e;
            side_.push_back(t);
        }
        while (joins_.size() < n) {
            cudaEvent_t j = nullptr;
            if (cudaError_t e = cudaEventCreateWithFlags(&j, cudaEventDisableTiming)) return e;
            joins_.push_back(j);
        }
        return cudaSuccess;
    }

    // one stream per group, with the fork and join events
    std::vector<cudaStream_t> side_;
    std::vector<cudaEvent_t> joins_;
    cudaEvent_t fork_ = nullptr;
};

}  // namespace qsg
