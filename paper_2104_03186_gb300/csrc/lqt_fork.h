// Auxiliary streams for the independent parts of one call (the state sizes of a
// batch or of a set of warm solves).
//
// A host thread keeps kForkSets sets per device and hands them out in turn, so
// that the calls it has in flight on several streams of its own do not queue on
// one another's auxiliary streams (with more calls in flight than sets, a set's
// later call waits for its earlier one; the results do not depend on it).  The
// sets are made on the thread's first forked call on a device and kept until
// the process exits (a thread_local destructor can run after the CUDA runtime
// has shut down).
#pragma once

#include <cuda_runtime.h>

namespace lqt {

constexpr int kForkStreams = 3, kForkSets = 4;

struct ForkSet {
    cudaStream_t s[kForkStreams] = {};
    cudaEvent_t fork = nullptr, join[kForkStreams] = {};
};

// The next set of this thread on the current device; nullptr if the streams
// cannot be created (the call then runs on one stream).
inline ForkSet* next_fork_set() {
    struct Sets {
        ForkSet set[kForkSets];
        int next = 0;
        bool ready = false;
    };
    thread_local Sets all[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    Sets& a = all[dev];
    if (!a.ready) {
        // handles made by an earlier, failed attempt are kept and not made again
        for (ForkSet& f : a.set) {
            if (!f.fork && cudaEventCreateWithFlags(&f.fork, cudaEventDisableTiming) != cudaSuccess)
                return nullptr;
            for (int i = 0; i < kForkStreams; ++i)
                if ((!f.s[i] && cudaStreamCreateWithFlags(&f.s[i], cudaStreamNonBlocking) !=
                                    cudaSuccess) ||
                    (!f.join[i] && cudaEventCreateWithFlags(&f.join[i], cudaEventDisableTiming) !=
                                       cudaSuccess))
                    return nullptr;
        }
        a.ready = true;
    }
    ForkSet* f = &a.set[a.next];
    a.next = (a.next + 1) % kForkSets;
    return f;
}

}  // namespace lqt
