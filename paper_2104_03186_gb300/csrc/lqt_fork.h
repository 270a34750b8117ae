// Auxiliary streams for the independent parts of one call (the state sizes of a
// batch or of a set of warm solves).
//
// A host thread holds kForkSets sets per device and takes them in turn, so
// that the calls it has in flight on several streams of its own do not queue on
// one another's auxiliary streams (with more calls in flight than sets, a set's
// later call waits for its earlier one; the results do not depend on it).  The
// sets are made on the thread's first forked call on a device, or taken over
// from a thread that has ended (its destructor puts them on a list and makes no
// CUDA call: it can run after the CUDA runtime has shut down), so a process
// keeps as many as it ever had threads in forked calls at once.
#pragma once

#include <cuda_runtime.h>

#include <mutex>
#include <vector>

namespace lqt {

constexpr int kForkStreams = 3, kForkSets = 4, kForkDevices = 64;

struct ForkSet {
    cudaStream_t s[kForkStreams] = {};
    cudaEvent_t fork = nullptr, join[kForkStreams] = {};
};

struct ForkSets {
    ForkSet set[kForkSets];
    int next = 0;
    bool ready = false;
};

// Sets of threads that have ended.  Never destroyed: a thread may end after the
// static destructors have run.
struct ForkPool {
    std::mutex lock;
    std::vector<ForkSets*> free[kForkDevices];

    static ForkPool& get() {
        static ForkPool* pool = new ForkPool;
        return *pool;
    }
};

struct ForkHolder {
    ForkSets* sets[kForkDevices] = {};

    ForkSets* on(int dev) {
        if (sets[dev]) return sets[dev];
        ForkPool& pool = ForkPool::get();
        std::lock_guard<std::mutex> g(pool.lock);
        if (pool.free[dev].empty()) return sets[dev] = new ForkSets;
        sets[dev] = pool.free[dev].back();
        pool.free[dev].pop_back();
        return sets[dev];
    }

    ~ForkHolder() {
        ForkPool& pool = ForkPool::get();
        std::lock_guard<std::mutex> g(pool.lock);
        for (int d = 0; d < kForkDevices; ++d)
            if (sets[d]) pool.free[d].push_back(sets[d]);
    }
};

// Makes what the sets still lack.  Handles made by an earlier, failed attempt
// are kept and not made again.
inline bool fork_sets_ready(ForkSets& a) {
    if (a.ready) return true;
    // the calling thread may be capturing: making streams and events is not
    // part of the capture, so it is done in the relaxed mode
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    if (cudaThreadExchangeStreamCaptureMode(&mode) != cudaSuccess) return false;
    bool ok = true;
    for (ForkSet& f : a.set) {
        ok = ok && (f.fork ||
                    cudaEventCreateWithFlags(&f.fork, cudaEventDisableTiming) == cudaSuccess);
        for (int i = 0; i < kForkStreams; ++i)
            ok = ok &&
                 (f.s[i] ||
                  cudaStreamCreateWithFlags(&f.s[i], cudaStreamNonBlocking) == cudaSuccess) &&
                 (f.join[i] || cudaEventCreateWithFlags(&f.join[i], cudaEventDisableTiming) ==
                                   cudaSuccess);
    }
    a.ready = ok;
    return cudaThreadExchangeStreamCaptureMode(&mode) == cudaSuccess && ok;
}

// The capture that stream s takes part in; 0 for none.
inline unsigned long long capture_of(cudaStream_t s) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    unsigned long long id = 0;
    if (cudaStreamGetCaptureInfo(s, &st, &id) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return st == cudaStreamCaptureStatusNone ? 0 : id;
}

// The next set of this thread for a call on stream s of the current device.  A
// set whose streams an open capture other than s's holds is passed over: work
// put there would become part of that capture.  nullptr if no set can be had
// (the call then runs on one stream).
inline ForkSet* next_fork_set(cudaStream_t s) {
    thread_local ForkHolder holder;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kForkDevices) return nullptr;
    ForkSets& a = *holder.on(dev);
    if (!fork_sets_ready(a)) return nullptr;
    const unsigned long long own = capture_of(s);
    for (int k = 0; k < kForkSets; ++k) {
        ForkSet* f = &a.set[a.next];
        a.next = (a.next + 1) % kForkSets;
        bool fits = true;
        for (int i = 0; i < kForkStreams; ++i) {
            const unsigned long long id = capture_of(f->s[i]);
            fits = fits && (id == 0 || id == own);
        }
        if (fits) return f;
    }
    return nullptr;
}

}  // namespace lqt
