// Arguments of the chunked pipeline's kernels and the layout of its chunk
// arrays in global memory (lqt_chain.cuh, lqt_team_chain.cuh).
#pragma once

#include <cuda_runtime.h>

#include "lqt_lane_step.cuh"

namespace lqt {
namespace chain {

using namespace lanes;

constexpr int kStatusSingular = 8;  // LQT_ESINGULAR

template <typename R>
struct Item {
    DescT<R> D;
    long long B;   // steps per chunk
    long long c0;  // first chunk in the chunk arrays (a multiple of NC)
    long long r0;  // first row of the residual kernel's index space (T + 1 rows each)
    int NC;        // chunks (a power of two)
    int pad_;
    R* u_out;      // correction pass: the output u* (holds u^ until then)
    const R* qh;   // correction pass: U^{-1} h_k (T x M)
    R* gi;         // refinement: G_k^{-1} of the first pass (T x M x M), or nullptr
};

template <typename R, typename RT>
struct Args {
    const Item<R>* items;  // count items, by decreasing NC (increasing c0)
    int count;
    long long C;     // total chunks
    RT* E;           // C chunk totals (LElem)
    RT* V;           // C value carries (LValue): the value at each chunk's end
    RT* FE;          // C chunk affine maps (LAffine)
    RT* X;           // C chunk start states
    int* status;
    int out_mask;    // bit 1: write S; bit 2: write K; bit 4: write v
    RT* maps;        // refinement: a copy of every chunk map, or nullptr
    int first_total; // 1: the problems' first chunks need whole totals (Method 2)
    int refine_add;  // 1: correction pass: x <- x^ + dx, u_out <- u^ + w - qh
};

// The item whose chunks contain chunk c (items sorted by c0).
template <typename R>
__device__ __forceinline__ int find_chunk(const Item<R>* items, int count, long long c) {
    int lo = 0, hi = count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (items[mid].c0 <= c) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// The item whose residual rows contain row q (items sorted by r0).
template <typename R>
__device__ __forceinline__ int find_row(const Item<R>* items, int count, long long q) {
    int lo = 0, hi = count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (items[mid].r0 <= q) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

template <typename A, typename B>
__device__ __forceinline__ void copy_in(A* dst, const B* src, int count, int lr, int lanes) {
    for (int i = lr; i < count; i += lanes) dst[i] = static_cast<A>(src[i]);
}

__device__ __forceinline__ void flag(int* status, bool ok) {
    if (!ok) atomicCAS(status, 0, kStatusSingular);
}

// Chunk totals, value carries and chunk maps in global memory: dense rows at
// n >= 8 (read by 16-byte loads, lqt_team.cuh), the lane kernels' odd row
// stride at n = 4.
template <int N>
constexpr int gld() {
    return N >= 8 ? N : lds(N);
}
template <int N>
struct GElem {
    static constexpr int LD = gld<N>();
    static constexpr int OA = 0, OB = N * LD, OC = OB + N, OE = OC + N * LD, OJ = OE + N,
                         SIZE = OJ + N * LD;
};
template <int N>
struct GValue {
    static constexpr int LD = gld<N>();
    static constexpr int OS = 0, OV = N * LD, SIZE = N * LD + N;
};
template <int N>
struct GAffine {
    static constexpr int LD = gld<N>();
    static constexpr int OF = 0, OC = N * LD, SIZE = N * LD + N;
};

}  // namespace chain
}  // namespace lqt
