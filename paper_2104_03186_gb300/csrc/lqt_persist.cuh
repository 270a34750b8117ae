// The chunked pipeline of lqt_chain.cuh in one persistent launch.
//
// The level-by-level pipeline launches one kernel per tree level (a batch of
// 4096 problems took about 100 launches per state size).  Here one
// cooperative launch of as many CTAs as are co-resident runs every phase in
// turn: the chunk folds, the up-sweep levels of Alg. 1, the terminal values,
// the down-sweep levels of the value carries, the Riccati re-folds, the
// up- and down-sweep levels of the trajectory maps and the rollouts.  Within
// a phase the CTAs' teams take work items: the chunks of the fold, re-fold and
// rollout from a counter (whichever team is free takes the next one), the
// pairs of a tree level by a grid stride; between phases a grid barrier orders
// the global-memory results.  The per-item work is the same device code as the
// level kernels' (lqt_team_chain.cuh, lqt_team.cuh).
//
// Each team owns a block sized for the largest phase; the terminal values run on
// the first N lanes of a team (lane-group code), the rollouts one warp a chunk.
//
// The barrier is a counter and a generation word in the workspace.  Every
// wait is bounded: a CTA that waits longer than the limit records
// LQT_ETIMEOUT in the status word and leaves the kernel, so a missing CTA can
// never hang the GPU.  The cooperative launch guarantees that all CTAs are
// resident at once, so the limit is never reached in a correct launch.
#pragma once

#include <cuda_runtime.h>

#include "lqt_chain.cuh"
#include "lqt_vector_walk.cuh"

namespace lqt {
namespace chain {

constexpr int kStatusTimeout = 6;  // LQT_ETIMEOUT
constexpr int kMaxLevels = 24;

struct GridBarrier {
    unsigned int count;
    unsigned int gen;
    unsigned long long next[3];  // work counters of the fold, re-fold and rollout phases
};

// The next chunk of a phase for the calling team (lane 0 draws, the team
// shares it through `slot`): chunks go to whichever team is free, as the
// hardware would hand out the CTAs of a launch, so chunks of different lengths
// balance.
template <int N>
__device__ __forceinline__ long long next_chunk(unsigned long long* counter,
                                                unsigned long long* slot, const Team<N>& g) {
    g.sync();  // the slot's last value has been read
    if (g.lane == 0) *slot = atomicAdd(counter, 1ull);
    g.sync();
    return (long long)*slot;
}

// Active chunk counts of the tree levels (as in the level-by-level launch).
struct LevelPlan {
    int levels;
    long long active[kMaxLevels];
};

// Grid-wide barrier; returns false (in every thread of the CTA) when the
// wait ran out.
__device__ __forceinline__ bool grid_sync(GridBarrier* b, unsigned int nblocks,
                                          long long limit, int* status) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        s_ok = 1;
        volatile unsigned int* vgen = &b->gen;
        const unsigned int my = *vgen;
        __threadfence();
        if (atomicAdd(&b->count, 1u) == nblocks - 1) {
            b->count = 0;
            __threadfence();
            atomicAdd(&b->gen, 1u);
        } else {
            long long i = 0;
            while (*vgen == my) {
                if (++i > limit) {
                    s_ok = 0;
                    atomicCAS(status, 0, kStatusTimeout);
                    break;
                }
                __nanosleep(64);
            }
        }
        __threadfence();
    }
    __syncthreads();
    return s_ok != 0;
}

// The terminal value of item q by one lane group (k_cterm's work): V[c0],
// S_T, v_T, the trajectory seed x_0 and, for T = 0, x_0 itself.  Y: group
// scratch of 2N x N + 2N elements of RT.
template <typename R, typename RT, int N>
__device__ __forceinline__ void b_cterm_group(const Args<R, RT>& a, int q, RT* Y,
                                              const Group<N>& g) {
    const Item<R>& it = a.items[q];
    const DescT<R>& D = it.D;
    const int r = g.lr;
    const int pT = D.pT;
    RT* xr = Y + 2 * N * N;
    for (int i = r; i < pT; i += N) {
        RT acc[N];
        RT t0 = RT(0);
#pragma unroll
        for (int j = 0; j < N; ++j) acc[j] = RT(0);
        for (int b = 0; b < pT; ++b) {
            const RT xib = static_cast<RT>(D.XT[i * pT + b]);
#pragma unroll
            for (int j = 0; j < N; ++j) acc[j] += xib * static_cast<RT>(D.HT[b * N + j]);
            if (D.rT) t0 += xib * static_cast<RT>(D.rT[b]);
        }
#pragma unroll
        for (int j = 0; j < N; ++j) Y[i * N + j] = acc[j];
        xr[i] = t0;
    }
    g.sync();
    RT acc[N];
    RT t = RT(0);
#pragma unroll
    for (int j = 0; j < N; ++j) acc[j] = RT(0);
    for (int i = 0; i < pT; ++i) {
        const RT hi = static_cast<RT>(D.HT[i * N + r]);
#pragma unroll
        for (int j = 0; j < N; ++j) acc[j] += hi * Y[i * N + j];
        t += hi * xr[i];
    }
    if (D.etaT) t = static_cast<RT>(D.etaT[r]);
    RT* val = a.V + it.c0 * GValue<N>::SIZE;
#pragma unroll
    for (int j = 0; j < N; ++j) val[GValue<N>::OS + r * GValue<N>::LD + j] = acc[j];
    val[GValue<N>::OV + r] = t;
    a.X[(it.c0 + it.NC - 1) * N + r] = static_cast<RT>(D.x0[r]);
    if (a.out_mask & 1) {
#pragma unroll
        for (int j = 0; j < N; ++j) D.S[D.T * N * N + r * N + j] = static_cast<R>(acc[j]);
    }
    if (a.out_mask & 4) D.v[D.T * N + r] = static_cast<R>(t);
    if (D.T == 0) D.x[r] = D.x0[r];
    g.sync();
}

// Shared memory of one team of the persistent kernel (bytes, a multiple of
// 16): the largest block of its phases.
template <typename R, typename RT, int N, int M>
constexpr int persist_team_bytes() {
    constexpr int sizes[] = {tstride_of<N, R>(TFoldSmem<N, M>::SIZE) * (int)sizeof(R),
                             tstride_of<N, R>(TRefoldSmem<N, M>::SIZE) * (int)sizeof(R),
                             VWalk<N, M>::FWD_SIZE * (int)sizeof(R) / (N == 8 ? 4 : 1),
                             tstride_of<N, RT>(team::CombineSmem<N>::SIZE) * (int)sizeof(RT),
                             tstride_of<N, RT>(team::ApplySmem<N>::SIZE) * (int)sizeof(RT),
                             (2 * N * N + 2 * N) * (int)sizeof(RT)};
    int m = 0;
    for (int s : sizes) m = s > m ? s : m;
    return (m + 15) / 16 * 16;
}

template <typename R, typename RT, int N, int M, int NT>
__global__ void __launch_bounds__(NT* Team<N>::LG) k_cpersist(Args<R, RT> a, LevelPlan lp,
                                                              GridBarrier* bar,
                                                              long long wait_limit) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned long long slots[NT];
    constexpr int GB = persist_team_bytes<R, RT, N, M>();
    const Team<N> g;
    const Group<N> lanes_g;  // the first N lanes of the team, in the lane-group phases
    const int gi = threadIdx.x / Team<N>::LG;
    const bool lead = g.lane < N;
    unsigned char* mine = smem_raw + gi * GB;
    R* sh = reinterpret_cast<R*>(mine);
    RT* sht = reinterpret_cast<RT*>(mine);
    unsigned long long* slot = &slots[gi];
    const long long first = (long long)blockIdx.x * NT + gi;
    const long long stride = (long long)gridDim.x * NT;
    const unsigned int nb = gridDim.x;
    const long long C = a.C;
    bool ok = true;
    // 1. chunk folds
    for (long long c = next_chunk(&bar->next[0], slot, g); c < C;
         c = next_chunk(&bar->next[0], slot, g))
        b_tfold<R, RT, N, M>(a, c, sh);
    if (!grid_sync(bar, nb, wait_limit, a.status)) return;
    // 2. up-sweep levels (a problem's root is in no suffix: level h sweeps the
    // problems with NC >= 4h)
    for (int l = 0; l + 1 < lp.levels; ++l) {
        const long long h = 1ll << l, pairs = lp.active[l + 1] / (2 * h);
        for (long long q = first; q < pairs; q += stride) {
            RT* e = a.E + q * 2 * h * DElem<N>::SIZE;
            ok &= team::combine<N>(e, e + h * DElem<N>::SIZE, e, sht, g);
            g.sync();
        }
        if (!grid_sync(bar, nb, wait_limit, a.status)) return;
    }
    // 3. terminal values, then the down-sweep levels of the value carries
    if (lead)
        for (long long q = first; q < a.count; q += stride)
            b_cterm_group<R, RT, N>(a, (int)q, sht, lanes_g);
    if (!grid_sync(bar, nb, wait_limit, a.status)) return;
    for (int l = lp.levels - 1; l >= 0; --l) {
        const long long h = 1ll << l, pairs = lp.active[l] / (2 * h);
        for (long long q = first; q < pairs; q += stride) {
            const long long i = q * 2 * h;
            RT* val = a.V + i * DValue<N>::SIZE;
            for (int t = g.lane; t < DValue<N>::SIZE; t += Team<N>::LG)
                val[h * DValue<N>::SIZE + t] = val[t];
            ok &= team::value_apply<N>(a.E + (i + h) * DElem<N>::SIZE, val, val, sht, g);
            g.sync();
        }
        if (!grid_sync(bar, nb, wait_limit, a.status)) return;
    }
    // 4. Riccati re-folds with the outputs and the chunk maps
    for (long long c = next_chunk(&bar->next[1], slot, g); c < C;
         c = next_chunk(&bar->next[1], slot, g))
        b_trefold<R, RT, N, M>(a, c, sh);
    if (!grid_sync(bar, nb, wait_limit, a.status)) return;
    // 5. trajectory maps: up-sweep, then down-sweep from x_0
    for (int l = 0; l < lp.levels; ++l) {
        const long long h = 1ll << l, pairs = lp.active[l] / (2 * h);
        for (long long q = first; q < pairs; q += stride) {
            RT* f = a.FE + (q * 2 * h + 2 * h - 1) * DAffine<N>::SIZE;
            team::affine_compose<N>(f - h * DAffine<N>::SIZE, f, f, sht, g);
            g.sync();
        }
        if (!grid_sync(bar, nb, wait_limit, a.status)) return;
    }
    for (int l = lp.levels - 1; l >= 0; --l) {
        const long long h = 1ll << l, pairs = lp.active[l] / (2 * h);
        for (long long q = first; q < pairs; q += stride) {
            const long long j = q * 2 * h + 2 * h - 1;
            RT y0, y1;
            for (int i = g.lane; i < N; i += Team<N>::LG) a.X[(j - h) * N + i] = a.X[j * N + i];
            team::affine_apply<N>(a.FE + (j - h) * DAffine<N>::SIZE, a.X + j * N, y0, y1, g);
            g.sync();  // every lane has read X[j]
            if (g.ci == 0) {
                a.X[j * N + g.ri] = y0;
                a.X[j * N + g.ri + N / 2] = y1;
            }
        }
        if (!grid_sync(bar, nb, wait_limit, a.status)) return;
    }
    // 6. rollouts, one warp per chunk: the first warp of a team, or (n = 8) every
    // warp in the blocks of its four teams
    constexpr int LG = Team<N>::LG, TW = LG < 32 ? 32 / LG : 1;  // teams per warp
    static_assert(VWalk<N, M>::FWD_SIZE * (int)sizeof(R) <= TW * GB, "a rollout's ring fits");
    if (g.lane < 32) {
        const int lane = threadIdx.x & 31;
        R* ring = reinterpret_cast<R*>(smem_raw + gi / TW * TW * GB);
        for (;;) {
            unsigned long long c = 0;
            if (lane == 0) c = atomicAdd(&bar->next[2], 1ull);
            c = __shfl_sync(0xffffffffu, c, 0);
            if ((long long)c >= C) break;
            b_vfwd<R, RT, N, M, false>(a, (long long)c, nullptr, ring);
            __syncwarp();
        }
    }
    flag(a.status, ok);
}

}  // namespace chain
}  // namespace lqt
