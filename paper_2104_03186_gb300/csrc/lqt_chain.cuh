// Chunked pipeline for the lane-group sizes (n = 8, 16, 32): one problem
// (lqt_solve) or a ragged batch of problems of one (n, m) (lqt_solve_batched).
//
// Problem i's T_i steps are cut into NC_i chunks (NC_i a power of two) of B_i
// steps; one team of lanes works on one chunk at a time, and the scans over the
// chunk results run over tree levels with the chunk results in global memory.
// The problems are laid out by decreasing NC_i, problem i's chunks at
// [c0_i, c0_i + NC_i), so every c0_i is a multiple of NC_i: at tree level h the
// pairs of all problems with NC_i >= 2h are the pairs (i, i + h), i a multiple of
// 2h, of one prefix of the chunk array, and the level kernels need no per-problem
// lookup.  Per pass (n >= 8, lqt_team_chain.cuh; k_c* of this file at n = 4, a
// lane group of N lanes per chunk and a launch per level):
//   k_tfold    chunk totals a_s (x) ... (x) a_{e-1} (eq. lqt_comb), folded one
//              step at a time from the end in the low-rank form of fold_step,
//   k_tup      up-sweep levels of the chunk totals (Alg. 1, left-anchored),
//   k_cterm    the terminal value (H_T^T X_T r_T, H_T^T X_T H_T),
//   k_tdown    down-sweep levels of the value carries (Lemma LQT_assoc: a
//              suffix applied to the value element (0, 0, 0, v, S)),
//   k_trefold  per chunk the Riccati recursion from its carry (Sec. II-B),
//              writing S_k, v_k, K_k and the feedforward d_k, and the chunk's
//              closed-loop affine map (Sec. IV-C),
//   k_tfup / k_tfdown  up- and down-sweeps of the affine maps from x_0
//              (right-anchored), giving every chunk's start state,
//   k_vfwd     per chunk the rollout of x*_k and u*_k (eq. Control_LQT,
//              lqt_vector_walk.cuh).
// The chunk phases compute in R; the tree levels store and compute in RT
// (RT = double with R = float is the mixed-precision form: FP32 chunk work,
// FP64 tree levels and their (I + C J) solves).
//
// Refinement (one step of iterative refinement of the KKT system of the QP):
// k_vresid (n = 4: k_cresid) evaluates, in twice the working precision (FP64 arithmetic, or
// compensated FP32 dot products for FP32 problems), the residuals of the
// optimality conditions at
// the first pass's iterate (x^, u^, lambda^ with lambda^_k = S_k x^_k - v_k,
// the gradient of the value function):
//   e_k = F_k x^_k + c_k + L_k u^_k - x^_{k+1}                    (dynamics)
//   g_k = H_k^T X_k (H_k x^_k - r_k) + F_k^T lambda^_{k+1} - lambda^_k (d/dx_k)
//   h_k = U_k u^_k + L_k^T lambda^_{k+1}                             (d/du_k)
//   g_T = H_T^T X_T (H_T x^_T - r_T) - lambda^_T
// The correction (dx, du) minimises sum 1/2 dx^T H^T X H dx + g^T dx +
// 1/2 du^T U du + h^T du subject to dx_{k+1} = F dx_k + L du_k + e_k, dx_0 = 0.
// With du = w - U^{-1} h this is the LQT problem of Sec. II-B with linear
// state terms eta_k = -g_k, eta_T = -g_T (no reference), offsets
// c~_k = e_k - L U^{-1} h_k and control w.  Its S and K equal the first pass's:
// at n >= 8 the second pass is vector walks and affine scans (k_vback, k_vfwd),
// otherwise (n = 4, Method 2, the sequential recursion, the least workspace) the
// same kernels again; it adds x = x^ + dx, u = u^ + w - U^{-1} h.
// After a Newton step (FULL) the walks read the corrected S and K, while the maps
// and G^{-1} kept by the re-fold are those before it.  They carry dx and dv, 1e-5
// of x and v at most, so their own error (that of the first pass's K, 1e-5 to 1e-2
// relative) stays below a rounding of x* and u*: the precision study (cond(X_k) =
// 1e6, T = 8192) has 2.56e-8 and 2.55e-8 with the mixed operators, 2.63e-8 and
// 2.64e-8 with a full second pass.
#pragma once

#include <cuda_runtime.h>

#include "lqt_chain_args.cuh"
#include "lqt_lane_step.cuh"
#include "lqt_refine.cuh"
#include "lqt_team_chain.cuh"
#include "lqt_tma.cuh"

namespace lqt {
namespace chain {

using namespace lanes;

// The constant matrices of the Newton correction problem: L = 0, U = I, H = I.
template <typename R, int N, int M>
__global__ void k_consts(R* L0, R* UI, R* HI) {
    const int r = threadIdx.x;
    for (int a = 0; a < M; ++a) L0[r * M + a] = R(0);
    if (r < M)
        for (int b = 0; b < M; ++b) UI[r * M + b] = r == b ? R(1) : R(0);
    for (int j = 0; j < N; ++j) HI[r * N + j] = r == j ? R(1) : R(0);
}

// Items of a one-problem call, from kernel parameters.
template <typename R>
__global__ void k_set_items(Item<R>* d1, Item<R> a, Item<R>* d2, Item<R> b) {
    *d1 = a;
    if (d2) *d2 = b;
}

// ---- shared-memory sizes per group (elements of the kernel's arithmetic type)
template <int N, int M, typename R>
struct FoldSmem {  // P | step (E, L, U) | scratch overlapping the step's Y
    static constexpr int P = 0;
    static constexpr int SB = LElem<N>::SIZE;
    static constexpr int SCR_OFF = SB + StepLayout<N, M>::Y;
    static constexpr int SCR =
        fold_scratch<N, M, R>() > StepLayout<N, M>::SIZE - StepLayout<N, M>::Y
            ? fold_scratch<N, M, R>()
            : StepLayout<N, M>::SIZE - StepLayout<N, M>::Y;
    static constexpr int SIZE = SCR_OFF + SCR;
};

template <int N, int M>
struct RefoldSmem {  // val | Phi | step | scratch (riccati + Kd + Ft) overlapping Y
    static constexpr int VAL = 0;
    static constexpr int PHI = LValue<N>::SIZE;
    static constexpr int SB = PHI + LAffine<N>::SIZE;
    static constexpr int SCR_OFF = SB + StepLayout<N, M>::Y;
    static constexpr int RIC = riccati_scratch<N, M>() + M * kd_ld<N>() + LAffine<N>::SIZE;
    static constexpr int SCR = RIC > StepLayout<N, M>::SIZE - StepLayout<N, M>::Y
                                   ? RIC
                                   : StepLayout<N, M>::SIZE - StepLayout<N, M>::Y;
    static constexpr int SIZE = SCR_OFF + SCR;
};

template <int N>
struct UpSmem {
    static constexpr int SIZE = 2 * LElem<N>::SIZE + combine_scratch<N>();
};

template <int N>
struct DownSmem {
    static constexpr int SIZE = LElem<N>::SIZE + LValue<N>::SIZE + value_scratch<N>();
};

template <int N>
struct FupSmem {
    static constexpr int SIZE = 2 * LAffine<N>::SIZE;
};

template <int N>
struct FdownSmem {
    static constexpr int SIZE = LAffine<N>::SIZE + N;
};

template <int N, int M>
struct RollSmem {  // x, u, then two buffers of F_k (N x lds(N)), L_k (N x lds(M)), K_k (M x lds(N))
    static constexpr int F = N + M;
    static constexpr int L = F + N * lds(N);
    static constexpr int K = L + N * lds(M);
    static constexpr int BUF = N * lds(N) + N * lds(M) + M * lds(N);  // one step's matrices
    static constexpr int SIZE = F + 2 * BUF;
};

// Groups per CTA: at most 256 threads, and at most 112 KB of shared memory so
// that two CTAs share an SM (228 KB, 1 KB of it reserved per CTA).
template <int N>
constexpr int groups_for(int bytes_per_group) {
    int g = 256 / N;
    while (g > 1 && g * bytes_per_group > 112 * 1024) --g;
    return g;
}

// H_k = I for every step (time-invariant identity with p = N): the step
// loader then skips the H^T X H products.  Uniform over the group.
template <typename R, int N>
__device__ __forceinline__ bool h_is_identity(const DescT<R>& D, const Group<N>& g) {
    if (D.sH != 0 || D.p != N || !D.H) return false;
    bool mine = true;
    for (int j = 0; j < N; ++j) mine = mine && D.H[g.lr * N + j] == (g.lr == j ? R(1) : R(0));
    return __all_sync(g.mask, mine);
}

// ---- chunk totals ----------------------------------------------------------
template <typename R, typename RT, int N, int M, int NG>
__device__ __forceinline__ void b_cfold(const Args<R, RT>& a, long long c,
                                        unsigned char* smem_raw, int gi) {
    using S = FoldSmem<N, M, R>;
    using E = LElem<N>;
    R* sh = reinterpret_cast<R*>(smem_raw);
    const Group<N> g;
    const Item<R>& it = a.items[find_chunk(a.items, a.count, c)];
    const DescT<R>& D = it.D;
    R* gs = sh + gi * gstride<N>(S::SIZE);
    R* P = gs + S::P;
    R* sb = gs + S::SB;
    R* scr = gs + S::SCR_OFF;
    const long long T = D.T;
    const long long lc = c - it.c0;
    const long long s0 = lc * it.B < T ? lc * it.B : T;
    const long long e0 = s0 + it.B < T ? s0 + it.B : T;
    bool ok = true;
    set_neutral<N, N>(P, g);
    // staging area for the step inputs: the scratch beyond the step's Y
    constexpr int YS = StepLayout<N, M>::SIZE - StepLayout<N, M>::Y;
    const bool hid = h_is_identity(D, g);
    for (long long k = e0 - 1; k >= s0; --k) {
        load_step<R, N, M, false>(D, k, sb, scr, g, ok, scr + YS, S::SCR - YS, hid);
        ok &= fold_step<R, N, M>(P, sb, scr, g);
    }
    RT* out = a.E + c * E::SIZE;
    for (int i = g.lr; i < E::SIZE; i += N) out[i] = static_cast<RT>(P[i]);
    flag(a.status, ok);
}

template <typename R, typename RT, int N, int M, int NG>
__global__ void __launch_bounds__(NG* N) k_cfold(Args<R, RT> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int gi = threadIdx.x / N;
    const long long c = (long long)blockIdx.x * NG + gi;
    if (c >= a.C) return;
    b_cfold<R, RT, N, M, NG>(a, c, smem_raw, gi);
}

// ---- up-sweep level h: E[i] <- E[i] (x) E[i + h], i a multiple of 2h -------
// (i < active: the chunks of the problems with NC >= 2h)
template <typename RT, int N, int NG>
__device__ __forceinline__ void b_cup(RT* E_, long long active, int h, int* status, long long i,
                                        unsigned char* smem_raw, int gi) {
    using E = LElem<N>;
    RT* sh = reinterpret_cast<RT*>(smem_raw);
    const Group<N> g;
    RT* e1 = sh + gi * gstride<N>(UpSmem<N>::SIZE);
    RT* e2 = e1 + E::SIZE;
    RT* scr = e2 + E::SIZE;
    copy_in(e1, E_ + i * E::SIZE, E::SIZE, g.lr, N);
    copy_in(e2, E_ + (i + h) * E::SIZE, E::SIZE, g.lr, N);
    g.sync();
    const bool ok = combine<N, N>(e1, e2, e1, scr, g);
    RT* out = E_ + i * E::SIZE;
    for (int t = g.lr; t < E::SIZE; t += N) out[t] = e1[t];
    flag(status, ok);
}

template <typename RT, int N, int NG>
__global__ void __launch_bounds__(NG* N) k_cup(RT* E_, long long active, int h, int* status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int gi = threadIdx.x / N;
    const long long i = ((long long)blockIdx.x * NG + gi) * 2 * h;
    if (i >= active) return;
    b_cup<RT, N, NG>(E_, active, h, status, i, smem_raw, gi);
}

// ---- terminal values (one CTA of N threads per problem): V[c0] <- the value
// element (H_T^T X_T r_T, H_T^T X_T H_T), S_T, v_T, and X[c0 + NC - 1] <- x_0
template <typename R, typename RT, int N>
__global__ void __launch_bounds__(N) k_cterm(Args<R, RT> a) {
    __shared__ RT Y[2 * N * N + 2 * N];  // X_T H_T (pT x N) and X_T r_T, pT <= 2N
    const Item<R>& it = a.items[blockIdx.x];
    const DescT<R>& D = it.D;
    const int r = threadIdx.x;
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
    __syncthreads();
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
}

// ---- down-sweep level h: V[i + h] <- V[i]; V[i] <- E[i + h] (x) V[i] --------
template <typename RT, int N, int NG>
__device__ __forceinline__ void b_cdown(const RT* E_, RT* V_, long long active, int h,
                                                 int* status, long long i,
                                        unsigned char* smem_raw, int gi) {
    using E = LElem<N>;
    using V = LValue<N>;
    RT* sh = reinterpret_cast<RT*>(smem_raw);
    const Group<N> g;
    RT* e = sh + gi * gstride<N>(DownSmem<N>::SIZE);
    RT* val = e + E::SIZE;
    RT* scr = val + V::SIZE;
    copy_in(e, E_ + (i + h) * E::SIZE, E::SIZE, g.lr, N);
    copy_in(val, V_ + i * V::SIZE, V::SIZE, g.lr, N);
    for (int t = g.lr; t < V::SIZE; t += N) V_[(i + h) * V::SIZE + t] = V_[i * V::SIZE + t];
    g.sync();
    const bool ok = value_apply<N, N>(e, val, scr, g);
    for (int t = g.lr; t < V::SIZE; t += N) V_[i * V::SIZE + t] = val[t];
    flag(status, ok);
}

template <typename RT, int N, int NG>
__global__ void __launch_bounds__(NG* N) k_cdown(const RT* E_, RT* V_, long long active, int h,
                                                 int* status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int gi = threadIdx.x / N;
    const long long i = ((long long)blockIdx.x * NG + gi) * 2 * h;
    if (i >= active) return;
    b_cdown<RT, N, NG>(E_, V_, active, h, status, i, smem_raw, gi);
}

// ---- per-chunk Riccati re-fold with outputs and the chunk affine map -------
template <typename R, typename RT, int N, int M, int NG>
__device__ __forceinline__ void b_crefold(const Args<R, RT>& a, long long c,
                                        unsigned char* smem_raw, int gi) {
    using S = RefoldSmem<N, M>;
    using V = LValue<N>;
    using A = LAffine<N>;
    R* sh = reinterpret_cast<R*>(smem_raw);
    const Group<N> g;
    const Item<R>& it = a.items[find_chunk(a.items, a.count, c)];
    const DescT<R>& D = it.D;
    R* gs = sh + gi * gstride<N>(S::SIZE);
    R* val = gs + S::VAL;
    R* Phi = gs + S::PHI;
    R* sb = gs + S::SB;
    R* scr = gs + S::SCR_OFF;
    R* Kd = scr + riccati_scratch<N, M>();
    R* Ft = Kd + M * kd_ld<N>();
    const int r = g.lr;
    const long long T = D.T;
    const long long lc = c - it.c0;
    const long long s0 = lc * it.B < T ? lc * it.B : T;
    const long long e0 = s0 + it.B < T ? s0 + it.B : T;
    copy_in(val, a.V + c * V::SIZE, V::SIZE, r, N);
#pragma unroll
    for (int j = 0; j < N; ++j) Phi[A::OF + r * A::LD + j] = r == j ? R(1) : R(0);
    Phi[A::OC + r] = R(0);
    g.sync();
    bool ok = true;
    constexpr int YS = StepLayout<N, M>::SIZE - StepLayout<N, M>::Y;
    const bool hid = h_is_identity(D, g);
    for (long long k = e0 - 1; k >= s0; --k) {
        load_step<R, N, M, false>(D, k, sb, scr, g, ok, scr + YS, S::SCR - YS, hid);
        ok &= riccati<R, N, M>(val, sb, Kd, Ft, scr, g);
        // outputs by coalesced stores (lane r writes column r of each row)
        if (a.out_mask & 1) {
#pragma unroll 8
            for (int i = 0; i < N; ++i) D.S[k * N * N + i * N + r] = val[V::OS + i * V::LD + r];
        }
        if (a.out_mask & 4) D.v[k * N + r] = val[V::OV + r];
        if (a.out_mask & 2) {
#pragma unroll 8
            for (int i = 0; i < M; ++i) D.K[k * M * N + i * N + r] = Kd[i * kd_ld<N>() + r];
        }
        if (r < M) D.u[k * M + r] = Kd[r * kd_ld<N>() + N];  // feedforward d_k, replaced in the rollout
        // chunk map after adding step k: Phi <- Phi Ft (two rows per lane pair
        // over half the columns each, as in row_mul_pair), gamma <- gamma + Phi ct
        constexpr int H = N / 2;
        const int r0 = r & ~1, c0 = (r & 1) * H;
        R p0[H], p1[H];
        R gm = Phi[A::OC + r];
#pragma unroll
        for (int j = 0; j < H; ++j) {
            p0[j] = R(0);
            p1[j] = R(0);
        }
#pragma unroll 4
        for (int l = 0; l < N; ++l) {
            const R x0 = Phi[A::OF + r0 * A::LD + l], x1 = Phi[A::OF + (r0 + 1) * A::LD + l];
#pragma unroll
            for (int j = 0; j < H; ++j) {
                const R y = Ft[A::OF + l * A::LD + c0 + j];
                p0[j] += x0 * y;
                p1[j] += x1 * y;
            }
            gm += (r & 1 ? x1 : x0) * Ft[A::OC + l];
        }
        g.sync();
        const bool odd = r & 1;  // stores in reverse order, as in row_mul_pair
#pragma unroll
        for (int j = 0; j < H; ++j) {
            const int jj = odd ? H - 1 - j : j;
            Phi[A::OF + r0 * A::LD + c0 + jj] = odd ? p0[H - 1 - j] : p0[j];
            Phi[A::OF + (r0 + 1) * A::LD + c0 + jj] = odd ? p1[H - 1 - j] : p1[j];
        }
        Phi[A::OC + r] = gm;
        g.sync();
    }
    RT* out = a.FE + c * A::SIZE;
    for (int t = r; t < A::SIZE; t += N) out[t] = static_cast<RT>(Phi[t]);
    flag(a.status, ok);
}

template <typename R, typename RT, int N, int M, int NG>
__global__ void __launch_bounds__(NG* N) k_crefold(Args<R, RT> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int gi = threadIdx.x / N;
    const long long c = (long long)blockIdx.x * NG + gi;
    if (c >= a.C) return;
    b_crefold<R, RT, N, M, NG>(a, c, smem_raw, gi);
}

// ---- forward up-sweep level h: FE[j] <- FE[j] o FE[j - h], j = 2h q + 2h - 1
template <typename RT, int N, int NG>
__device__ __forceinline__ void b_cfup(RT* FE, long long active, int h, long long j,
                                        unsigned char* smem_raw, int gi) {
    using A = LAffine<N>;
    RT* sh = reinterpret_cast<RT*>(smem_raw);
    const Group<N> g;
    RT* f1 = sh + gi * gstride<N>(FupSmem<N>::SIZE);
    RT* f2 = f1 + A::SIZE;
    copy_in(f1, FE + (j - h) * A::SIZE, A::SIZE, g.lr, N);
    copy_in(f2, FE + j * A::SIZE, A::SIZE, g.lr, N);
    g.sync();
    affine_compose<N, N>(f1, f2, f2, f1, g);
    for (int t = g.lr; t < A::SIZE; t += N) FE[j * A::SIZE + t] = f2[t];
}

template <typename RT, int N, int NG>
__global__ void __launch_bounds__(NG* N) k_cfup(RT* FE, long long active, int h) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int gi = threadIdx.x / N;
    const long long j = ((long long)blockIdx.x * NG + gi) * 2 * h + 2 * h - 1;
    if (j >= active) return;
    b_cfup<RT, N, NG>(FE, active, h, j, smem_raw, gi);
}

// ---- forward down-sweep level h: X[j - h] <- X[j]; X[j] <- FE[j - h](X[j]) -
// (each problem's top slot X[c0 + NC - 1] holds x_0 from k_cterm)
template <typename RT, int N, int NG>
__device__ __forceinline__ void b_cfdown(const RT* FE, RT* X, long long active, int h, long long j,
                                        unsigned char* smem_raw, int gi) {
    using A = LAffine<N>;
    RT* sh = reinterpret_cast<RT*>(smem_raw);
    const Group<N> g;
    RT* f = sh + gi * gstride<N>(FdownSmem<N>::SIZE);
    RT* x = f + A::SIZE;
    const int r = g.lr;
    copy_in(f, FE + (j - h) * A::SIZE, A::SIZE, r, N);
    const RT xv = X[j * N + r];
    x[r] = xv;
    X[(j - h) * N + r] = xv;
    g.sync();
    affine_apply<N, N>(f, x, g);
    X[j * N + r] = x[r];
}

template <typename RT, int N, int NG>
__global__ void __launch_bounds__(NG* N) k_cfdown(const RT* FE, RT* X, long long active, int h) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int gi = threadIdx.x / N;
    const long long j = ((long long)blockIdx.x * NG + gi) * 2 * h + 2 * h - 1;
    if (j >= active) return;
    b_cfdown<RT, N, NG>(FE, X, active, h, j, smem_raw, gi);
}

// ---- per-chunk rollout of x*_k and u*_k ------------------------------------
template <typename R, typename RT, int N, int M, int NG>
__device__ __forceinline__ void b_croll(const Args<R, RT>& a, long long c,
                                        unsigned char* smem_raw, int gi) {
    R* sh = reinterpret_cast<R*>(smem_raw);
    const Group<N> g;
    const Item<R>& it = a.items[find_chunk(a.items, a.count, c)];
    const DescT<R>& D = it.D;
    R* xc = sh + gi * gstride<N>(RollSmem<N, M>::SIZE);
    R* us = xc + N;
    const int r = g.lr;
    const long long T = D.T;
    const long long lc = c - it.c0;
    const long long s0 = lc * it.B < T ? lc * it.B : T;
    const long long e0 = s0 + it.B < T ? s0 + it.B : T;
    xc[r] = lc == 0 ? D.x0[r] : static_cast<R>(a.X[c * N + r]);
    g.sync();
    using RS = RollSmem<N, M>;
    constexpr int LD = lds(N), LM = lds(M);
    R* base = sh + gi * gstride<N>(RS::SIZE);
    // F_k, L_k, K_k into shared memory by coalesced asynchronous copies, one
    // step ahead (two buffers), so each step's loads overlap the step before
    auto stage = [&](long long k, int b) {
        R* Fb = base + RS::F + b * RS::BUF;
        R* Lb = base + RS::L + b * RS::BUF;
        R* Kb = base + RS::K + b * RS::BUF;
        const R* F = D.F + k * D.sF;
        const R* Lk = D.L + k * D.sL;
#pragma unroll 8
        for (int t = r; t < N * N; t += N) cp_async<sizeof(R)>(Fb + (t / N) * LD + t % N, F + t);
#pragma unroll 4
        for (int t = r; t < N * M; t += N) cp_async<sizeof(R)>(Lb + (t / M) * LM + t % M, Lk + t);
#pragma unroll 4
        for (int t = r; t < M * N; t += N)
            cp_async<sizeof(R)>(Kb + (t / N) * LD + t % N, D.K + k * M * N + t);
        cp_async_commit();
    };
    if (s0 < e0) stage(s0, 0);
    for (long long k = s0; k < e0; ++k) {
        const int b = (int)((k - s0) & 1);
        const R* Fs = base + RS::F + b * RS::BUF;
        const R* Ls = base + RS::L + b * RS::BUF;
        const R* Ks = base + RS::K + b * RS::BUF;
        if (k + 1 < e0) stage(k + 1, b ^ 1);  // that buffer was last read before step k's syncs
        const R xr = xc[r];
        D.x[k * N + r] = a.refine_add ? D.x[k * N + r] + xr : xr;
        if (k + 1 < e0)
            cp_async_wait<1>();
        else
            cp_async_wait<0>();
        g.sync();
        // u = d - K x (lanes a < M), published through shared memory
        if (r < M) {
            R t = D.u[k * M + r];
#pragma unroll
            for (int j = 0; j < N; ++j) t -= Ks[r * LD + j] * xc[j];
            us[r] = t;
            if (a.refine_add)
                it.u_out[k * M + r] = it.u_out[k * M + r] + (t - it.qh[k * M + r]);
            else
                D.u[k * M + r] = t;
        }
        g.sync();
        R t = D.c ? D.c[k * D.sc + r] : R(0);
#pragma unroll
        for (int j = 0; j < N; ++j) t += Fs[r * LD + j] * xc[j];
#pragma unroll
        for (int b = 0; b < M; ++b) t += Ls[r * LM + b] * us[b];
        g.sync();
        xc[r] = t;
        g.sync();
        if (k == T - 1) D.x[T * N + r] = a.refine_add ? D.x[T * N + r] + t : t;
    }
}

template <typename R, typename RT, int N, int M, int NG>
__global__ void __launch_bounds__(NG* N) k_croll(Args<R, RT> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int gi = threadIdx.x / N;
    const long long c = (long long)blockIdx.x * NG + gi;
    if (c >= a.C) return;
    b_croll<R, RT, N, M, NG>(a, c, smem_raw, gi);
}

// ---- Method 2 (Lemma LQT_trajectory_method2) --------------------------------
// The forward conditional value functions V_{S->k} are the prefix products
// e_0 (x) a_0 (x) ... (x) a_{k-1} of the same elements, seeded with the element
// (0, x_0, 0, 0, 0) of Remark LQT_init2 (so A_{S,k} = 0).  The chunk totals E2
// (a copy of the fold's output) are swept up right-anchored, the prefixes
// swept down from the seed, and each chunk walks its steps:
//   x*_k = (I + C_k S_k)^{-1} (b_k + C_k v_k)   (eq. lqt_method_2),
//   u*_k = d_k - K_k x*_k, then P <- P (x) a_k.
template <int N, int M>
struct M2Smem {  // P | step | scratch (combine, and the state solve)
    static constexpr int P = 0;
    static constexpr int SB = LElem<N>::SIZE;
    static constexpr int SCR_OFF = SB + StepLayout<N, M>::SIZE;
    static constexpr int SCR = combine_scratch<N>() > load_scratch<N, M>() ? combine_scratch<N>()
                                                                          : load_scratch<N, M>();
    static constexpr int SIZE = SCR_OFF + SCR;
};

// an element between global memory (GElem) and shared memory (LElem)
template <int N, typename A, typename B>
__device__ __forceinline__ void elem_in(A* dst, const B* src, int lr) {
    using E = LElem<N>;
    using G = GElem<N>;
    for (int t = lr; t < N * N; t += N) {
        const int i = t / N, j = t % N;
        dst[E::OA + i * E::LD + j] = static_cast<A>(src[G::OA + i * G::LD + j]);
        dst[E::OC + i * E::LD + j] = static_cast<A>(src[G::OC + i * G::LD + j]);
        dst[E::OJ + i * E::LD + j] = static_cast<A>(src[G::OJ + i * G::LD + j]);
    }
    dst[E::OB + lr] = static_cast<A>(src[G::OB + lr]);
    dst[E::OE + lr] = static_cast<A>(src[G::OE + lr]);
}
template <int N, typename A, typename B>
__device__ __forceinline__ void elem_out(A* dst, const B* src, int lr) {
    using E = LElem<N>;
    using G = GElem<N>;
    for (int t = lr; t < N * N; t += N) {
        const int i = t / N, j = t % N;
        dst[G::OA + i * G::LD + j] = src[E::OA + i * E::LD + j];
        dst[G::OC + i * G::LD + j] = src[E::OC + i * E::LD + j];
        dst[G::OJ + i * G::LD + j] = src[E::OJ + i * E::LD + j];
    }
    dst[G::OB + lr] = src[E::OB + lr];
    dst[G::OE + lr] = src[E::OE + lr];
}

// up-sweep level h: E2[j] <- E2[j - h] (x) E2[j], j = 2h q + 2h - 1
template <typename RT, int N, int NG>
__global__ void __launch_bounds__(NG* N) k_m2up(RT* E2, long long active, int h, int* status) {
    using E = LElem<N>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    RT* sh = reinterpret_cast<RT*>(smem_raw);
    const Group<N> g;
    const int gi = threadIdx.x / N;
    const long long j = ((long long)blockIdx.x * NG + gi) * 2 * h + 2 * h - 1;
    if (j >= active) return;
    RT* e1 = sh + gi * gstride<N>(UpSmem<N>::SIZE);
    RT* e2 = e1 + E::SIZE;
    RT* scr = e2 + E::SIZE;
    elem_in<N>(e1, E2 + (j - h) * GElem<N>::SIZE, g.lr);
    elem_in<N>(e2, E2 + j * GElem<N>::SIZE, g.lr);
    g.sync();
    const bool ok = combine<N, N>(e1, e2, e2, scr, g);
    elem_out<N>(E2 + j * GElem<N>::SIZE, e2, g.lr);
    flag(status, ok);
}

// the seed of each problem's prefix sweep: Pref[c0 + NC - 1] <- (0, x_0, 0, 0, 0)
template <typename R, typename RT, int N>
__global__ void __launch_bounds__(N) k_m2seed(const Item<R>* items, RT* Pref) {
    using E = GElem<N>;
    const Item<R>& it = items[blockIdx.x];
    RT* e = Pref + (it.c0 + it.NC - 1) * E::SIZE;
    const int r = threadIdx.x;
    for (int t = r; t < E::SIZE; t += N) e[t] = RT(0);
    __syncthreads();
    e[E::OB + r] = static_cast<RT>(it.D.x0[r]);
}

// down-sweep level h: Pref[j - h] <- Pref[j]; Pref[j] <- Pref[j] (x) E2[j - h]
template <typename RT, int N, int NG>
__global__ void __launch_bounds__(NG* N) k_m2down(const RT* E2, RT* Pref, long long active, int h,
                                                  int* status) {
    using E = LElem<N>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    RT* sh = reinterpret_cast<RT*>(smem_raw);
    const Group<N> g;
    const int gi = threadIdx.x / N;
    const long long j = ((long long)blockIdx.x * NG + gi) * 2 * h + 2 * h - 1;
    if (j >= active) return;
    RT* e1 = sh + gi * gstride<N>(UpSmem<N>::SIZE);
    RT* e2 = e1 + E::SIZE;
    RT* scr = e2 + E::SIZE;
    elem_in<N>(e1, Pref + j * GElem<N>::SIZE, g.lr);
    elem_in<N>(e2, E2 + (j - h) * GElem<N>::SIZE, g.lr);
    for (int t = g.lr; t < GElem<N>::SIZE; t += N)
        Pref[(j - h) * GElem<N>::SIZE + t] = Pref[j * GElem<N>::SIZE + t];
    g.sync();
    const bool ok = combine<N, N>(e1, e2, e1, scr, g);
    elem_out<N>(Pref + j * GElem<N>::SIZE, e1, g.lr);
    flag(status, ok);
}

// x = (I + C S)^{-1} (b + C v) for the prefix P and the value (S_k, v_k) of
// step k (read from the outputs); writes x into xo (N values in shared memory)
template <typename R, int N>
__device__ bool m2_state(const R* P, const R* S, const R* v, R* xo, R* scr, const Group<N>& g) {
    using E = LElem<N>;
    constexpr int LD = E::LD;
    R* Mx = scr;          // N x LD
    R* w = Mx + N * LD;   // N (right side, stride 1)
    const int r = g.lr;
    {
        R acc[N];
        R t = P[E::OB + r];
#pragma unroll
        for (int j = 0; j < N; ++j) acc[j] = r == j ? R(1) : R(0);
#pragma unroll 4
        for (int k = 0; k < N; ++k) {
            const R ck = P[E::OC + r * LD + k];
#pragma unroll
            for (int j = 0; j < N; ++j) acc[j] += ck * S[k * N + j];
            t += ck * v[k];
        }
#pragma unroll
        for (int j = 0; j < N; ++j) Mx[r * LD + j] = acc[j];
        w[r] = t;
    }
    g.sync();
    const bool ok = solve_gj<N, N, 1>(Mx, LD, w, 1, g);
    xo[r] = w[r];
    g.sync();
    return ok;
}

template <typename R, typename RT, int N, int M, int NG>
__global__ void __launch_bounds__(NG* N) k_m2roll(Args<R, RT> a, const RT* Pref) {
    using S = M2Smem<N, M>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    R* sh = reinterpret_cast<R*>(smem_raw);
    const Group<N> g;
    const int gi = threadIdx.x / N;
    const long long c = (long long)blockIdx.x * NG + gi;
    if (c >= a.C) return;
    const Item<R>& it = a.items[find_chunk(a.items, a.count, c)];
    const DescT<R>& D = it.D;
    R* gs = sh + gi * gstride<N>(S::SIZE);
    R* P = gs + S::P;
    R* sb = gs + S::SB;
    R* scr = gs + S::SCR_OFF;
    const int r = g.lr;
    const long long T = D.T;
    const long long lc = c - it.c0;
    const long long s0 = lc * it.B < T ? lc * it.B : T;
    const long long e0 = s0 + it.B < T ? s0 + it.B : T;
    elem_in<N>(P, Pref + c * GElem<N>::SIZE, r);
    g.sync();
    bool ok = true;
    R* xs = scr + combine_scratch<N>() - N;  // the state (end of the scratch)
    for (long long k = s0; k < e0; ++k) {
        ok &= m2_state<R, N>(P, D.S + k * N * N, D.v + k * N, xs, scr, g);
        const R xr = xs[r];
        D.x[k * N + r] = a.refine_add ? D.x[k * N + r] + xr : xr;
        if (r < M) {
            R t = D.u[k * M + r];
#pragma unroll 8
            for (int j = 0; j < N; ++j) t -= D.K[k * M * N + r * N + j] * xs[j];
            if (a.refine_add)
                it.u_out[k * M + r] = it.u_out[k * M + r] + (t - it.qh[k * M + r]);
            else
                D.u[k * M + r] = t;
        }
        g.sync();
        // P <- P (x) a_k
        load_step<R, N, M, true>(D, k, sb, scr, g, ok);
        ok &= combine<N, N>(P, sb + StepLayout<N, M>::E, P, scr, g);
        if (k == T - 1) {
            ok &= m2_state<R, N>(P, D.S + T * N * N, D.v + T * N, xs, scr, g);
            D.x[T * N + r] = a.refine_add ? D.x[T * N + r] + xs[r] : xs[r];
            g.sync();
        }
    }
    flag(a.status, ok);
}

// ---- KKT residuals of the first pass's iterate (refinement) -----------------
// One group per step k = 0..T (k = T: the terminal condition and x'_0 = 0).
// The residuals are small differences of large terms, so every sum runs in
// twice the working precision: FP64 arithmetic for FP64 problems, and for FP32
// problems the compensated dot product of lqt_refine.cuh on the FP32 pipe
// (GB300's FP64 rate is 1/64 of FP32).  Products of FP32 inputs are exact in
// either form; the intermediate vectors H x^ - r and X (H x^ - r) are carried
// as (hi, lo) pairs.
template <typename R>
struct XAcc;

template <>
struct XAcc<double> {
    double s;
    __device__ XAcc() : s(0.0) {}
    __device__ explicit XAcc(double a) : s(a) {}
    __device__ void add(double a) { s += a; }
    __device__ void add_prod(double a, double b) { s = fma(a, b, s); }
    __device__ void add_prod2(double a, double bh, double bl) { s = fma(a, bh + bl, s); }
    __device__ void split(double& h, double& l) const {
        h = s;
        l = 0.0;
    }
    __device__ double value() const { return s; }
};

template <>
struct XAcc<float> {
    Dot2<float> d;
    __device__ XAcc() : d(0.0f) {}
    __device__ explicit XAcc(float a) : d(a) {}
    __device__ void add(float a) { d.add(a); }
    __device__ void add_prod(float a, float b) { d.add_prod(a, b); }
    // a (bh + bl) with bl below the rounding of bh: the small product joins
    // the compensation term
    __device__ void add_prod2(float a, float bh, float bl) {
        d.add_prod(a, bh);
        d.c = fma_rn(a, bl, d.c);
    }
    __device__ void split(float& h, float& l) const {  // h + l = s + c, |l| <= ulp(h) / 2
        h = add_rn(d.s, d.c);
        l = sub_rn(d.c, sub_rn(h, d.s));
    }
    __device__ float value() const { return d.value(); }
};

template <int N, int M>
struct ResidSmem {  // work vectors and the step's matrices (odd row strides), type R
    static constexpr int PMAX = 2 * N;
    static constexpr int XK = 0, XK1 = N, UK = 2 * N, L0 = 2 * N + M, L1 = 3 * N + M,
                         HXH = 4 * N + M, HXL = HXH + PMAX, YH = HXL + PMAX, YL = YH + PMAX,
                         UM = YL + PMAX, RH = UM + M * lds(M), VEC = RH + M;
    // S_k, S_{k+1}, F_k (N x lds(N)), L_k (N x lds(M)), U_k (M x lds(M))
    static constexpr int SK = VEC, SK1 = SK + N * lds(N), FK = SK1 + N * lds(N),
                         LK = FK + N * lds(N), UKM = LK + N * lds(M), SIZE = UKM + M * lds(M);
    template <typename R>
    static constexpr int bytes() {
        return gstride<N>(SIZE) * (int)sizeof(R);
    }
};

template <typename R, int N, int M, int NG>
__global__ void __launch_bounds__(NG* N) k_cresid(const Item<R>* items1, const Item<R>* items2,
                                                  int count, long long rows, int* status) {
    using S = ResidSmem<N, M>;
    using X = XAcc<R>;
    constexpr int LD = lds(N), LM = lds(M);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Group<N> g;
    const int gi = threadIdx.x / N;
    const int r = g.lr;
    R* sh = reinterpret_cast<R*>(smem_raw + (size_t)gi * S::template bytes<R>());
    R* xk = sh + S::XK;
    R* xk1 = sh + S::XK1;
    R* uk = sh + S::UK;
    R* lam0 = sh + S::L0;
    R* lam1 = sh + S::L1;
    R* hxh = sh + S::HXH;
    R* hxl = sh + S::HXL;
    R* yh = sh + S::YH;
    R* yl = sh + S::YL;
    R* Um = sh + S::UM;
    R* rh = sh + S::RH;
    R* Sk = sh + S::SK;
    R* Sk1 = sh + S::SK1;
    R* Fs = sh + S::FK;
    R* Ls = sh + S::LK;
    R* Us = sh + S::UKM;
    const long long stride = (long long)gridDim.x * NG;
    bool ok = true;
    for (long long q = (long long)blockIdx.x * NG + gi; q < rows; q += stride) {
        const int ii = find_row(items1, count, q);
        const DescT<R>& D = items1[ii].D;
        const DescT<R>& D2 = items2[ii].D;
        const long long k = q - items1[ii].r0;
        const long long T = D.T;
        const bool term = k == T;
        const int p = term ? D.pT : D.p;
        const R* H = term ? D.HT : D.H + k * D.sH;
        const R* Xm = term ? D.XT : D.X + k * D.sX;
        const R* rr = term ? D.rT : (D.r ? D.r + k * D.sr : nullptr);
        // the step's matrices by coalesced asynchronous copies
#pragma unroll 8
        for (int t = r; t < N * N; t += N) cp_async<sizeof(R)>(Sk + (t / N) * LD + t % N, D.S + k * N * N + t);
        if (!term) {
#pragma unroll 8
            for (int t = r; t < N * N; t += N)
                cp_async<sizeof(R)>(Sk1 + (t / N) * LD + t % N, D.S + (k + 1) * N * N + t);
#pragma unroll 8
            for (int t = r; t < N * N; t += N)
                cp_async<sizeof(R)>(Fs + (t / N) * LD + t % N, D.F + k * D.sF + t);
#pragma unroll 4
            for (int t = r; t < N * M; t += N)
                cp_async<sizeof(R)>(Ls + (t / M) * LM + t % M, D.L + k * D.sL + t);
#pragma unroll 4
            for (int t = r; t < M * M; t += N)
                cp_async<sizeof(R)>(Us + (t / M) * LM + t % M, D.U + k * D.sU + t);
        }
        cp_async_commit();
        xk[r] = D.x[k * N + r];
        if (!term) {
            xk1[r] = D.x[(k + 1) * N + r];
            if (r < M) uk[r] = D.u[k * M + r];
        }
        cp_async_wait<0>();
        g.sync();
        // the iterate's multipliers lambda^_k = S_k x^_k - v_k in the working
        // precision R: the refinement needs exact residuals of some iterate,
        // and these R values enter the products below exactly
        {
            R t = -D.v[k * N + r];
#pragma unroll 8
            for (int j = 0; j < N; ++j) t += Sk[r * LD + j] * xk[j];
            lam0[r] = t;
            if (!term) {
                R t1 = -D.v[(k + 1) * N + r];
#pragma unroll 8
                for (int j = 0; j < N; ++j) t1 += Sk1[r * LD + j] * xk1[j];
                lam1[r] = t1;
            }
        }
        // H x^ - r (H = I: x^ - r), as (hi, lo)
        const bool hid = D.sH == 0 && p == N && !term && h_is_identity(D, g);
        if (hid) {
            X h(xk[r]);
            if (rr) h.add(-rr[r]);
            h.split(hxh[r], hxl[r]);
        } else {
            for (int i = r; i < p; i += N) {
                X h(rr ? -rr[i] : R(0));
                for (int j = 0; j < N; ++j) h.add_prod(H[i * N + j], xk[j]);
                h.split(hxh[i], hxl[i]);
            }
        }
        g.sync();
        // y = X (H x^ - r), as (hi, lo)
        for (int i = r; i < p; i += N) {
            X t(R(0));
            for (int b = 0; b < p; ++b) t.add_prod2(Xm[i * p + b], hxh[b], hxl[b]);
            t.split(yh[i], yl[i]);
        }
        g.sync();
        // g = H^T X (H x^ - r) - lambda^_k (+ F^T lambda^_{k+1})
        X gr(-lam0[r]);
        if (hid) {
            gr.add(yh[r]);
            gr.add(yl[r]);
        } else {
            for (int i = 0; i < p; ++i) gr.add_prod2(H[i * N + r], yh[i], yl[i]);
        }
        if (term) {
            const_cast<R*>(D2.etaT)[r] = -gr.value();
            const_cast<R*>(D2.x0)[r] = R(0);
            g.sync();
            continue;
        }
        for (int j = 0; j < N; ++j) gr.add_prod(Fs[j * LD + r], lam1[j]);
        // e = F x^ + c + L u^ - x^_{k+1}
        X e(D.c ? D.c[k * D.sc + r] : R(0));
        e.add(-xk1[r]);
        for (int j = 0; j < N; ++j) e.add_prod(Fs[r * LD + j], xk[j]);
        for (int b = 0; b < M; ++b) e.add_prod(Ls[r * LM + b], uk[b]);
        // h = U u^ + L^T lambda^_{k+1}; U^{-1} h in the working precision (h is
        // the residual itself, so its rounding is relative to h)
        if (r < M) {
            X h(R(0));
            for (int b = 0; b < M; ++b) {
                const R ub = Us[r * LM + b];
                Um[r * LM + b] = ub;
                h.add_prod(ub, uk[b]);
            }
            for (int j = 0; j < N; ++j) h.add_prod(Ls[j * LM + r], lam1[j]);
            rh[r] = h.value();
        }
        g.sync();
        ok &= solve_spd<N, M, 1>(Um, LM, rh, 1, g);
        for (int b = 0; b < M; ++b) e.add_prod(-Ls[r * LM + b], rh[b]);
        const_cast<R*>(D2.eta)[k * N + r] = -gr.value();
        const_cast<R*>(D2.c)[k * N + r] = e.value();
        if (r < M) const_cast<R*>(items2[ii].qh)[k * M + r] = rh[r];
        g.sync();
    }
    flag(status, ok);
}

// ---- Newton step of the Riccati recursion (refinement of S, v and K) -------
// At the first pass's (S^, v^) the Riccati map of Sec. II-B has residuals
//   R_k = Ric_k(S^_{k+1}) - S^_k,  rho_k = Vrec_k(S^_{k+1}, v^_{k+1}) - v^_k,
//   R_T = H_T^T X_T H_T - S^_T,    rho_T = H_T^T X_T r_T - v^_T,
// and its derivative at S^ is dS -> Phi_k^T dS Phi_k with the closed loop
// Phi_k = F_k - L_k K_k (and dv -> Phi_k^T (dv - dS ct_k), ct_k = c_k + L_k d_k).
// The Newton correction (dS, dv) therefore follows
//   dS_k = Phi_k^T dS_{k+1} Phi_k + R_k,  dv_k = Phi_k^T (dv_{k+1} - dS_{k+1} ct_k) + rho_k,
// which is the value recursion of the same operator for step elements with
// A = Phi_k, b = ct_k, C = 0, J = R_k, eta = rho_k: the pipeline solves it as the
// LQT problem F = Phi, c = ct, L = 0, U = I, H = I, X_k = R_k, eta_k = rho_k.
// k_nresid forms that problem (FP64 arithmetic, stored in R); k_ngains
// recomputes K_k in FP64 from S^_{k+1} + dS_{k+1}; k_nadd adds the corrections.
template <int N, int M>
struct NewtonSmem {  // double: val | step | riccati scratch | Kd | Ft
    static constexpr int VAL = 0;
    static constexpr int SB = LValue<N>::SIZE;
    static constexpr int SCR = SB + StepLayout<N, M>::SIZE;
    static constexpr int KD = SCR + riccati_scratch<N, M>();
    static constexpr int FT = KD + M * kd_ld<N>();
    static constexpr int SIZE = FT + LAffine<N>::SIZE;
};

template <typename R, int N, int M, int NG>
__global__ void __launch_bounds__(NG* N) k_nresid(const Item<R>* items1, const Item<R>* items3,
                                                  int count, long long rows, int* status) {
    using S = NewtonSmem<N, M>;
    using V = LValue<N>;
    using A = LAffine<N>;
    using D64 = double;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Group<N> g;
    const int gi = threadIdx.x / N;
    const int r = g.lr;
    D64* sh = reinterpret_cast<D64*>(smem_raw) + gi * gstride<N>(S::SIZE);
    D64* val = sh + S::VAL;
    D64* sb = sh + S::SB;
    D64* scr = sh + S::SCR;
    D64* Kd = sh + S::KD;
    D64* Ft = sh + S::FT;
    const long long stride = (long long)gridDim.x * NG;
    bool ok = true;
    for (long long q = (long long)blockIdx.x * NG + gi; q < rows; q += stride) {
        const int ii = find_row(items1, count, q);
        const DescT<R>& D = items1[ii].D;
        const DescT<R>& D3 = items3[ii].D;
        const long long k = q - items1[ii].r0;
        const long long T = D.T;
        R* Rk = const_cast<R*>(D3.X) + k * N * N;
        if (k == T) {
            D64 acc[N];
            D64 t = 0.0;
#pragma unroll
            for (int j = 0; j < N; ++j) acc[j] = 0.0;
            for (int i = 0; i < D.pT; ++i) {
                const D64 hi = static_cast<D64>(D.HT[i * N + r]);
                for (int b = 0; b < D.pT; ++b) {
                    const D64 hx = hi * static_cast<D64>(D.XT[i * D.pT + b]);
#pragma unroll
                    for (int j = 0; j < N; ++j) acc[j] += hx * static_cast<D64>(D.HT[b * N + j]);
                    if (D.rT) t += hx * static_cast<D64>(D.rT[b]);
                }
            }
#pragma unroll
            for (int j = 0; j < N; ++j)
                Rk[r * N + j] = static_cast<R>(acc[j] - static_cast<D64>(D.S[T * N * N + r * N + j]));
            const_cast<R*>(D3.etaT)[r] = static_cast<R>(t - static_cast<D64>(D.v[T * N + r]));
            continue;
        }
        load_step<D64, N, M, false, R>(D, k, sb, scr, g, ok);
        for (int i = r; i < N * N; i += N)
            val[V::OS + (i / N) * V::LD + i % N] = static_cast<D64>(D.S[(k + 1) * N * N + i]);
        copy_in(val + V::OV, D.v + (k + 1) * N, N, r, N);
        g.sync();
        ok &= riccati<D64, N, M>(val, sb, Kd, Ft, scr, g);
#pragma unroll 8
        for (int i = 0; i < N; ++i) {  // coalesced: lane r writes column r
            Rk[i * N + r] = static_cast<R>(val[V::OS + i * V::LD + r] -
                                           static_cast<D64>(D.S[k * N * N + i * N + r]));
            const_cast<R*>(D3.F)[k * N * N + i * N + r] = static_cast<R>(Ft[A::OF + i * A::LD + r]);
        }
        const_cast<R*>(D3.eta)[k * N + r] =
            static_cast<R>(val[V::OV + r] - static_cast<D64>(D.v[k * N + r]));
        const_cast<R*>(D3.c)[k * N + r] = static_cast<R>(Ft[A::OC + r]);
        g.sync();
    }
    flag(status, ok);
}

// K_k from S_{k+1} = S^_{k+1} + dS_{k+1}, v_{k+1} = v^_{k+1} + dv_{k+1} (FP64).
template <typename R, int N, int M, int NG>
__global__ void __launch_bounds__(NG* N) k_ngains(const Item<R>* items1, const Item<R>* items3,
                                                  int count, long long rows, int* status) {
    using S = NewtonSmem<N, M>;
    using V = LValue<N>;
    using D64 = double;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Group<N> g;
    const int gi = threadIdx.x / N;
    const int r = g.lr;
    D64* sh = reinterpret_cast<D64*>(smem_raw) + gi * gstride<N>(S::SIZE);
    D64* val = sh + S::VAL;
    D64* sb = sh + S::SB;
    D64* scr = sh + S::SCR;
    D64* Kd = sh + S::KD;
    const long long stride = (long long)gridDim.x * NG;
    bool ok = true;
    for (long long q = (long long)blockIdx.x * NG + gi; q < rows; q += stride) {
        const int ii = find_row(items1, count, q);
        const DescT<R>& D = items1[ii].D;
        const DescT<R>& D3 = items3[ii].D;
        const long long k = q - items1[ii].r0;
        if (k == D.T) continue;
        load_step<D64, N, M, false, R, false>(D, k, sb, scr, g, ok);
        const R* S1 = D.S + (k + 1) * N * N;
        const R* dS1 = D3.S + (k + 1) * N * N;
        for (int i = r; i < N * N; i += N)
            val[V::OS + (i / N) * V::LD + i % N] = static_cast<D64>(S1[i]) + static_cast<D64>(dS1[i]);
        val[V::OV + r] = static_cast<D64>(D.v[(k + 1) * N + r]) +
                         static_cast<D64>(D3.v[(k + 1) * N + r]);
        g.sync();
        ok &= gains<D64, N, M>(val, sb, Kd, scr, g);
#pragma unroll 8
        for (int i = 0; i < M; ++i) D.K[k * M * N + i * N + r] = static_cast<R>(Kd[i * kd_ld<N>() + r]);
        g.sync();
    }
    flag(status, ok);
}

// ---- the Newton step in compensated FP32 (FP32 problems) -------------------
// The same residuals and gains as k_nresid / k_ngains, with every sum in twice
// the working precision on the FP32 pipe (XAcc<float>).  The residual of the
// Riccati map is evaluated in its symmetric form around the first pass's FP32
// gain K~ (which the pass wrote into the K output):
//   (F - L K~)^T S (F - L K~) + K~^T U K~ + Q
//     = F^T S F - K~^T W - W^T K~ + K~^T G K~ + Q = Ric(S) + (K~ - K)^T G (K~ - K),
//   W = L^T S F, G = L^T S L + U, K = G^{-1} W,
// so the error of K~ enters only to second order; likewise for the vector
// recursion with e = v - S c, w = L^T e, d~ = G^{-1} w (FP32):
//   F^T e - K~^T w - W^T d~ + K~^T G d~ + q = Vrec(S, v) + (K~ - K)^T G (d - d~).
// The gains at S^ + dS take one step of iterative refinement of G K = W from
// K~, with the residual W - G K~ in twice the working precision.
// Row a of L^T Y (+ Z row a), Y = (Yh, Yl) N x C in shared memory (stride ldy):
// out[c] = sum_j L[j][a] Y[j][c], CH independent compensated accumulators at a
// time (each sum is a serial chain, so several run side by side).
template <int N, int M, int CH>
__device__ __forceinline__ void lt_times_x(const float* L, int a, const float* Yh,
                                           const float* Yl, int ldy, int C, float* outh,
                                           float* outl, const float* init = nullptr) {
    using X = XAcc<float>;
    for (int c0 = 0; c0 < C; c0 += CH) {
        X t[CH];
#pragma unroll
        for (int cc = 0; cc < CH; ++cc)
            if (init) t[cc].add(init[c0 + cc]);
        for (int j = 0; j < N; ++j) {
            const float l = L[j * M + a];
#pragma unroll
            for (int cc = 0; cc < CH; ++cc) t[cc].add_prod2(l, Yh[j * ldy + c0 + cc], Yl[j * ldy + c0 + cc]);
        }
#pragma unroll
        for (int cc = 0; cc < CH; ++cc) t[cc].split(outh[c0 + cc], outl[c0 + cc]);
    }
}

template <int N, int M>
struct NewtonCSmem {  // float: (hi, lo) intermediates, odd row strides
    static constexpr int LD = lds(N), LM = lds(M), PMAX = 2 * N;
    static constexpr int SFH = 0, SFL = SFH + N * LD, SLH = SFL + N * LD, SLL = SLH + N * LM,
                         WH = SLL + N * LM, WL = WH + M * LD, GH = WL + M * LD, GL = GH + M * LM,
                         GKH = GL + M * LM, GKL = GKH + M * LD, XHH = GKL + M * LD,
                         XHL = XHH + PMAX * LD, RR = XHL + PMAX * LD, EH = RR + N * LD,
                         EL = EH + N, WVH = EL + N, WVL = WVH + M, DD = WVL + M, GDH = DD + M,
                         GDL = GDH + M, XRH = GDL + M, XRL = XRH + PMAX, SIZE = XRL + PMAX;
};

template <int N, int M, int NG>
__global__ void __launch_bounds__(NG* N) k_nresid_c(const Item<float>* items1,
                                                    const Item<float>* items3, int count,
                                                    long long rows, int* status) {
    using S = NewtonCSmem<N, M>;
    using X = XAcc<float>;
    constexpr int LD = S::LD, LM = S::LM, NCH = N < 8 ? N : 8, MCH = M < 8 ? M : 8;
    static_assert(N % NCH == 0 && M % MCH == 0, "column chunks");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Group<N> g;
    const int gi = threadIdx.x / N;
    const int r = g.lr;
    float* sh = reinterpret_cast<float*>(smem_raw) + gi * gstride<N>(S::SIZE);
    float *SFh = sh + S::SFH, *SFl = sh + S::SFL, *SLh = sh + S::SLH, *SLl = sh + S::SLL;
    float *Wh = sh + S::WH, *Wl = sh + S::WL, *Gh = sh + S::GH, *Gl = sh + S::GL;
    float *GKh = sh + S::GKH, *GKl = sh + S::GKL, *XHh = sh + S::XHH, *XHl = sh + S::XHL;
    float *RR = sh + S::RR, *eh = sh + S::EH, *el = sh + S::EL, *wvh = sh + S::WVH;
    float *wvl = sh + S::WVL, *dd = sh + S::DD, *gdh = sh + S::GDH, *gdl = sh + S::GDL;
    float *xrh = sh + S::XRH, *xrl = sh + S::XRL;
    const long long stride = (long long)gridDim.x * NG;
    bool ok = true;
    for (long long q = (long long)blockIdx.x * NG + gi; q < rows; q += stride) {
        const int ii = find_row(items1, count, q);
        const DescT<float>& D = items1[ii].D;
        const DescT<float>& D3 = items3[ii].D;
        const long long k = q - items1[ii].r0;
        const long long T = D.T;
        float* Rk = const_cast<float*>(D3.X) + k * N * N;
        if (k == T) {
            // R_T = H_T^T X_T H_T - S^_T, rho_T = H_T^T X_T r_T - v^_T
            const int pT = D.pT;
            for (int i = r; i < pT; i += N) {
                for (int c = 0; c < N; ++c) {
                    X t(0.0f);
                    for (int b = 0; b < pT; ++b) t.add_prod(D.XT[i * pT + b], D.HT[b * N + c]);
                    t.split(XHh[i * LD + c], XHl[i * LD + c]);
                }
                X t(0.0f);
                if (D.rT)
                    for (int b = 0; b < pT; ++b) t.add_prod(D.XT[i * pT + b], D.rT[b]);
                t.split(xrh[i], xrl[i]);
            }
            g.sync();
            for (int c = 0; c < N; ++c) {
                X t(-D.S[T * N * N + r * N + c]);
                for (int i = 0; i < pT; ++i) t.add_prod2(D.HT[i * N + r], XHh[i * LD + c], XHl[i * LD + c]);
                RR[r * LD + c] = t.value();
            }
            X rho(-D.v[T * N + r]);
            for (int i = 0; i < pT; ++i) rho.add_prod2(D.HT[i * N + r], xrh[i], xrl[i]);
            g.sync();
#pragma unroll 8
            for (int i = 0; i < N; ++i) Rk[i * N + r] = 0.5f * (RR[i * LD + r] + RR[r * LD + i]);
            const_cast<float*>(D3.etaT)[r] = rho.value();
            g.sync();
            continue;
        }
        const float* F = D.F + k * D.sF;
        const float* L = D.L + k * D.sL;
        const float* U = D.U + k * D.sU;
        const float* c = D.c ? D.c + k * D.sc : nullptr;
        const float* S1 = D.S + (k + 1) * N * N;
        const float* Sk = D.S + k * N * N;
        const float* Kt = D.K + k * M * N;
        const int p = D.p;
        const float* H = D.H ? D.H + k * D.sH : nullptr;
        const float* Xm = D.X ? D.X + k * D.sX : nullptr;
        const float* rr = D.r ? D.r + k * D.sr : nullptr;
        const bool hid = D.sH == 0 && p == N && h_is_identity(D, g);
        // S F and S L (row r), e = v - S c, and X H, X r
        for (int c0 = 0; c0 < N; c0 += NCH) {
            X t[NCH];
            for (int j = 0; j < N; ++j) {
                const float sj = S1[r * N + j];
#pragma unroll
                for (int cc = 0; cc < NCH; ++cc) t[cc].add_prod(sj, F[j * N + c0 + cc]);
            }
#pragma unroll
            for (int cc = 0; cc < NCH; ++cc) t[cc].split(SFh[r * LD + c0 + cc], SFl[r * LD + c0 + cc]);
        }
        for (int a0 = 0; a0 < M; a0 += MCH) {
            X t[MCH];
            for (int j = 0; j < N; ++j) {
                const float sj = S1[r * N + j];
#pragma unroll
                for (int aa = 0; aa < MCH; ++aa) t[aa].add_prod(sj, L[j * M + a0 + aa]);
            }
#pragma unroll
            for (int aa = 0; aa < MCH; ++aa) t[aa].split(SLh[r * LM + a0 + aa], SLl[r * LM + a0 + aa]);
        }
        {
            X e(D.v[(k + 1) * N + r]);
            if (c)
                for (int j = 0; j < N; ++j) e.add_prod(-S1[r * N + j], c[j]);
            e.split(eh[r], el[r]);
        }
        if (hid) {
            X t(0.0f);
            if (rr)
                for (int b = 0; b < N; ++b) t.add_prod(Xm[r * N + b], rr[b]);
            t.split(xrh[r], xrl[r]);
        } else {
            for (int i = r; i < p; i += N) {
                for (int cl = 0; cl < N; ++cl) {
                    X t(0.0f);
                    for (int b = 0; b < p; ++b) t.add_prod(Xm[i * p + b], H[b * N + cl]);
                    t.split(XHh[i * LD + cl], XHl[i * LD + cl]);
                }
                X t(0.0f);
                if (rr)
                    for (int b = 0; b < p; ++b) t.add_prod(Xm[i * p + b], rr[b]);
                t.split(xrh[i], xrl[i]);
            }
        }
        g.sync();
        // W = L^T S F, G = L^T S L + U, w = L^T e (rows a = r < M)
        if (r < M) {
            lt_times_x<N, M, NCH>(L, r, SFh, SFl, LD, N, Wh + r * LD, Wl + r * LD);
            lt_times_x<N, M, MCH>(L, r, SLh, SLl, LM, M, Gh + r * LM, Gl + r * LM, U + r * M);
            X w(0.0f);
            for (int j = 0; j < N; ++j) w.add_prod2(L[j * M + r], eh[j], el[j]);
            w.split(wvh[r], wvl[r]);
            dd[r] = wvh[r] + wvl[r];
        }
        g.sync();
        // d~ = G^{-1} w in FP32; G K~ (rows a = r < M)
        ok &= solve_spd<N, M, 1>(Gh, LM, dd, 1, g);
        if (r < M)
            for (int c0 = 0; c0 < N; c0 += NCH) {
                X t[NCH];
                for (int b = 0; b < M; ++b) {
                    const float gh = Gh[r * LM + b], gl = Gl[r * LM + b];
#pragma unroll
                    for (int cc = 0; cc < NCH; ++cc) t[cc].add_prod2(Kt[b * N + c0 + cc], gh, gl);
                }
#pragma unroll
                for (int cc = 0; cc < NCH; ++cc) t[cc].split(GKh[r * LD + c0 + cc], GKl[r * LD + c0 + cc]);
            }
        if (r < M) {
            X t(0.0f);
            for (int b = 0; b < M; ++b) t.add_prod2(dd[b], Gh[r * LM + b], Gl[r * LM + b]);
            t.split(gdh[r], gdl[r]);
        }
        g.sync();
        // row r of R_k = F^T S F - K~^T W - W^T K~ + K~^T G K~ + Q - S^_k
        for (int c0 = 0; c0 < N; c0 += NCH) {
            X t[NCH];
#pragma unroll
            for (int cc = 0; cc < NCH; ++cc) {
                t[cc].add(-Sk[r * N + c0 + cc]);
                if (hid) t[cc].add(Xm[r * N + c0 + cc]);
            }
            for (int j = 0; j < N; ++j) {
                const float f = F[j * N + r];
#pragma unroll
                for (int cc = 0; cc < NCH; ++cc)
                    t[cc].add_prod2(f, SFh[j * LD + c0 + cc], SFl[j * LD + c0 + cc]);
            }
            for (int a = 0; a < M; ++a) {
                const float kr = Kt[a * N + r];
                const float wrh = Wh[a * LD + r], wrl = Wl[a * LD + r];
#pragma unroll
                for (int cc = 0; cc < NCH; ++cc) {
                    t[cc].add_prod2(-kr, Wh[a * LD + c0 + cc], Wl[a * LD + c0 + cc]);
                    t[cc].add_prod2(-Kt[a * N + c0 + cc], wrh, wrl);
                    t[cc].add_prod2(kr, GKh[a * LD + c0 + cc], GKl[a * LD + c0 + cc]);
                }
            }
            if (!hid)
                for (int i = 0; i < p; ++i) {
                    const float h = H[i * N + r];
#pragma unroll
                    for (int cc = 0; cc < NCH; ++cc)
                        t[cc].add_prod2(h, XHh[i * LD + c0 + cc], XHl[i * LD + c0 + cc]);
                }
#pragma unroll
            for (int cc = 0; cc < NCH; ++cc) RR[r * LD + c0 + cc] = t[cc].value();
        }
        // rho_k = F^T e - K~^T w - W^T d~ + K~^T G d~ + q - v^_k
        X rho(-D.v[k * N + r]);
        if (hid) {
            rho.add(xrh[r]);
            rho.add(xrl[r]);
        } else {
            for (int i = 0; i < p; ++i) rho.add_prod2(H[i * N + r], xrh[i], xrl[i]);
        }
        for (int j = 0; j < N; ++j) rho.add_prod2(F[j * N + r], eh[j], el[j]);
        for (int a = 0; a < M; ++a) {
            const float kr = Kt[a * N + r];
            rho.add_prod2(-kr, wvh[a], wvl[a]);
            rho.add_prod2(-dd[a], Wh[a * LD + r], Wl[a * LD + r]);
            rho.add_prod2(kr, gdh[a], gdl[a]);
        }
        g.sync();
        // symmetrised R_k, the closed loop Phi_k = F - L K~ and ct_k = c + L d~
        // (FP32: they enter the correction's dynamics, whose relative error is
        // then of the order of K~'s)
#pragma unroll 4
        for (int i = 0; i < N; ++i) {
            Rk[i * N + r] = 0.5f * (RR[i * LD + r] + RR[r * LD + i]);
            float f = F[i * N + r];
            for (int a = 0; a < M; ++a) f -= L[i * M + a] * Kt[a * N + r];
            const_cast<float*>(D3.F)[k * N * N + i * N + r] = f;
        }
        const_cast<float*>(D3.eta)[k * N + r] = rho.value();
        {
            float t = c ? c[r] : 0.0f;
            for (int a = 0; a < M; ++a) t += L[r * M + a] * dd[a];
            const_cast<float*>(D3.c)[k * N + r] = t;
        }
        g.sync();
    }
    flag(status, ok);
}

// K_k at S^_{k+1} + dS_{k+1}: one step of iterative refinement of G K = W from
// the first pass's K~, with S held as the (hi, lo) pair (S^, dS).
template <int N, int M>
struct NewtonGSmem {  // float: S F, S L, W, G as (hi, lo), and the residual Z
    static constexpr int LD = lds(N), LM = lds(M);
    static constexpr int SFH = 0, SFL = SFH + N * LD, SLH = SFL + N * LD, SLL = SLH + N * LM,
                         WH = SLL + N * LM, WL = WH + M * LD, GH = WL + M * LD, GL = GH + M * LM,
                         Z = GL + M * LM, SIZE = Z + M * LD;
};

template <int N, int M, int NG>
__global__ void __launch_bounds__(NG* N) k_ngains_c(const Item<float>* items1,
                                                    const Item<float>* items3, int count,
                                                    long long rows, int* status) {
    using S = NewtonGSmem<N, M>;
    using X = XAcc<float>;
    constexpr int LD = S::LD, LM = S::LM, NCH = N < 8 ? N : 8, MCH = M < 8 ? M : 8;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Group<N> g;
    const int gi = threadIdx.x / N;
    const int r = g.lr;
    float* sh = reinterpret_cast<float*>(smem_raw) + gi * gstride<N>(S::SIZE);
    float *SFh = sh + S::SFH, *SFl = sh + S::SFL, *SLh = sh + S::SLH, *SLl = sh + S::SLL;
    float *Wh = sh + S::WH, *Wl = sh + S::WL, *Gh = sh + S::GH, *Gl = sh + S::GL;
    float* Z = sh + S::Z;  // M x LD
    const long long stride = (long long)gridDim.x * NG;
    bool ok = true;
    for (long long q = (long long)blockIdx.x * NG + gi; q < rows; q += stride) {
        const int ii = find_row(items1, count, q);
        const DescT<float>& D = items1[ii].D;
        const DescT<float>& D3 = items3[ii].D;
        const long long k = q - items1[ii].r0;
        if (k == D.T) continue;
        const float* F = D.F + k * D.sF;
        const float* L = D.L + k * D.sL;
        const float* U = D.U + k * D.sU;
        const float* Sh = D.S + (k + 1) * N * N;
        const float* Sl = D3.S + (k + 1) * N * N;
        float* Kt = D.K + k * M * N;
        for (int c0 = 0; c0 < N; c0 += NCH) {
            X t[NCH];
            for (int j = 0; j < N; ++j) {
                const float sh_ = Sh[r * N + j], sl_ = Sl[r * N + j];
#pragma unroll
                for (int cc = 0; cc < NCH; ++cc) t[cc].add_prod2(F[j * N + c0 + cc], sh_, sl_);
            }
#pragma unroll
            for (int cc = 0; cc < NCH; ++cc) t[cc].split(SFh[r * LD + c0 + cc], SFl[r * LD + c0 + cc]);
        }
        for (int a0 = 0; a0 < M; a0 += MCH) {
            X t[MCH];
            for (int j = 0; j < N; ++j) {
                const float sh_ = Sh[r * N + j], sl_ = Sl[r * N + j];
#pragma unroll
                for (int aa = 0; aa < MCH; ++aa) t[aa].add_prod2(L[j * M + a0 + aa], sh_, sl_);
            }
#pragma unroll
            for (int aa = 0; aa < MCH; ++aa) t[aa].split(SLh[r * LM + a0 + aa], SLl[r * LM + a0 + aa]);
        }
        g.sync();
        if (r < M) {
            lt_times_x<N, M, NCH>(L, r, SFh, SFl, LD, N, Wh + r * LD, Wl + r * LD);
            lt_times_x<N, M, MCH>(L, r, SLh, SLl, LM, M, Gh + r * LM, Gl + r * LM, U + r * M);
        }
        g.sync();
        // Z = W - G K~ (rows a = r < M)
        if (r < M)
            for (int c0 = 0; c0 < N; c0 += NCH) {
                X t[NCH];
#pragma unroll
                for (int cc = 0; cc < NCH; ++cc) {
                    t[cc].add(Wh[r * LD + c0 + cc]);
                    t[cc].add(Wl[r * LD + c0 + cc]);
                }
                for (int b = 0; b < M; ++b) {
                    const float gh = Gh[r * LM + b], gl = Gl[r * LM + b];
#pragma unroll
                    for (int cc = 0; cc < NCH; ++cc) t[cc].add_prod2(-Kt[b * N + c0 + cc], gh, gl);
                }
#pragma unroll
                for (int cc = 0; cc < NCH; ++cc) Z[r * LD + c0 + cc] = t[cc].value();
            }
        g.sync();
        ok &= solve_spd<N, M, N>(Gh, LM, Z, LD, g);
#pragma unroll 4
        for (int a = 0; a < M; ++a) Kt[a * N + r] += Z[a * LD + r];
        g.sync();
    }
    flag(status, ok);
}

// S_k <- S^_k + dS_k, v_k <- v^_k + dv_k for every problem (one thread per value).
template <typename R, int N>
__global__ void k_nadd(const Item<R>* items1, const Item<R>* items3, int count, long long rows) {
    const long long per = (long long)N * N + N;
    const long long total = rows * per;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const long long q = t / per;
        const long long e = t - q * per;
        const int ii = find_row(items1, count, q);
        const DescT<R>& D = items1[ii].D;
        const DescT<R>& D3 = items3[ii].D;
        const long long k = q - items1[ii].r0;
        if (e < (long long)N * N) {
            const long long o = k * N * N + e;
            D.S[o] = static_cast<R>(static_cast<double>(D.S[o]) + static_cast<double>(D3.S[o]));
        } else {
            const long long o = k * N + (e - (long long)N * N);
            D.v[o] = static_cast<R>(static_cast<double>(D.v[o]) + static_cast<double>(D3.v[o]));
        }
    }
}

}  // namespace chain
}  // namespace lqt
