// Vector walks of the chunked pipeline at n = 8, 16, 32: the recursions that
// need no matrix product once S_k and K_k are known, one warp per chunk.
//
//   k_vfwd   the rollout of x*_k and u*_k from each chunk's start state
//            (eq. Control_LQT), or (MAP) a chunk's closed-loop offset gamma,
//   k_vback  the value vector v_k = Ft_k^T w_k + eta_k, w_k = v_{k+1} - S_{k+1} c_k,
//            Ft_k = F_k - L_k K_k (Sec. II-B) from v at the chunk's end with the
//            feedforward d_k = G_k^{-1} L_k^T w_k, or (MAP) a chunk's offset beta.
//
// The correction pass of the refinement (lqt_chain.cuh) has the matrices of the
// first pass, so it is these walks and two affine scans: the value maps are the
// transposes of the first pass's chunk maps, kept with the G_k^{-1} it formed.
//
// Bound: every step reads F, L, K (and S, G^{-1}) once, 8 to 13 KB at n = 32,
// against a few thousand FMAs.  A ring of cp.async stages keeps the next steps'
// matrices on the way; products read the ring by columns (x^T A) or by rows
// (A x), both conflict-free in the swizzled layout of lqt_team.cuh.  n = 32,
// T = 65536: k_vfwd 98 us for 0.55 GB (5.6 TB/s), k_vback 123 (map) and 135 us
// for 0.82 and 0.89 GB (6.6 TB/s); the correction pass made of them and the
// affine scans takes 0.58 ms, a full second pass 2.9.
#pragma once

#include "lqt_chain_args.cuh"
#include "lqt_team_chain.cuh"

namespace lqt {
namespace chain {

template <int N, int M>
struct VWalk {
    static constexpr int r4(int x) { return (x + 3) / 4 * 4; }
    // one stage of k_vfwd: F, L, K, c, d and (correction) x^, u^, U^{-1} h; of
    // k_vback: F, L, K, c, S_{k+1}, G^{-1}, eta
    static constexpr int F = 0, L = N * N, K = L + N * M, C = K + M * N, D = C + N, XH = D + M,
                         UH = XH + N, QH = UH + M, FWD = r4(QH + M), S = D, GI = S + N * N,
                         E = GI + M * M, BACK = r4(E + N);
    static constexpr int ST = N == 32 ? 3 : 4;   // stages
    static constexpr int NT = N == 32 ? 1 : 4;   // warps (chunks) per CTA
    static constexpr int VEC = 2 * N + 2 * M;    // w | y or x | u
    static constexpr int FWD_SIZE = ST * FWD + VEC, BACK_SIZE = ST * BACK + VEC;
};

// The warp's lanes as N columns (or rows) x G blocks, and as M x GM blocks.
template <int N, int M>
struct VLane {
    static constexpr int G = 32 / N, GM = 32 / M;
    static constexpr int BN = N / G;                    // rows of N per block
    static constexpr int BNM = N / GM;                  // rows of N per block of M lanes
    static constexpr int BM = M / G > 0 ? M / G : 1;    // rows of M per block
    static constexpr int BMM = M / GM > 0 ? M / GM : 1; // rows of M per block of M lanes
    int lane, j, h, a, ha;
    __device__ __forceinline__ VLane() {
        lane = threadIdx.x & 31;
        j = lane % N;
        h = lane / N;
        a = lane % M;
        ha = lane / M;
    }
    template <typename R>
    __device__ __forceinline__ R sum_n(R x) const {  // over the blocks of N lanes
#pragma unroll
        for (int d = N; d < 32; d <<= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
        return x;
    }
    template <typename R>
    __device__ __forceinline__ R sum_m(R x) const {
#pragma unroll
        for (int d = M; d < 32; d <<= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
        return x;
    }
};

// sum_r A[r0 + r][col] x[r0 + r], r < ROWS (A swizzled with COLS columns)
template <int ROWS, int COLS, typename R>
__device__ __forceinline__ R col_dot(const R* A, const R* x, int r0, int col) {
    R t = R(0);
#pragma unroll
    for (int r = 0; r < ROWS; ++r) t = team::fma_(A[Sw<R, COLS>::at(r0 + r, col)], x[r0 + r], t);
    return t;
}
// sum_c A[row][c0 + c] x[c0 + c], c < CN
template <int CN, int COLS, typename R>
__device__ __forceinline__ R row_dot(const R* A, const R* x, int row, int c0) {
    constexpr int E = 16 / (int)sizeof(R), V = CN < E ? CN : E;
    R t = R(0);
#pragma unroll
    for (int c = 0; c < CN; c += V) {
        R v[V];
        ldrow<COLS, V>(A, row, c0 + c, v);
#pragma unroll
        for (int q = 0; q < V; ++q) t = team::fma_(v[q], x[c0 + c + q], t);
    }
    return t;
}

// ROWS x COLS dense global matrix into the swizzled layout, by one warp
template <int ROWS, int COLS, typename R>
__device__ __forceinline__ void warp_cp_mat(R* dst, const R* src, bool vec, int lane) {
    constexpr int E = 16 / (int)sizeof(R), RC = COLS / E;
    if (vec) {
#pragma unroll
        for (int t = lane; t < ROWS * RC; t += 32)
            cp_async_cg16(dst + Sw<R, COLS>::chunk(t / RC, t % RC), src + t * E);
    } else {
        for (int t = lane; t < ROWS * COLS; t += 32)
            cp_async<sizeof(R)>(dst + Sw<R, COLS>::at(t / COLS, t % COLS), src + t);
    }
}

// The chunk of a walk: its item and steps [s, e).
template <typename R>
struct VChunk {
    const Item<R>* it;
    long long lc, s, e, T;
    __device__ VChunk(const Item<R>* items, int count, long long c) {
        it = &items[find_chunk(items, count, c)];
        T = it->D.T;
        const long long B = it->B;
        lc = c - it->c0;
        s = lc * B < T ? lc * B : T;
        e = s + B < T ? s + B : T;
    }
};

// ---- forward ---------------------------------------------------------------
// MAP: x from 0; the map (Phi, gamma) of chunk c to FE[c], Phi from `maps`.
// Otherwise the outputs: x from X[c] (x_0 for a first chunk), u = d - K x.
template <typename R, typename RT, int N, int M, bool MAP>
__device__ __forceinline__ void b_vfwd(const Args<R, RT>& a, long long c, const RT* maps, R* sh) {
    using W = VWalk<N, M>;
    using VL = VLane<N, M>;
    const VL l;
    const VChunk<R> ch(a.items, a.count, c);
    const Item<R>& it = *ch.it;
    const DescT<R>& D = it.D;
    const R *F = D.F, *L = D.L, *K = D.K, *cp = D.c, *up = D.u, *uo = it.u_out, *qh = it.qh;
    const long long sF = D.sF, sL = D.sL, sc = D.sc;
    const bool vF = vec_ok(F, sF), vL = vec_ok(L, sL), vK = vec_ok(K, 0);
    R* xs = sh + W::ST * W::FWD;
    R* us = xs + N;
    R x = R(0);
    if (!MAP) x = ch.lc == 0 ? D.x0[l.j] : static_cast<R>(a.X[c * N + l.j]);
    if (l.h == 0) xs[l.j] = x;
    auto stage = [&](long long k) {
        if (k < ch.e) {
            R* b = sh + (int)((k - ch.s) % W::ST) * W::FWD;
            warp_cp_mat<N, N>(b + W::F, F + k * sF, vF, l.lane);
            warp_cp_mat<N, M>(b + W::L, L + k * sL, vL, l.lane);
            warp_cp_mat<M, N>(b + W::K, K + k * (M * N), vK, l.lane);
            if (cp && l.h == 0) cp_async<sizeof(R)>(b + W::C + l.j, cp + k * sc + l.j);
            if (l.ha == 0) cp_async<sizeof(R)>(b + W::D + l.a, up + k * M + l.a);
            if (!MAP && a.refine_add) {
                if (l.h == 0) cp_async<sizeof(R)>(b + W::XH + l.j, D.x + k * N + l.j);
                if (l.ha == 0) {
                    cp_async<sizeof(R)>(b + W::UH + l.a, uo + k * M + l.a);
                    cp_async<sizeof(R)>(b + W::QH + l.a, qh + k * M + l.a);
                }
            }
        }
        cp_async_commit();
    };
#pragma unroll
    for (int q = 0; q < W::ST - 1; ++q) stage(ch.s + q);
    for (long long k = ch.s; k < ch.e; ++k) {
        cp_async_wait<W::ST - 2>();
        __syncwarp();  // the stage is in, and the one to refill is read
        stage(k + W::ST - 1);
        const R* b = sh + (int)((k - ch.s) % W::ST) * W::FWD;
        if (!MAP && l.h == 0) D.x[k * N + l.j] = a.refine_add ? b[W::XH + l.j] + x : x;
        const R u = b[W::D + l.a] -
                    l.sum_m(row_dot<VL::BNM, N>(b + W::K, xs, l.a, l.ha * VL::BNM));
        if (l.ha == 0) {
            us[l.a] = u;
            if (!MAP) {
                if (a.refine_add)
                    it.u_out[k * M + l.a] = b[W::UH + l.a] + (u - b[W::QH + l.a]);
                else
                    D.u[k * M + l.a] = u;
            }
        }
        __syncwarp();
        R t = row_dot<VL::BN, N>(b + W::F, xs, l.j, l.h * VL::BN);
        if (l.h * VL::BM < M) t += row_dot<VL::BM, M>(b + W::L, us, l.j, l.h * VL::BM);
        x = l.sum_n(t) + (cp ? b[W::C + l.j] : R(0));
        __syncwarp();
        if (l.h == 0) {
            xs[l.j] = x;
            if (!MAP && k == ch.T - 1) D.x[ch.T * N + l.j] = a.refine_add ? D.x[ch.T * N + l.j] + x : x;
        }
    }
    cp_async_wait<0>();
    __syncwarp();
    if (MAP) {
        using A = DAffine<N>;
        RT* out = a.FE + c * A::SIZE;
        const RT* m = maps + c * A::SIZE;
        for (int t = l.lane; t < N * N; t += 32) out[A::OF + t] = m[A::OF + t];
        if (l.h == 0) out[A::OC + l.j] = static_cast<RT>(x);
    }
}

template <typename R, typename RT, int N, int M, bool MAP>
__global__ void __launch_bounds__(32 * VWalk<N, M>::NT) k_vfwd(Args<R, RT> a, const RT* maps) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using W = VWalk<N, M>;
    const int gi = threadIdx.x / 32;
    const long long c = (long long)blockIdx.x * W::NT + gi;
    if (c >= a.C) return;
    b_vfwd<R, RT, N, M, MAP>(a, c, maps, reinterpret_cast<R*>(smem_raw) + gi * W::FWD_SIZE);
}

// ---- backward (the correction problem: offsets c, linear terms eta) ---------
// MAP: v from 0; the map (Phi^T, beta) of chunk c at the mirrored slot of FE (so
// that the forward scan runs from the last chunk to the first).  Otherwise v
// from X at the mirrored slot, and the feedforward d_k to D.u.
template <typename R, typename RT, int N, int M, bool MAP>
__global__ void __launch_bounds__(32 * VWalk<N, M>::NT) k_vback(Args<R, RT> a, const RT* maps) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using W = VWalk<N, M>;
    using VL = VLane<N, M>;
    const int gi = threadIdx.x / 32;
    const long long c = (long long)blockIdx.x * W::NT + gi;
    if (c >= a.C) return;
    R* sh = reinterpret_cast<R*>(smem_raw) + gi * W::BACK_SIZE;
    const VL l;
    const VChunk<R> ch(a.items, a.count, c);
    const Item<R>& it = *ch.it;
    const DescT<R>& D = it.D;
    const R *F = D.F, *L = D.L, *K = D.K, *S = D.S, *cp = D.c, *ep = D.eta, *gp = it.gi;
    const long long sF = D.sF, sL = D.sL, sc = D.sc, se = D.seta;
    const bool vF = vec_ok(F, sF), vL = vec_ok(L, sL), vK = vec_ok(K, 0), vS = vec_ok(S, 0);
    const long long cr = it.c0 + (it.NC - 1 - ch.lc);
    R* ws = sh + W::ST * W::BACK;
    R* ys = ws + N;
    R v = MAP ? R(0) : static_cast<R>(a.X[cr * N + l.j]);
    auto stage = [&](long long k) {
        if (k >= ch.s) {
            R* b = sh + (int)((ch.e - 1 - k) % W::ST) * W::BACK;
            warp_cp_mat<N, N>(b + W::F, F + k * sF, vF, l.lane);
            warp_cp_mat<N, M>(b + W::L, L + k * sL, vL, l.lane);
            warp_cp_mat<M, N>(b + W::K, K + k * (M * N), vK, l.lane);
            warp_cp_mat<N, N>(b + W::S, S + (k + 1) * (N * N), vS, l.lane);
            if (!MAP) warp_cp_mat<M, M>(b + W::GI, gp + k * (M * M), true, l.lane);
            if (l.h == 0) {
                cp_async<sizeof(R)>(b + W::C + l.j, cp + k * sc + l.j);
                cp_async<sizeof(R)>(b + W::E + l.j, ep + k * se + l.j);
            }
        }
        cp_async_commit();
    };
#pragma unroll
    for (int q = 0; q < W::ST - 1; ++q) stage(ch.e - 1 - q);
    for (long long k = ch.e - 1; k >= ch.s; --k) {
        cp_async_wait<W::ST - 2>();
        __syncwarp();
        stage(k - (W::ST - 1));
        const R* b = sh + (int)((ch.e - 1 - k) % W::ST) * W::BACK;
        // w = v - S c (S symmetric: by columns)
        const R w = v - l.sum_n(col_dot<VL::BN, N>(b + W::S, b + W::C, l.h * VL::BN, l.j));
        if (l.h == 0) ws[l.j] = w;
        __syncwarp();
        R f = col_dot<VL::BN, N>(b + W::F, ws, l.h * VL::BN, l.j);
        const R y = l.sum_m(col_dot<VL::BNM, M>(b + W::L, ws, l.ha * VL::BNM, l.a));
        if (l.ha == 0) ys[l.a] = y;
        __syncwarp();
        if (l.h * VL::BM < M) f -= col_dot<VL::BM, N>(b + W::K, ys, l.h * VL::BM, l.j);
        v = b[W::E + l.j] + l.sum_n(f);
        if (!MAP) {
            R d = R(0);
            if (l.ha * VL::BMM < M)
                d = col_dot<VL::BMM, M>(b + W::GI, ys, l.ha * VL::BMM, l.a);
            d = l.sum_m(d);
            if (l.ha == 0) D.u[k * M + l.a] = d;
        }
    }
    cp_async_wait<0>();
    if (MAP) {
        using A = DAffine<N>;
        RT* out = a.FE + cr * A::SIZE;
        const RT* m = maps + c * A::SIZE;
        for (int t = l.lane; t < N * N; t += 32) out[A::OF + t] = m[A::OF + t % N * N + t / N];
        if (l.h == 0) out[A::OC + l.j] = static_cast<RT>(v);
    }
}

// The seed of a scan in each problem's top slot: v_T of the correction problem
// (VALUE) or x_0.
template <typename R, typename RT, int N, bool VALUE>
__global__ void __launch_bounds__(N) k_vseed(Args<R, RT> a) {
    const Item<R>& it = a.items[blockIdx.x];
    a.X[(it.c0 + it.NC - 1) * N + threadIdx.x] =
        static_cast<RT>(VALUE ? it.D.etaT[threadIdx.x] : it.D.x0[threadIdx.x]);
}

// ---- KKT residuals of the first pass's iterate -------------------------------
// k_cresid's residuals (lqt_chain.cuh: e_k, g_k, h_k and U^{-1} h_k, g_T) at the
// team sizes, one warp per run of consecutive steps, walked from the last:
// lambda_{k+1} and x_{k+1} of a step are the step before's, so S_k is read once
// instead of twice, and a ring of stages keeps the next step's matrices on the
// way, where k_cresid waited for every step's loads (n = 32, T = 65536:
// 853 -> 307 us).  The sums are compensated as there; blocks of a sum in
// different lanes are merged by compensated additions.  A time-invariant U is
// inverted once per run.  resid_run: the steps of a run, 16 where that leaves
// 4096 warps, fewer down to 2 for shorter horizons (n = 16, T = 10007: runs of 16
// took 52 us, of 2 24, k_cresid 37).
inline int resid_run(long long T) {
    const long long r = T / 4096;
    return r > 16 ? 16 : r < 2 ? 2 : (int)r;
}

template <int N, int M>
struct VResid {
    static constexpr int r4(int x) { return (x + 3) / 4 * 4; }
    // one stage: F, L, U, S_k, X_k (p = N) | x, u, v, c, r
    static constexpr int F = 0, L = N * N, U = L + N * M, S = U + M * M, X = S + N * N,
                         XV = X + N * N, UV = XV + N, VV = UV + M, CV = VV + N, RV = CV + N,
                         STAGE = r4(RV + N);
    static constexpr int ST = 2;
    static constexpr int NT = N == 32 ? 1 : 4;  // warps per CTA
    // vectors: lambda_{k+1}, x_{k+1}, H x - r and X (H x - r) as (hi, lo), U^{-1} h
    static constexpr int L1 = ST * STAGE, X1 = L1 + N, HH = X1 + N, HL = HH + 2 * N,
                         YH = HL + 2 * N, YL = YH + 2 * N, Q = YL + 2 * N, SIZE = r4(Q + M);
};

// Dot2 (or plain FP64) sums of a block each in the lanes of a row, merged over
// lanes D apart, 2D apart, ... 16 apart
template <int D, typename R>
__device__ __forceinline__ void merge(XAcc<R>& a) {
#pragma unroll
    for (int d = D; d < 32; d <<= 1) {
        if constexpr (sizeof(R) == 4) {
            const float s = __shfl_xor_sync(0xffffffffu, a.d.s, d);
            const float c = __shfl_xor_sync(0xffffffffu, a.d.c, d);
            // the same operand order in both lanes keeps them identical
            const bool low = ((threadIdx.x & 31) & d) == 0;
            float t, e;
            two_sum(low ? a.d.s : s, low ? s : a.d.s, t, e);
            a.d.s = t;
            a.d.c = add_rn(add_rn(a.d.c, c), e);
        } else {
            a.s += __shfl_xor_sync(0xffffffffu, a.s, d);
        }
    }
}

template <typename R, int N, int M>
__global__ void __launch_bounds__(32 * VResid<N, M>::NT)
    k_vresid(const Item<R>* items1, const Item<R>* items2, int steps, int* status) {
    using W = VResid<N, M>;
    using VL = VLane<N, M>;
    using A = XAcc<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    R* sh = reinterpret_cast<R*>(smem_raw) + (threadIdx.x / 32) * W::SIZE;
    const VL l;
    const DescT<R>& D = items1[blockIdx.y].D;
    const DescT<R>& D2 = items2[blockIdx.y].D;
    R* const qh = const_cast<R*>(items2[blockIdx.y].qh);
    R* const eta = const_cast<R*>(D2.eta);
    R* const ctil = const_cast<R*>(D2.c);
    const long long T = D.T;
    const long long run = (long long)blockIdx.x * W::NT + threadIdx.x / 32;
    const long long s = run * steps, e = s + steps < T ? s + steps : T;
    if (s >= T) return;
    R *lam1 = sh + W::L1, *x1 = sh + W::X1, *hh = sh + W::HH, *hl = sh + W::HL, *yh = sh + W::YH,
      *yl = sh + W::YL, *qv = sh + W::Q;
    const int p = D.p;
    const R *F = D.F, *L = D.L, *U = D.U, *H = D.H, *X = D.X, *rp = D.r, *cp = D.c, *S = D.S;
    const long long sF = D.sF, sL = D.sL, sU = D.sU, sH = D.sH, sX = D.sX, sr = D.sr, sc = D.sc;
    const bool vF = vec_ok(F, sF), vL = vec_ok(L, sL), vU = vec_ok(U, sU), vS = vec_ok(S, 0),
               vX = vec_ok(X, sX);
    bool hid = sH == 0 && p == N;
    if (hid)
        for (int t = l.lane; t < N * N; t += 32)
            hid = hid && H[t] == (t / N == t % N ? R(1) : R(0));
    hid = __all_sync(0xffffffffu, hid);
    auto stage = [&](long long k) {
        if (k >= s) {
            R* b = sh + (int)((e - 1 - k) % W::ST) * W::STAGE;
            warp_cp_mat<N, N>(b + W::F, F + k * sF, vF, l.lane);
            warp_cp_mat<N, M>(b + W::L, L + k * sL, vL, l.lane);
            if (sU != 0 || k == e - 1) warp_cp_mat<M, M>(b + W::U, U + k * sU, vU, l.lane);
            warp_cp_mat<N, N>(b + W::S, S + k * (N * N), vS, l.lane);
            if (p == N) warp_cp_mat<N, N>(b + W::X, X + k * sX, vX, l.lane);
            if (l.h == 0) {
                cp_async<sizeof(R)>(b + W::XV + l.j, D.x + k * N + l.j);
                cp_async<sizeof(R)>(b + W::VV + l.j, D.v + k * N + l.j);
                if (cp) cp_async<sizeof(R)>(b + W::CV + l.j, cp + k * sc + l.j);
                if (p == N && rp) cp_async<sizeof(R)>(b + W::RV + l.j, rp + k * sr + l.j);
            }
            if (l.ha == 0) cp_async<sizeof(R)>(b + W::UV + l.a, D.u + k * M + l.a);
        }
        cp_async_commit();
    };
    stage(e - 1);
    // lambda_e = S_e x_e - v_e and x_e; the last run also the terminal condition
    {
        const R xe = D.x[e * N + l.j];
        if (l.h == 0) x1[l.j] = xe;
        __syncwarp();
        R t = R(0);
        for (int i = l.h * VL::BN; i < (l.h + 1) * VL::BN; ++i)
            t = team::fma_(S[e * (N * N) + i * N + l.j], x1[i], t);
        const R lam = l.sum_n(t) - D.v[e * N + l.j];
        if (l.h == 0) lam1[l.j] = lam;
        __syncwarp();
        if (e == T) {
            for (int i = l.lane; i < D.pT; i += 32) {
                A h(D.rT ? -D.rT[i] : R(0));
                for (int j = 0; j < N; ++j) h.add_prod(D.HT[i * N + j], x1[j]);
                h.split(hh[i], hl[i]);
            }
            __syncwarp();
            for (int i = l.lane; i < D.pT; i += 32) {
                A t2(R(0));
                for (int b = 0; b < D.pT; ++b) t2.add_prod2(D.XT[i * D.pT + b], hh[b], hl[b]);
                t2.split(yh[i], yl[i]);
            }
            __syncwarp();
            if (l.h == 0) {
                A g(-lam1[l.j]);
                for (int i = 0; i < D.pT; ++i) g.add_prod2(D.HT[i * N + l.j], yh[i], yl[i]);
                const_cast<R*>(D2.etaT)[l.j] = -g.value();
                const_cast<R*>(D2.x0)[l.j] = R(0);
            }
            __syncwarp();
        }
    }
    constexpr int EP = 16 / (int)sizeof(R), V = VL::BN < EP ? VL::BN : EP;
    bool ok = true;
    R ui[M];  // a time-invariant U: column a of U^{-1} in lane a < M
    for (long long k = e - 1; k >= s; --k) {
        cp_async_wait<0>();
        __syncwarp();
        stage(k - 1);
        const R* b = sh + (int)((e - 1 - k) % W::ST) * W::STAGE;
        // h's solve: U (lanes a < M, column a) eliminated once or with its right side
        const bool invert = sU == 0 && k == e - 1;
        const R *xv = b + W::XV, *uv = b + W::UV;
        // H x^ - r as (hi, lo)
        if (hid) {
            if (l.h == 0) {
                A h(xv[l.j]);
                if (rp) h.add(-b[W::RV + l.j]);
                h.split(hh[l.j], hl[l.j]);
            }
        } else {
            const R* Hk = H + k * sH;
            const R* rk = rp ? rp + k * sr : nullptr;
            for (int i = l.lane; i < p; i += 32) {
                A h(rk ? -rk[i] : R(0));
                for (int j = 0; j < N; ++j) h.add_prod(Hk[i * N + j], xv[j]);
                h.split(hh[i], hl[i]);
            }
        }
        __syncwarp();
        // y = X (H x^ - r) as (hi, lo)
        if (p == N) {
            A t;
#pragma unroll
            for (int q = 0; q < VL::BN; q += V) {
                const int i = l.h * VL::BN + q;
                R x[V];
                ldrow<N, V>(b + W::X, l.j, i, x);
#pragma unroll
                for (int w = 0; w < V; ++w) t.add_prod2(x[w], hh[i + w], hl[i + w]);
            }
            merge<N>(t);
            if (l.h == 0) t.split(yh[l.j], yl[l.j]);
        } else {
            const R* Xk = X + k * sX;
            for (int i = l.lane; i < p; i += 32) {
                A t;
                for (int q = 0; q < p; ++q) t.add_prod2(Xk[i * p + q], hh[q], hl[q]);
                t.split(yh[i], yl[i]);
            }
        }
        __syncwarp();
        // lambda_k in the working precision (any iterate's exact residuals do)
        const R lam =
            l.sum_n(col_dot<VL::BN, N>(b + W::S, xv, l.h * VL::BN, l.j)) - b[W::VV + l.j];
        // g = H^T y - lambda_k + F^T lambda_{k+1}
        A g(l.h == 0 ? -lam : R(0));
        if (hid) {
            if (l.h == 0) {
                g.add(yh[l.j]);
                g.add(yl[l.j]);
            }
        } else {
            const R* Hk = H + k * sH;
            for (int i = l.h; i < p; i += VL::G) g.add_prod2(Hk[i * N + l.j], yh[i], yl[i]);
        }
#pragma unroll
        for (int q = 0; q < VL::BN; ++q) {
            const int i = l.h * VL::BN + q;
            g.add_prod(b[W::F + Sw<R, N>::at(i, l.j)], lam1[i]);
        }
        merge<N>(g);
        // h = U u^ + L^T lambda_{k+1}
        const R* Uk = sU == 0 ? sh + W::U : b + W::U;  // an invariant U stays in slot 0
        A hr;
#pragma unroll
        for (int q = 0; q < VL::BMM; ++q) {
            const int i = l.ha * VL::BMM + q;
            if (i < M) hr.add_prod(Uk[Sw<R, M>::at(l.a, i)], uv[i]);
        }
#pragma unroll
        for (int q = 0; q < VL::BNM; ++q) {
            const int i = l.ha * VL::BNM + q;
            hr.add_prod(b[W::L + Sw<R, M>::at(i, l.a)], lam1[i]);
        }
        merge<M>(hr);
        const R h = hr.value();
        // U^{-1} h in the working precision (h is the residual itself)
        R qa;
        if (sU != 0 || invert) {
            // column a of [U | h] per lane (lane M: h), Gauss-Jordan without
            // pivoting; an invariant U's columns become those of U^{-1}
            R col[M];
#pragma unroll
            for (int i = 0; i < M; ++i) {
                const R hi = __shfl_sync(0xffffffffu, h, i);
                col[i] = l.lane < M ? Uk[Sw<R, M>::at(l.a, i)] : hi;
            }
#pragma unroll
            for (int q = 0; q < M; ++q) {
                const R piv = __shfl_sync(0xffffffffu, col[q], q);
                ok = ok && piv > R(0) && isfinite(piv);
                const R inv = rcp(piv);
                const bool own = invert && l.lane == q;
                const R pk = own ? inv : col[q] * inv;
#pragma unroll
                for (int i = 0; i < M; ++i) {
                    if (i == q) continue;
                    const R f = __shfl_sync(0xffffffffu, col[i], q);
                    col[i] = team::fma_(-f, pk, own ? R(0) : col[i]);
                }
                col[q] = pk;
            }
            qa = R(0);
#pragma unroll
            for (int i = 0; i < M; ++i) {
                const R t = __shfl_sync(0xffffffffu, col[i], M);  // lane M's solution
                if (l.a == i) qa = t;
                ui[i] = col[i];
            }
        } else {
            qa = R(0);
#pragma unroll
            for (int i = 0; i < M; ++i)  // U^{-1} symmetric: row a is lane a's column
                qa = team::fma_(__shfl_sync(0xffffffffu, ui[i], l.a), __shfl_sync(0xffffffffu, h, i),
                                qa);
        }
        if (l.ha == 0) {
            qv[l.a] = qa;
            qh[k * M + l.a] = qa;
        }
        __syncwarp();
        // e = F x^ + c + L (u^ - U^{-1} h) - x^_{k+1}
        A er(l.h == 0 && cp ? b[W::CV + l.j] : R(0));
        if (l.h == 0) er.add(-x1[l.j]);
#pragma unroll
        for (int q = 0; q < VL::BN; q += V) {
            const int i = l.h * VL::BN + q;
            R f[V];
            ldrow<N, V>(b + W::F, l.j, i, f);
#pragma unroll
            for (int w = 0; w < V; ++w) er.add_prod(f[w], xv[i + w]);
        }
#pragma unroll
        for (int q = 0; q < VL::BM; ++q) {
            const int i = l.h * VL::BM + q;
            if (i < M) {
                const R lv = b[W::L + Sw<R, M>::at(l.j, i)];
                er.add_prod(lv, uv[i]);
                er.add_prod(-lv, qv[i]);
            }
        }
        merge<N>(er);
        __syncwarp();  // lam1 and x1 are read
        if (l.h == 0) {
            eta[k * N + l.j] = -g.value();
            ctil[k * N + l.j] = er.value();
            lam1[l.j] = lam;
            x1[l.j] = xv[l.j];
        }
        __syncwarp();
    }
    cp_async_wait<0>();
    flag(status, ok);
}

}  // namespace chain
}  // namespace lqt
