// Chunk and tree-level kernels of the chunked pipeline (lqt_chain.cuh) at
// n = 8, 16, 32: the team algebra of lqt_team.cuh.  Included by lqt_chain.cuh.
//
// k_tfold and k_trefold walk a chunk's steps; a step's F, L, U, c come by
// cp.async into one of two buffers while the step before is computed, and with
// H = I the tile of X_k and r_k goes straight to registers.  Bound: the
// shared-memory data pipe, 91% busy over a batch at n = 16 (97% on the busiest
// SM); 512 problems of n = 16, fold / re-fold: a lane group with a row per lane
// 2.16 / 2.10 ms, teams 0.90 / 1.12; n = 8 0.40 / 0.43 and 0.20 / 0.26; n = 32,
// T = 65536: 1.16 / 1.39 ms of a plain scan that went from 6.5 to 2.9.
// k_tup, k_tdown,
// k_tfup, k_tfdown run several tree levels per launch: a CTA of TT teams owns
// 2 TT neighbouring nodes, and its teams meet at a CTA barrier between the
// levels, where the global-memory results of one level are read by the next.
// They are operator latency (a 16 x 16 operator by one lane group took 27 to
// 33 us a level, launch included; T = 10007, n = 16, 2048 chunks: 10 levels up and
// 11 down now take 126 us in 6 launches).
#pragma once

#include "lqt_chain_args.cuh"
#include "lqt_team.cuh"

namespace lqt {
namespace chain {

using team::DAffine;
using team::DElem;
using team::DValue;
using team::Sw;
using team::Team;
using team::ldrow;
using team::strow;

// ROWS x COLS dense global matrix -> swizzled shared matrix by cp.async
template <int ROWS, int COLS, int N, int RT, typename R>
__device__ __forceinline__ void cp_mat(R* dst, const R* src, bool vec, const Team<N, RT>& g) {
    constexpr int E = 16 / (int)sizeof(R), RC = COLS / E, LG = Team<N, RT>::LG;
    if (vec) {
#pragma unroll
        for (int t = g.lane; t < ROWS * RC; t += LG)
            cp_async_cg16(dst + Sw<R, COLS>::chunk(t / RC, t % RC), src + t * E);
    } else {
        for (int t = g.lane; t < ROWS * COLS; t += LG)
            cp_async<sizeof(R)>(dst + Sw<R, COLS>::at(t / COLS, t % COLS), src + t);
    }
}

template <typename R>
__device__ __forceinline__ bool vec_ok(const R* p, long long stride) {
    return (reinterpret_cast<uintptr_t>(p) & 15) == 0 &&
           (stride & (16 / (int)sizeof(R) - 1)) == 0;
}

// Staged inputs of a step: two buffers of F, L, U, c (offsets in elements).
template <int N, int M>
struct TeamIn {
    static constexpr int F = 0, L = 2 * N * N, U = L + 2 * N * M, C = U + 2 * M * M,
                         SIZE = C + 2 * N;
};

// The problem's descriptor in the team's shared memory: a walk reads pointers
// and strides at every step, and with the SM's memory given to the teams a copy
// in global memory would mostly be read from L2.
constexpr int kDescElems = 64;  // elements reserved per team (at least 256 bytes)
template <int N, int RT, typename R>
__device__ __forceinline__ const DescT<R>& desc_in(R* dst, const DescT<R>& src,
                                                   const Team<N, RT>& g) {
    static_assert(sizeof(DescT<R>) <= kDescElems * sizeof(float), "descriptor area");
    static_assert(sizeof(DescT<R>) % 4 == 0, "copied in words");
    const int* s = reinterpret_cast<const int*>(&src);
    int* d = reinterpret_cast<int*>(dst);
    for (int i = g.lane; i < (int)(sizeof(DescT<R>) / 4); i += Team<N, RT>::LG) d[i] = s[i];
    g.sync();
    return *reinterpret_cast<const DescT<R>*>(dst);
}

// What a chunk walk knows about its problem's arrays.
template <typename R, int N, int M, int RT>
struct TeamWalk {
    using Tm = Team<N, RT>;
    bool vF, vL, vU, vX, vr, hid, has_c, u_once;
    __device__ TeamWalk(const DescT<R>& D, const Tm& g) {
        vF = vec_ok(D.F, D.sF);
        vL = vec_ok(D.L, D.sL);
        vU = vec_ok(D.U, D.sU);
        vX = vec_ok(D.X, D.sX);
        vr = D.r && vec_ok(D.r, D.sr);
        has_c = D.c != nullptr;
        u_once = D.sU == 0;
        // H = I at every step (p = N)?
        bool mine = D.sH == 0 && D.p == N && D.H;
        if (mine) {
#pragma unroll 8
            for (int t = g.lane; t < N * N; t += Tm::LG)
                mine = mine & (D.H[t] == (t / N == t % N ? R(1) : R(0)));
        }
        hid = g.all(mine);
    }
    __device__ __forceinline__ void stage(const DescT<R>& D, long long k, R* in, int b, bool first,
                                          const Tm& g) const {
        using I = TeamIn<N, M>;
        cp_mat<N, N>(in + I::F + b * N * N, D.F + k * D.sF, vF, g);
        cp_mat<N, M>(in + I::L + b * N * M, D.L + k * D.sL, vL, g);
        if (first || !u_once) cp_mat<M, M>(in + I::U + b * M * M, D.U + k * D.sU, vU, g);
        if (has_c)
            for (int i = g.lane; i < N; i += Tm::LG)
                cp_async<sizeof(R)>(in + I::C + b * N + i, D.c + k * D.sc + i);
        cp_async_commit();
    }
};

// Q_k = H^T X H (TN tile) and the entries of q_k = H^T X r a lane needs.
template <typename R, int RT>
struct CostTile {
    R x[RT][4], r[4];
};

// H = I: the tile of X_k and four entries of r_k from global memory
template <int N, int M, int RT, typename R>
__device__ __forceinline__ void cost_prefetch(CostTile<R, RT>& ct, const DescT<R>& D, long long k,
                                              const TeamWalk<R, N, M, RT>& w,
                                              const Team<N, RT>& g) {
    const R* X = D.X + k * D.sX;
#pragma unroll
    for (int i = 0; i < RT; ++i) team::ldg_row<N, 4>(X, RT * g.ri + i, 4 * g.ci, ct.x[i], w.vX);
    if (D.r && !D.eta) {
        team::ldg_row<N, 4>(D.r + k * D.sr, 0, 4 * g.ci, ct.r, w.vr);
    } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) ct.r[c] = R(0);
    }
}

// General H and X: Y = X H and X r in the scratch (p <= 2N; with p <= N also H
// and X staged there), then the TN tile of H^T Y and its rows of H^T X r.
// scr: 3 N^2 + N elements, xr: 2 N.  Ends with a sync.
template <int N, int RT, typename R>
__device__ void cost_general(R (&x)[RT][4], R (&q)[RT], const DescT<R>& D, long long k, R* scr,
                             R* xr, const Team<N, RT>& g) {
    using Tm = Team<N, RT>;
    const int p = D.p, ri = g.ri, ci = g.ci;
    const bool staged = p <= N;
    R* Y = scr;  // p x N
    const int lp = staged ? p | 1 : p;  // row stride of X: odd where it is staged
    const R* X = D.X + k * D.sX;
    const R* H = D.H + k * D.sH;
    const R* rk = D.r ? D.r + k * D.sr : nullptr;
    if (staged) {
        R* Hs = scr + N * N;
        R* Xs = scr + 2 * N * N;
        for (int t = g.lane; t < p * N; t += Tm::LG) cp_async<sizeof(R)>(Hs + t, H + t);
        for (int i = ri; i < p; i += Tm::LR)
            for (int j = ci; j < p; j += Tm::LC) cp_async<sizeof(R)>(Xs + i * lp + j, X + i * p + j);
        cp_async_commit();
        cp_async_wait<0>();
        H = Hs;
        X = Xs;
    }
    g.sync();
    for (int i = ri; i < p; i += Tm::LR) {
        R y[4] = {R(0), R(0), R(0), R(0)};
        R t = R(0);
#pragma unroll 4
        for (int b = 0; b < p; ++b) {
            const R v = X[i * lp + b];
#pragma unroll
            for (int c = 0; c < 4; ++c) y[c] = team::fma_(v, H[b * N + 4 * ci + c], y[c]);
            if (rk && ci == 0) t = team::fma_(v, rk[b], t);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) Y[i * N + 4 * ci + c] = y[c];
        if (ci == 0) xr[i] = t;
    }
    g.sync();
    team::zero(x);
#pragma unroll
    for (int i = 0; i < RT; ++i) q[i] = R(0);
#pragma unroll 4
    for (int b = 0; b < p; ++b) {
        R y[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) y[c] = Y[b * N + 4 * ci + c];
        const R xb = xr[b];
#pragma unroll
        for (int i = 0; i < RT; ++i) {
            const R h = H[b * N + RT * ri + i];
#pragma unroll
            for (int c = 0; c < 4; ++c) x[i][c] = team::fma_(h, y[c], x[i][c]);
            q[i] = team::fma_(h, xb, q[i]);
        }
    }
    g.sync();
}

// q's rows with H = I (every lane of the row gets them)
template <int N, int RT, typename R>
__device__ __forceinline__ void cost_q(const CostTile<R, RT>& ct, R (&q)[RT],
                                       const Team<N, RT>& g) {
#pragma unroll
    for (int i = 0; i < RT; ++i) {
        R t = R(0);
#pragma unroll
        for (int c = 0; c < 4; ++c) t = team::fma_(ct.x[i][c], ct.r[c], t);
        q[i] = g.row_sum(t);
    }
}

// Shared memory of one team (elements): the running total P | staged inputs |
// JF, JL, the m x m system [G | Z | P2^T | L^T w] | vectors.
template <int N, int M>
struct TFoldSmem {
    using Sy = team::Sys<N, M, 2 * N + 1>;
    static constexpr int at_least(int a, int b) { return a > b ? a : b; }
    static constexpr int PA = 0, PC = N * N, PJ = 2 * N * N, IN = 3 * N * N,
                         JF = IN + TeamIn<N, M>::SIZE, JL = JF + N * N, SY = JL + N * M,
                         // at least cost_general's scratch from JF on
                         V = JF + at_least(N * N + N * M + Sy::SIZE, 3 * N * N + N), PB = V,
                         PE = PB + N, W = PE + N, AC = W + N, DESC = AC + N,
                         SIZE = DESC + kDescElems;
    static_assert(IN % 4 == 0 && SY % 4 == 0 && V % 4 == 0 && DESC % 2 == 0, "aligned parts");
};

// Distance between the blocks of neighbouring teams (elements, a multiple of
// 16 bytes).  At n = 8 four teams share a warp and read 4 rows of 32 bytes
// each at once: the extra 16 bytes put neighbours on the other banks.
template <int N, typename R>
constexpr int tstride_of(int size) {
    constexpr int E = 16 / (int)sizeof(R);
    return (size + 31) / 32 * 32 + (N == 8 ? E : 0);
}

// ---- chunk totals: P <- a_k (x) P from the chunk's end (eq. lqt_comb with a
// step element on the left, the low-rank form of lanes::fold_step):
//   Z = L^T J F, G = U + L^T J L = Rc Rc^T, w = eta - J c, P2 = A L,
//   [Zt | om | Wt] = Rc^{-1} [Z | L^T w | P2^T],
//   A <- A F - Wt^T Zt, b <- A c + Wt^T om + b, C <- C + Wt^T Wt,
//   J <- H^T X H + F^T J F - Zt^T Zt, eta <- q + F^T w - Zt^T om.
// The forward substitution alone suffices: G^{-1} only occurs between two of
// its right sides.
template <typename R, typename RT, int N, int M, int TR = 2>
__device__ __forceinline__ void b_tfold(const Args<R, RT>& a, long long c, R* sh) {
    static_assert(M == N / 2, "tiles of L, K and G assume m = n / 2");
    using S = TFoldSmem<N, M>;
    using I = TeamIn<N, M>;
    using E = DElem<N>;
    using Tm = Team<N, TR>;
    constexpr int H = Tm::LR, TM = TR / 2;  // row step of NN tiles; rows of M x . tiles
    const Tm g;
    const int ri = g.ri, ci = g.ci;
    const Item<R>& it = a.items[find_chunk(a.items, a.count, c)];
    const DescT<R>& D = desc_in(sh + S::DESC, it.D, g);
    R *PA = sh + S::PA, *PC = sh + S::PC, *PJ = sh + S::PJ;
    R *b = sh + S::PB, *e = sh + S::PE, *w = sh + S::W, *ac = sh + S::AC;
    R *JF = sh + S::JF, *JL = sh + S::JL, *sy = sh + S::SY;
    constexpr int LD = S::Sy::LD, CZ = M, CW = M + N, CO = M + 2 * N;  // columns of the system
    const long long T = D.T;
    const long long lc = c - it.c0, B = it.B;
    // no suffix holds a problem's first chunk.  Unless Method 2 wants its total, it
    // is walked for its status alone: U_k has to be positive definite, which the
    // re-fold, whose G_k has the terminal cost in S, does not see.  Every U of a
    // time-invariant one is the G of the chunk's last step (J = 0 there).
    const long long e0 = lc * B + B < T ? lc * B + B : T;
    long long s0 = lc * B < T ? lc * B : T;
    if (lc == 0 && !a.first_total && D.sU == 0 && s0 < e0) s0 = e0 - 1;
    const TeamWalk<R, N, M, TR> wk(D, g);
    if (s0 < e0) wk.stage(D, e0 - 1, sh + S::IN, 0, true, g);
    {
        R z[TR][4], o[TR][4];
        team::zero(z);
#pragma unroll
        for (int i = 0; i < TR; ++i) {
#pragma unroll
            for (int q = 0; q < 4; ++q) o[i][q] = ri + i * H == 4 * ci + q ? R(1) : R(0);
            if (ci == 0) b[ri + i * H] = e[ri + i * H] = R(0);
        }
        team::sttile<N>(PA, ri, H, 4 * ci, o);
        team::sttile<N>(PC, ri, H, 4 * ci, z);
        team::sttile<N>(PJ, ri, H, 4 * ci, z);
    }
    bool ok = true;
    for (long long k = e0 - 1; k >= s0; --k) {
        const int cur = (int)((e0 - 1 - k) & 1);
        const R* F = sh + S::IN + I::F + cur * N * N;
        const R* L = sh + S::IN + I::L + cur * N * M;
        const R* U = sh + S::IN + I::U + (wk.u_once ? 0 : cur) * M * M;
        const R* cv = sh + S::IN + I::C + cur * N;
        cp_async_wait<0>();
        g.sync();  // the inputs are in; the step before is done with the other buffer
        CostTile<R, TR> cost;  // with H = I read before the solve
        R q[TR];
        if (k > s0) wk.stage(D, k - 1, sh + S::IN, cur ^ 1, false, g);
        if (!wk.hid) cost_general<N>(cost.x, q, D, k, JF, w, g);
        // JF = J F, JL = J L, P2^T = (A L)^T to shared memory, A F in registers
        R af[TR][4];
        {
            R jf[TR][4], jl[TR][2], al[TR][2];
            team::zero(af);
            team::zero(jf);
            team::zero(jl);
            team::zero(al);
            constexpr int EP = 16 / (int)sizeof(R);
#pragma unroll(team::k_unroll(N) / EP)
            for (int kk = 0; kk < N; kk += EP) {
                R jr[TR][EP], ar[TR][EP];
                team::ldtile<N>(PJ, ri, H, kk, jr);
                team::ldtile<N>(PA, ri, H, kk, ar);
#pragma unroll
                for (int x = 0; x < EP; ++x) {
                    R f[4], l[2];
                    ldrow<N, 4>(F, kk + x, 4 * ci, f);
                    ldrow<M, 2>(L, kk + x, 2 * ci, l);
#pragma unroll
                    for (int i = 0; i < TR; ++i) {
#pragma unroll
                        for (int y = 0; y < 4; ++y) {
                            jf[i][y] = team::fma_(jr[i][x], f[y], jf[i][y]);
                            af[i][y] = team::fma_(ar[i][x], f[y], af[i][y]);
                        }
#pragma unroll
                        for (int y = 0; y < 2; ++y) {
                            jl[i][y] = team::fma_(jr[i][x], l[y], jl[i][y]);
                            al[i][y] = team::fma_(ar[i][x], l[y], al[i][y]);
                        }
                    }
                }
            }
            team::sttile<N>(JF, ri, H, 4 * ci, jf);
            team::sttile<M>(JL, ri, H, 2 * ci, jl);
#pragma unroll
            for (int i = 0; i < TR; ++i)
#pragma unroll
                for (int y = 0; y < 2; ++y) sy[(2 * ci + y) * LD + CW + ri + i * H] = al[i][y];
            if (wk.has_c) {
                R jr[TR][4], ar[TR][4], cx[4];
                team::ldtile<N>(PJ, ri, H, 4 * ci, jr);
                team::ldtile<N>(PA, ri, H, 4 * ci, ar);
#pragma unroll
                for (int x = 0; x < 4; ++x) cx[x] = cv[4 * ci + x];
#pragma unroll
                for (int i = 0; i < TR; ++i) {
                    R s = R(0), t = R(0);
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        s = team::fma_(-jr[i][x], cx[x], s);
                        t = team::fma_(ar[i][x], cx[x], t);
                    }
                    s = g.row_sum(s);
                    t = g.row_sum(t);
                    if (ci == 0) {
                        w[ri + i * H] = e[ri + i * H] + s;
                        ac[ri + i * H] = t;
                    }
                }
            } else if (ci == 0) {
#pragma unroll
                for (int i = 0; i < TR; ++i) {
                    w[ri + i * H] = e[ri + i * H];
                    ac[ri + i * H] = R(0);
                }
            }
        }
        g.sync();
        // G = U + L^T JL, Z = L^T JF; L^T w; F^T JF and F^T w in registers
        R fw[TR], jj[TR][4];
        team::zero(jj);
        {
            R zz[TM][4], gg[TM][2];
            team::zero(zz);
            team::ldtile<M>(U, TM * ri, 1, 2 * ci, gg);
#pragma unroll(team::k_unroll(N))
            for (int kk = 0; kk < N; ++kk) {
                R f[TR], l[TM], jf[4], jl[2];
                ldrow<N, TR>(F, kk, TR * ri, f);
                ldrow<M, TM>(L, kk, TM * ri, l);
                ldrow<N, 4>(JF, kk, 4 * ci, jf);
                ldrow<M, 2>(JL, kk, 2 * ci, jl);
#pragma unroll
                for (int i = 0; i < TR; ++i)
#pragma unroll
                    for (int y = 0; y < 4; ++y)
                        jj[i][y] = team::fma_(f[i], jf[y], jj[i][y]);
#pragma unroll
                for (int i = 0; i < TM; ++i) {
#pragma unroll
                    for (int y = 0; y < 4; ++y) zz[i][y] = team::fma_(l[i], jf[y], zz[i][y]);
#pragma unroll
                    for (int y = 0; y < 2; ++y) gg[i][y] = team::fma_(l[i], jl[y], gg[i][y]);
                }
            }
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                team::stsys<LD>(sy, TM * ri + i, CZ + 4 * ci, zz[i]);
                team::stsys<LD>(sy, TM * ri + i, 2 * ci, gg[i]);
            }
            R lw[TM];
#pragma unroll
            for (int i = 0; i < TR; ++i) fw[i] = R(0);
#pragma unroll
            for (int i = 0; i < TM; ++i) lw[i] = R(0);
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const R wx = w[4 * ci + x];
                R f[TR], l[TM];
                ldrow<N, TR>(F, 4 * ci + x, TR * ri, f);
                ldrow<M, TM>(L, 4 * ci + x, TM * ri, l);
#pragma unroll
                for (int i = 0; i < TR; ++i) fw[i] = team::fma_(f[i], wx, fw[i]);
#pragma unroll
                for (int i = 0; i < TM; ++i) lw[i] = team::fma_(l[i], wx, lw[i]);
            }
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                lw[i] = g.row_sum(lw[i]);
                if (ci == 0) sy[(TM * ri + i) * LD + CO] = lw[i];
            }
        }
        g.sync();
        if (wk.hid) cost_prefetch<N, M>(cost, D, k, wk, g);
        // G = Rc Rc^T; [Zt | Wt | om] = Rc^{-1} [Z | P2^T | L^T w] in place
        ok &= team::solve_spd<false, M, 2 * N + 1>(sy, g);
        g.sync();
        // A <- A F - Wt^T Zt (NN rows), C <- C + Wt^T Wt and J <- H^T X H + F^T J F
        // - Zt^T Zt (TN rows), b <- A c + Wt^T om + b, eta <- q + F^T w - Zt^T om.
        // C stays symmetric to the last bit; raw J goes to the step's F, which
        // nothing reads any more, and is symmetrised.
        R* rawJ = sh + S::IN + I::F + cur * N * N;
        {
            R cc[TR][4];
            team::ldtile<N>(PC, TR * ri, 1, 4 * ci, cc);
#pragma unroll(team::k_unroll(M))
            for (int kk = 0; kk < M; ++kk) {
                R zt[4], wt[4], z[TR], wn[TR], wr[TR];
                team::ldsys<LD>(sy, kk, CZ + 4 * ci, zt);
                team::ldsys<LD>(sy, kk, CW + 4 * ci, wt);
                team::ldsys<LD>(sy, kk, CZ + TR * ri, z);
                team::ldsys<LD>(sy, kk, CW + TR * ri, wr);
#pragma unroll
                for (int i = 0; i < TR; ++i) wn[i] = sy[kk * LD + CW + ri + i * H];
#pragma unroll
                for (int i = 0; i < TR; ++i)
#pragma unroll
                    for (int y = 0; y < 4; ++y) {
                        af[i][y] = team::fma_(-wn[i], zt[y], af[i][y]);
                        cc[i][y] = team::fma_(wr[i], wt[y], cc[i][y]);
                        jj[i][y] = team::fma_(-z[i], zt[y], jj[i][y]);
                    }
            }
            R s[TR];
#pragma unroll
            for (int i = 0; i < TR; ++i) s[i] = R(0);
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                const int row = 2 * ci + x;
                const R o = sy[row * LD + CO];
                R z[TR];
                team::ldsys<LD>(sy, row, CZ + TR * ri, z);
#pragma unroll
                for (int i = 0; i < TR; ++i) {
                    s[i] = team::fma_(sy[row * LD + CW + ri + i * H], o, s[i]);
                    fw[i] = team::fma_(-z[i], o, fw[i]);
                }
            }
            if (wk.hid) cost_q<N>(cost, q, g);
            if (D.eta) {
#pragma unroll
                for (int i = 0; i < TR; ++i) q[i] = D.eta[k * D.seta + TR * ri + i];
            }
#pragma unroll
            for (int i = 0; i < TR; ++i) {
                s[i] = g.row_sum(s[i]);
                fw[i] = g.row_sum(fw[i]);
                if (ci == 0) {
                    b[ri + i * H] += ac[ri + i * H] + s[i];
                    e[TR * ri + i] = q[i] + fw[i];
                }
#pragma unroll
                for (int y = 0; y < 4; ++y) jj[i][y] += cost.x[i][y];
            }
            team::sttile<N>(PA, ri, H, 4 * ci, af);
            team::sttile<N>(PC, TR * ri, 1, 4 * ci, cc);
            team::sttile<N>(rawJ, TR * ri, 1, 4 * ci, jj);
        }
        g.sync();
        team::symmetrise<N>(jj, rawJ, g);
        team::sttile<N>(PJ, TR * ri, 1, 4 * ci, jj);
    }
    g.sync();
    RT* out = a.E + c * E::SIZE;
    for (int t = g.lane; t < N * N; t += Tm::LG) {
        const int q = Sw<R, N>::at(t / N, t % N);
        out[E::OA + t] = static_cast<RT>(PA[q]);
        out[E::OC + t] = static_cast<RT>(PC[q]);
        out[E::OJ + t] = static_cast<RT>(PJ[q]);
    }
    for (int i = g.lane; i < N; i += Tm::LG) {
        out[E::OB + i] = static_cast<RT>(b[i]);
        out[E::OE + i] = static_cast<RT>(e[i]);
    }
    flag(a.status, ok);
}

template <typename R, typename RT, int N, int M, int TR, int NT, int MINB>
__global__ void __launch_bounds__(NT * Team<N, TR>::LG, MINB) k_tfold(Args<R, RT> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int gi = threadIdx.x / Team<N, TR>::LG;
    const long long c = (long long)blockIdx.x * NT + gi;
    if (c >= a.C) return;
    b_tfold<R, RT, N, M, TR>(a, c, reinterpret_cast<R*>(smem_raw) +
                                       gi * tstride_of<N, R>(TFoldSmem<N, M>::SIZE));
}

// ---- per-chunk Riccati re-fold with outputs and the chunk affine map -------
template <int N, int M>
struct TRefoldSmem {
    using Sy = team::Sys<N, M, N + 1>;
    // the raw S_k takes SL and the system once both are read
    static constexpr int SV = 0, PHI = N * N, IN = 2 * N * N, SL = IN + TeamIn<N, M>::SIZE,
                         SY = SL + N * M, FT = SY + Sy::SIZE, SFT = FT + N * N, V = SFT + N * N,
                         VV = V, GM = VV + N, EV = GM + N, CT = EV + N, DESC = CT + N,
                         SIZE = DESC + kDescElems;
    static_assert(N < 8 || FT - SL >= N * N, "raw S_k");
    static_assert(N < 8 || V - SL >= 3 * N * N + N, "cost_general's scratch");
    static_assert(SL % 4 == 0 && SY % 4 == 0 && FT % 4 == 0 && V % 4 == 0 && DESC % 2 == 0,
                  "aligned parts");
};

template <typename R, typename RT, int N, int M, int TR = 2>
__device__ __forceinline__ void b_trefold(const Args<R, RT>& a, long long c, R* sh) {
    using S = TRefoldSmem<N, M>;
    using I = TeamIn<N, M>;
    using Tm = Team<N, TR>;
    constexpr int H = Tm::LR, LG = Tm::LG, TM = TR / 2;
    const Tm g;
    const int ri = g.ri, ci = g.ci;
    const Item<R>& it = a.items[find_chunk(a.items, a.count, c)];
    const DescT<R>& D = desc_in(sh + S::DESC, it.D, g);
    R *Sm = sh + S::SV, *Phi = sh + S::PHI, *SL = sh + S::SL, *Ft = sh + S::FT, *SFt = sh + S::SFT,
      *sy = sh + S::SY;
    R *v = sh + S::VV, *ev = sh + S::EV, *gm = sh + S::GM, *ct = sh + S::CT;
    constexpr int LD = S::Sy::LD, CK = M, CD = M + N;  // columns of the system: K, d
    const long long T = D.T;
    const long long lc = c - it.c0, B = it.B;
    const long long s0 = lc * B < T ? lc * B : T;
    const long long e0 = s0 + B < T ? s0 + B : T;
    const TeamWalk<R, N, M, TR> wk(D, g);
    const bool vS = vec_ok(D.S, 0), vK = vec_ok(D.K, 0);
    // no prefix holds a problem's last chunk: its map is left neutral, unless the
    // refinement keeps it (the value scan runs the other way)
    const bool map = lc + 1 < it.NC || a.maps;
    R* gi = it.gi;
    if (s0 < e0) wk.stage(D, e0 - 1, sh + S::IN, 0, true, g);
    {
        const RT* val = a.V + c * DValue<N>::SIZE;
        for (int t = g.lane; t < N * N; t += LG) {
            const int q = Sw<R, N>::at(t / N, t % N);
            Sm[q] = static_cast<R>(val[DValue<N>::OS + t]);
            Phi[q] = t / N == t % N ? R(1) : R(0);
        }
        for (int i = g.lane; i < N; i += LG) {
            v[i] = static_cast<R>(val[DValue<N>::OV + i]);
            gm[i] = R(0);
        }
    }
    bool ok = true;
    for (long long k = e0 - 1; k >= s0; --k) {
        const int cur = (int)((e0 - 1 - k) & 1);
        const R* F = sh + S::IN + I::F + cur * N * N;
        const R* L = sh + S::IN + I::L + cur * N * M;
        const R* U = sh + S::IN + I::U + (wk.u_once ? 0 : cur) * M * M;
        const R* cv = sh + S::IN + I::C + cur * N;
        cp_async_wait<0>();
        g.sync();
        CostTile<R, TR> cost;  // with H = I read before the solve
        R q[TR];
        if (k > s0) wk.stage(D, k - 1, sh + S::IN, cur ^ 1, false, g);
        if (!wk.hid) cost_general<N>(cost.x, q, D, k, SL, ev, g);
        // S F in registers, S L to shared memory, ev = v - S c
        R sf[TR][4];
        {
            R sl[TR][2];
            team::zero(sf);
            team::zero(sl);
            constexpr int EP = 16 / (int)sizeof(R);
#pragma unroll(team::k_unroll(N) / EP)
            for (int kk = 0; kk < N; kk += EP) {
                R sr[TR][EP];
                team::ldtile<N>(Sm, ri, H, kk, sr);
#pragma unroll
                for (int x = 0; x < EP; ++x) {
                    R f[4], l[2];
                    ldrow<N, 4>(F, kk + x, 4 * ci, f);
                    ldrow<M, 2>(L, kk + x, 2 * ci, l);
#pragma unroll
                    for (int i = 0; i < TR; ++i) {
#pragma unroll
                        for (int y = 0; y < 4; ++y)
                            sf[i][y] = team::fma_(sr[i][x], f[y], sf[i][y]);
#pragma unroll
                        for (int y = 0; y < 2; ++y)
                            sl[i][y] = team::fma_(sr[i][x], l[y], sl[i][y]);
                    }
                }
            }
            team::sttile<M>(SL, ri, H, 2 * ci, sl);
            R t[TR];
#pragma unroll
            for (int i = 0; i < TR; ++i) t[i] = R(0);
            if (wk.has_c) {
                R sr[TR][4];
                team::ldtile<N>(Sm, ri, H, 4 * ci, sr);
#pragma unroll
                for (int i = 0; i < TR; ++i) {
#pragma unroll
                    for (int x = 0; x < 4; ++x) t[i] = team::fma_(-sr[i][x], cv[4 * ci + x], t[i]);
                    t[i] = g.row_sum(t[i]);
                }
            }
            if (ci == 0) {
#pragma unroll
                for (int i = 0; i < TR; ++i) ev[ri + i * H] = v[ri + i * H] + t[i];
            }
        }
        g.sync();
        // G = U + L^T SL, W = SL^T F, L^T ev
        {
            R ww[TM][4], gg[TM][2];
            team::zero(ww);
            team::ldtile<M>(U, TM * ri, 1, 2 * ci, gg);
#pragma unroll(team::k_unroll(N))
            for (int kk = 0; kk < N; ++kk) {
                R f[4], l[TM], sl[TM], s2[2];
                ldrow<N, 4>(F, kk, 4 * ci, f);
                ldrow<M, TM>(L, kk, TM * ri, l);
                ldrow<M, TM>(SL, kk, TM * ri, sl);
                ldrow<M, 2>(SL, kk, 2 * ci, s2);
#pragma unroll
                for (int i = 0; i < TM; ++i) {
#pragma unroll
                    for (int y = 0; y < 4; ++y) ww[i][y] = team::fma_(sl[i], f[y], ww[i][y]);
#pragma unroll
                    for (int y = 0; y < 2; ++y) gg[i][y] = team::fma_(l[i], s2[y], gg[i][y]);
                }
            }
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                team::stsys<LD>(sy, TM * ri + i, CK + 4 * ci, ww[i]);
                team::stsys<LD>(sy, TM * ri + i, 2 * ci, gg[i]);
            }
            R lw[TM];
#pragma unroll
            for (int i = 0; i < TM; ++i) lw[i] = R(0);
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                R l[TM];
                ldrow<M, TM>(L, 4 * ci + x, TM * ri, l);
#pragma unroll
                for (int i = 0; i < TM; ++i) lw[i] = team::fma_(l[i], ev[4 * ci + x], lw[i]);
            }
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                lw[i] = g.row_sum(lw[i]);
                if (ci == 0) sy[(TM * ri + i) * LD + CD] = lw[i];
            }
        }
        g.sync();
        if (wk.hid) cost_prefetch<N, M>(cost, D, k, wk, g);
        // [K | d] = G^{-1} [W | L^T ev] in place
        ok &= team::solve_spd<true, M, N + 1>(sy, g, gi != nullptr);
        g.sync();
        // Ft = F - L K, S Ft = S F - SL K, ct = c + L d; K_k and d_k out
        {
            R ft[TR][4];
            team::ldtile<N>(F, ri, H, 4 * ci, ft);
            constexpr int EP = 16 / (int)sizeof(R), EM = EP < M ? EP : M;
#pragma unroll(team::k_unroll(M) / EM)
            for (int kk = 0; kk < M; kk += EM) {
                R lr[TR][EM], sr[TR][EM];
                team::ldtile<M>(L, ri, H, kk, lr);
                team::ldtile<M>(SL, ri, H, kk, sr);
#pragma unroll
                for (int x = 0; x < EM; ++x) {
                    R y[4];
                    team::ldsys<LD>(sy, kk + x, CK + 4 * ci, y);
#pragma unroll
                    for (int i = 0; i < TR; ++i)
#pragma unroll
                        for (int z = 0; z < 4; ++z) {
                            ft[i][z] = team::fma_(-lr[i][x], y[z], ft[i][z]);
                            sf[i][z] = team::fma_(-sr[i][x], y[z], sf[i][z]);
                        }
                }
            }
            team::sttile<N>(Ft, ri, H, 4 * ci, ft);
            team::sttile<N>(SFt, ri, H, 4 * ci, sf);
            R lr[TR][2];
            team::ldtile<M>(L, ri, H, 2 * ci, lr);
#pragma unroll
            for (int i = 0; i < TR; ++i) {
                R t = R(0);
#pragma unroll
                for (int x = 0; x < 2; ++x)
                    t = team::fma_(lr[i][x], sy[(2 * ci + x) * LD + CD], t);
                t = g.row_sum(t);
                if (ci == 0) ct[ri + i * H] = (wk.has_c ? cv[ri + i * H] : R(0)) + t;
            }
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                const int row = ri + i * H;  // a row of K; TM H = M
                // the feedforward d_k, replaced in the rollout
                if (ci == 0) D.u[k * M + row] = sy[row * LD + CD];
                if (a.out_mask & 2) {
                    R y[4];
                    team::ldsys<LD>(sy, row, CK + 4 * ci, y);
                    team::stg_row<N, 4>(D.K + k * M * N, row, 4 * ci, y, vK);
                }
                if (gi) {
                    R y[2];
                    team::ldsys<LD>(sy, row, 2 * ci, y);
                    team::stg_row<M, 2>(gi + k * M * M, row, 2 * ci, y, true);
                }
            }
        }
        g.sync();
        // S <- Q + F^T S Ft (raw into SL and the system), v <- q + Ft^T ev; Phi <- Phi Ft,
        // gamma <- gamma + Phi ct
        R ph[TR][4];
        R* raw = SL;
        {
            if (wk.hid) cost_q<N>(cost, q, g);
            if (D.eta) {
#pragma unroll
                for (int i = 0; i < TR; ++i) q[i] = D.eta[k * D.seta + TR * ri + i];
            }
            team::tn<N, N, N, false>(cost.x, F, SFt, TR * ri, 4 * ci);
            team::sttile<N>(raw, TR * ri, 1, 4 * ci, cost.x);
            if (map) {
                team::zero(ph);
                team::nn<N, N, N, false>(ph, Phi, Ft, ri, H, 4 * ci);
            }
            R t[TR], gt[TR], pr[TR][4];
            team::ldtile<N>(Phi, ri, H, 4 * ci, pr);
#pragma unroll
            for (int i = 0; i < TR; ++i) t[i] = gt[i] = R(0);
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                R f[TR];
                ldrow<N, TR>(Ft, 4 * ci + x, TR * ri, f);
                const R ex = ev[4 * ci + x], cx = ct[4 * ci + x];
#pragma unroll
                for (int i = 0; i < TR; ++i) {
                    t[i] = team::fma_(f[i], ex, t[i]);
                    gt[i] = team::fma_(pr[i][x], cx, gt[i]);
                }
            }
#pragma unroll
            for (int i = 0; i < TR; ++i) {
                t[i] = q[i] + g.row_sum(t[i]);
                gt[i] = g.row_sum(gt[i]);
                if (ci == 0) {
                    v[TR * ri + i] = t[i];
                    gm[ri + i * H] += gt[i];
                    if (a.out_mask & 4) D.v[k * N + TR * ri + i] = t[i];
                }
            }
        }
        g.sync();
        team::symmetrise<N>(cost.x, raw, g);
        team::sttile<N>(Sm, TR * ri, 1, 4 * ci, cost.x);
        if (map) team::sttile<N>(Phi, ri, H, 4 * ci, ph);
        if (a.out_mask & 1) {
#pragma unroll
            for (int i = 0; i < TR; ++i)
                team::stg_row<N, 4>(D.S + k * N * N, TR * ri + i, 4 * ci, cost.x[i], vS);
        }
    }
    g.sync();
    RT* out = a.FE + c * DAffine<N>::SIZE;
    for (int t = g.lane; t < N * N; t += LG) {
        const RT x = static_cast<RT>(Phi[Sw<R, N>::at(t / N, t % N)]);
        out[DAffine<N>::OF + t] = x;
        if (a.maps) a.maps[c * DAffine<N>::SIZE + DAffine<N>::OF + t] = x;
    }
    for (int i = g.lane; i < N; i += LG) out[DAffine<N>::OC + i] = static_cast<RT>(gm[i]);
    flag(a.status, ok);
}

template <typename R, typename RT, int N, int M, int TR, int NT, int MINB>
__global__ void __launch_bounds__(NT * Team<N, TR>::LG, MINB) k_trefold(Args<R, RT> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int gi = threadIdx.x / Team<N, TR>::LG;
    const long long c = (long long)blockIdx.x * NT + gi;
    if (c >= a.C) return;
    b_trefold<R, RT, N, M, TR>(a, c, reinterpret_cast<R*>(smem_raw) +
                                         gi * tstride_of<N, R>(TRefoldSmem<N, M>::SIZE));
}

// ---- tree levels: LV levels from spacing h0 up (or down to h0) per launch --
// A CTA's nodes are [base, base + 2 TT h0); a pair of level h exists while its
// left node is below active[level] (the chunks of the problems with NC >= 2h).
struct TreeRun {
    int levels;              // levels of this launch
    int h0;                  // spacing of its lowest level
    long long active[8];     // active[l]: level h0 << l
};

template <typename RT, int N, int TT>
__global__ void __launch_bounds__(TT* Team<N>::LG) k_tup(RT* E_, TreeRun tr, int* status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using E = DElem<N>;
    const Team<N> g;
    const int gi = threadIdx.x / Team<N>::LG;
    RT* sh = reinterpret_cast<RT*>(smem_raw) +
             gi * tstride_of<N, RT>(team::CombineSmem<N>::SIZE);
    const long long base = (long long)blockIdx.x * 2 * TT * tr.h0;
    bool ok = true;
    for (int l = 0; l < tr.levels; ++l) {
        const long long h = (long long)tr.h0 << l;
        const long long i = base + (long long)gi * 2 * h;
        if (gi < (TT >> l) && i < tr.active[l])
            ok &= team::combine<N>(E_ + i * E::SIZE, E_ + (i + h) * E::SIZE, E_ + i * E::SIZE, sh,
                                   g);
        __syncthreads();
    }
    flag(status, ok);
}

template <typename RT, int N, int TT>
__global__ void __launch_bounds__(TT* Team<N>::LG)
    k_tdown(const RT* E_, RT* V_, TreeRun tr, int* status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using E = DElem<N>;
    using V = DValue<N>;
    const Team<N> g;
    const int gi = threadIdx.x / Team<N>::LG;
    RT* sh = reinterpret_cast<RT*>(smem_raw) + gi * tstride_of<N, RT>(team::ApplySmem<N>::SIZE);
    const long long base = (long long)blockIdx.x * 2 * TT * tr.h0;
    bool ok = true;
    for (int l = tr.levels - 1; l >= 0; --l) {
        const long long h = (long long)tr.h0 << l;
        const long long i = base + (long long)gi * 2 * h;
        if (gi < (TT >> l) && i < tr.active[l]) {
            // the right half keeps the parent's value, the left half gets it
            // through the right half's element
            for (int t = g.lane; t < V::SIZE; t += Team<N>::LG)
                V_[(i + h) * V::SIZE + t] = V_[i * V::SIZE + t];
            ok &= team::value_apply<N>(E_ + (i + h) * E::SIZE, V_ + i * V::SIZE, V_ + i * V::SIZE,
                                       sh, g);
        }
        __syncthreads();
    }
    flag(status, ok);
}

// forward maps, right-anchored: FE[j] <- FE[j] o FE[j - h], j = 2h q + 2h - 1
template <typename RT, int N, int TT>
__global__ void __launch_bounds__(TT* Team<N>::LG) k_tfup(RT* FE, TreeRun tr) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using A = DAffine<N>;
    const Team<N> g;
    const int gi = threadIdx.x / Team<N>::LG;
    RT* sh = reinterpret_cast<RT*>(smem_raw) + gi * tstride_of<N, RT>(2 * N * N);
    const long long base = (long long)blockIdx.x * 2 * TT * tr.h0;
    for (int l = 0; l < tr.levels; ++l) {
        const long long h = (long long)tr.h0 << l;
        const long long j = base + (long long)gi * 2 * h + 2 * h - 1;
        if (gi < (TT >> l) && j < tr.active[l])
            team::affine_compose<N>(FE + (j - h) * A::SIZE, FE + j * A::SIZE, FE + j * A::SIZE, sh,
                                    g);
        __syncthreads();
    }
}

// X[j - h] <- X[j]; X[j] <- FE[j - h](X[j])
template <typename RT, int N, int TT>
__global__ void __launch_bounds__(TT* Team<N>::LG) k_tfdown(const RT* FE, RT* X, TreeRun tr) {
    using A = DAffine<N>;
    const Team<N> g;
    const int gi = threadIdx.x / Team<N>::LG;
    const long long base = (long long)blockIdx.x * 2 * TT * tr.h0;
    for (int l = tr.levels - 1; l >= 0; --l) {
        const long long h = (long long)tr.h0 << l;
        const long long j = base + (long long)gi * 2 * h + 2 * h - 1;
        const bool act = gi < (TT >> l) && j < tr.active[l];
        RT y0 = RT(0), y1 = RT(0);
        if (act) {
            for (int i = g.lane; i < N; i += Team<N>::LG) X[(j - h) * N + i] = X[j * N + i];
            team::affine_apply<N>(FE + (j - h) * A::SIZE, X + j * N, y0, y1, g);
        }
        __syncthreads();  // every lane has read X[j]
        if (act && g.ci == 0) {
            X[j * N + g.ri] = y0;
            X[j * N + g.ri + N / 2] = y1;
        }
        __syncthreads();
    }
}

}  // namespace chain
}  // namespace lqt
