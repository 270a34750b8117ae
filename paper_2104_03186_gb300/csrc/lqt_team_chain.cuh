// Chunk and tree-level kernels of the chunked pipeline (lqt_chain.cuh) at
// n = 8, 16, 32: the team algebra of lqt_team.cuh.  Included by lqt_chain.cuh.
//
// k_tfold and k_trefold walk a chunk's steps; a step's F, L, U, c come by
// cp.async into one of two buffers while the step before is computed, and with
// H = I the tile of X_k and r_k goes straight to registers.  k_tup, k_tdown,
// k_tfup, k_tfdown run several tree levels per launch: a CTA of TT teams owns
// 2 TT neighbouring nodes, and its teams meet at a CTA barrier between the
// levels, where the global-memory results of one level are read by the next.
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
template <int ROWS, int COLS, int N, typename R>
__device__ __forceinline__ void cp_mat(R* dst, const R* src, bool vec, const Team<N>& g) {
    constexpr int E = 16 / (int)sizeof(R), RC = COLS / E, LG = Team<N>::LG;
    if (vec) {
#pragma unroll
        for (int t = g.lane; t < ROWS * RC; t += LG)
            cp_async<16>(dst + Sw<R, COLS>::chunk(t / RC, t % RC), src + t * E);
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

// What a chunk walk knows about its problem's arrays.
template <typename R, int N, int M>
struct TeamWalk {
    bool vF, vL, vU, vX, vr, hid, has_c, u_once;
    __device__ TeamWalk(const DescT<R>& D, const Team<N>& g) {
        vF = vec_ok(D.F, D.sF);
        vL = vec_ok(D.L, D.sL);
        vU = vec_ok(D.U, D.sU);
        vX = vec_ok(D.X, D.sX);
        vr = D.r && vec_ok(D.r, D.sr);
        has_c = D.c != nullptr;
        u_once = D.sU == 0;
        // H = I at every step (p = N): every warp of the team looks at all of H
        bool mine = D.sH == 0 && D.p == N && D.H;
        if (mine)
            for (int t = g.lane % Team<N>::LW; t < N * N; t += Team<N>::LW)
                mine = mine && D.H[t] == (t / N == t % N ? R(1) : R(0));
        hid = __all_sync(g.mask, mine);
    }
    __device__ __forceinline__ void stage(const DescT<R>& D, long long k, R* in, int b, bool first,
                                          const Team<N>& g) const {
        using I = TeamIn<N, M>;
        cp_mat<N, N>(in + I::F + b * N * N, D.F + k * D.sF, vF, g);
        cp_mat<N, M>(in + I::L + b * N * M, D.L + k * D.sL, vL, g);
        if (first || !u_once) cp_mat<M, M>(in + I::U + b * M * M, D.U + k * D.sU, vU, g);
        if (has_c)
            for (int i = g.lane; i < N; i += Team<N>::LG)
                cp_async<sizeof(R)>(in + I::C + b * N + i, D.c + k * D.sc + i);
        cp_async_commit();
    }
};

// Q_k = H^T X H (TN tile) and the entries of q_k = H^T X r a lane needs.
template <typename R>
struct CostTile {
    R x[2][4], r[4];
};

// H = I: the tile of X_k and four entries of r_k from global memory
template <int N, int M, typename R>
__device__ __forceinline__ void cost_prefetch(CostTile<R>& ct, const DescT<R>& D, long long k,
                                              const TeamWalk<R, N, M>& w, const Team<N>& g) {
    const R* X = D.X + k * D.sX;
    team::ldg_row<N, 4>(X, 2 * g.ri, 4 * g.ci, ct.x[0], w.vX);
    team::ldg_row<N, 4>(X, 2 * g.ri + 1, 4 * g.ci, ct.x[1], w.vX);
    if (D.r && !D.eta) {
        team::ldg_row<N, 4>(D.r + k * D.sr, 0, 4 * g.ci, ct.r, w.vr);
    } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) ct.r[c] = R(0);
    }
}

// General H and X: Y = X H and X r in the scratch (p <= 2N; with p <= N also H
// and X staged there), then the TN tile of H^T Y and rows 2 ri, 2 ri + 1 of
// H^T X r.  scr: 3 N^2 + 3 N elements.  Ends with a sync.
template <int N, typename R>
__device__ void cost_general(R (&x)[2][4], R& q0, R& q1, const DescT<R>& D, long long k, R* scr,
                             const Team<N>& g) {
    const int p = D.p, ri = g.ri, ci = g.ci;
    const bool staged = p <= N;
    R* Y = scr;  // p x N
    R* xr = scr + 3 * N * N + N;
    const int lp = staged ? p | 1 : p;  // row stride of X: odd where it is staged
    const R* X = D.X + k * D.sX;
    const R* H = D.H + k * D.sH;
    const R* rk = D.r ? D.r + k * D.sr : nullptr;
    if (staged) {
        R* Hs = scr + N * N;
        R* Xs = scr + 2 * N * N;
        for (int t = g.lane; t < p * N; t += Team<N>::LG) cp_async<sizeof(R)>(Hs + t, H + t);
        for (int i = ri; i < p; i += N / 2)
            for (int j = ci; j < p; j += N / 4) cp_async<sizeof(R)>(Xs + i * lp + j, X + i * p + j);
        cp_async_commit();
        cp_async_wait<0>();
        H = Hs;
        X = Xs;
    }
    g.sync();
    for (int i = ri; i < p; i += N / 2) {
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
    q0 = q1 = R(0);
#pragma unroll 4
    for (int i = 0; i < p; ++i) {
        const R h0 = H[i * N + 2 * ri], h1 = H[i * N + 2 * ri + 1];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const R y = Y[i * N + 4 * ci + c];
            x[0][c] = team::fma_(h0, y, x[0][c]);
            x[1][c] = team::fma_(h1, y, x[1][c]);
        }
        q0 = team::fma_(h0, xr[i], q0);
        q1 = team::fma_(h1, xr[i], q1);
    }
    g.sync();
}

// q rows 2 ri, 2 ri + 1 with H = I (every lane of the row gets them)
template <int N, typename R>
__device__ __forceinline__ void cost_q(const CostTile<R>& ct, R& q0, R& q1, const Team<N>& g) {
    q0 = q1 = R(0);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        q0 = team::fma_(ct.x[0][c], ct.r[c], q0);
        q1 = team::fma_(ct.x[1][c], ct.r[c], q1);
    }
    q0 = g.row_sum(q0);
    q1 = g.row_sum(q1);
}

// Shared memory of one team (elements): the running total P | staged inputs |
// JF, JL, P2, Z, Zt, Pt, G | vectors.
template <int N, int M>
struct TFoldSmem {
    static constexpr int PA = 0, PC = N * N, PJ = 2 * N * N, IN = 3 * N * N,
                         JF = IN + TeamIn<N, M>::SIZE, JL = JF + N * N, P2 = JL + N * M,
                         Z = P2 + N * M, ZT = Z + M * N, PT = ZT + M * N, G = PT + M * N,
                         V = G + M * M, PB = V, PE = PB + N, W = PE + N, AC = W + N,
                         OM = AC + N, SIZE = OM + M;
    static_assert(N < 8 || G - JF >= 3 * N * N + 3 * N, "cost_general's scratch");
    static_assert(IN % 4 == 0 && JF % 4 == 0 && V % 4 == 0, "16-byte matrices");
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
//   Z = L^T J F, G = U + L^T J L, w = eta - J c, P2 = A L,
//   [Zt | om | Pt] = G^{-1} [Z | L^T w | P2^T],
//   A <- A F - P2 Zt, b <- A c + P2 om + b, C <- C + P2 Pt,
//   J <- H^T X H + F^T J F - Z^T Zt, eta <- q + F^T w - Z^T om.
template <typename R, typename RT, int N, int M>
__device__ __forceinline__ void b_tfold(const Args<R, RT>& a, long long c, R* sh) {
    static_assert(M == N / 2, "tiles of L, K and G assume m = n / 2");
    using S = TFoldSmem<N, M>;
    using I = TeamIn<N, M>;
    using E = DElem<N>;
    constexpr int H = N / 2;
    const Team<N> g;
    const int ri = g.ri, ci = g.ci;
    const Item<R>& it = a.items[find_chunk(a.items, a.count, c)];
    const DescT<R>& D = it.D;
    R *PA = sh + S::PA, *PC = sh + S::PC, *PJ = sh + S::PJ;
    R *b = sh + S::PB, *e = sh + S::PE, *w = sh + S::W, *ac = sh + S::AC, *om = sh + S::OM;
    R *JF = sh + S::JF, *JL = sh + S::JL, *P2 = sh + S::P2, *Z = sh + S::Z, *ZT = sh + S::ZT,
      *PT = sh + S::PT, *G = sh + S::G;
    const long long T = D.T;
    const long long lc = c - it.c0;
    const long long s0 = lc * it.B < T ? lc * it.B : T;
    const long long e0 = s0 + it.B < T ? s0 + it.B : T;
    const TeamWalk<R, N, M> wk(D, g);
    CostTile<R> next;
    if (s0 < e0) {
        wk.stage(D, e0 - 1, sh + S::IN, 0, true, g);
        if (wk.hid) cost_prefetch<N, M>(next, D, e0 - 1, wk, g);
    }
    {
        R z[4] = {R(0), R(0), R(0), R(0)}, o[4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = ri + h * H;
#pragma unroll
            for (int q = 0; q < 4; ++q) o[q] = row == 4 * ci + q ? R(1) : R(0);
            strow<N, 4>(PA, row, 4 * ci, o);
            strow<N, 4>(PC, row, 4 * ci, z);
            strow<N, 4>(PJ, row, 4 * ci, z);
            if (ci == 0) b[row] = e[row] = R(0);
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
        g.sync();  // the inputs are in; the step before is done with the other buffer
        CostTile<R> now = next;
        R q0, q1;
        if (k > s0) wk.stage(D, k - 1, sh + S::IN, cur ^ 1, false, g);
        if (wk.hid) {
            if (k > s0) cost_prefetch<N, M>(next, D, k - 1, wk, g);
            cost_q<N>(now, q0, q1, g);
        } else {
            cost_general<N>(now.x, q0, q1, D, k, sh + S::JF, g);
        }
        if (D.eta) {
            q0 = D.eta[k * D.seta + 2 * ri];
            q1 = D.eta[k * D.seta + 2 * ri + 1];
        }
        // JF = J F, JL = J L, P2 = A L to shared memory, A F in registers
        R af[2][4];
        {
            R jf[2][4], jl[2][2], al[2][2];
            team::zero(af);
            team::zero(jf);
            team::zero(jl);
            team::zero(al);
            constexpr int EP = 16 / (int)sizeof(R);
#pragma unroll(team::k_unroll(N) / EP)
            for (int kk = 0; kk < N; kk += EP) {
                R j0[EP], j1[EP], a0[EP], a1[EP];
                ldrow<N, EP>(PJ, ri, kk, j0);
                ldrow<N, EP>(PJ, ri + H, kk, j1);
                ldrow<N, EP>(PA, ri, kk, a0);
                ldrow<N, EP>(PA, ri + H, kk, a1);
#pragma unroll
                for (int q = 0; q < EP; ++q) {
                    R f[4], l[2];
                    ldrow<N, 4>(F, kk + q, 4 * ci, f);
                    ldrow<M, 2>(L, kk + q, 2 * ci, l);
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        jf[0][x] = team::fma_(j0[q], f[x], jf[0][x]);
                        jf[1][x] = team::fma_(j1[q], f[x], jf[1][x]);
                        af[0][x] = team::fma_(a0[q], f[x], af[0][x]);
                        af[1][x] = team::fma_(a1[q], f[x], af[1][x]);
                    }
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
                        jl[0][x] = team::fma_(j0[q], l[x], jl[0][x]);
                        jl[1][x] = team::fma_(j1[q], l[x], jl[1][x]);
                        al[0][x] = team::fma_(a0[q], l[x], al[0][x]);
                        al[1][x] = team::fma_(a1[q], l[x], al[1][x]);
                    }
                }
            }
            strow<N, 4>(JF, ri, 4 * ci, jf[0]);
            strow<N, 4>(JF, ri + H, 4 * ci, jf[1]);
            strow<M, 2>(JL, ri, 2 * ci, jl[0]);
            strow<M, 2>(JL, ri + H, 2 * ci, jl[1]);
            strow<M, 2>(P2, ri, 2 * ci, al[0]);
            strow<M, 2>(P2, ri + H, 2 * ci, al[1]);
            if (wk.has_c) {
                R j0[4], j1[4], a0[4], a1[4], s[4] = {R(0), R(0), R(0), R(0)};
                ldrow<N, 4>(PJ, ri, 4 * ci, j0);
                ldrow<N, 4>(PJ, ri + H, 4 * ci, j1);
                ldrow<N, 4>(PA, ri, 4 * ci, a0);
                ldrow<N, 4>(PA, ri + H, 4 * ci, a1);
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const R cx = cv[4 * ci + x];
                    s[0] = team::fma_(-j0[x], cx, s[0]);
                    s[1] = team::fma_(-j1[x], cx, s[1]);
                    s[2] = team::fma_(a0[x], cx, s[2]);
                    s[3] = team::fma_(a1[x], cx, s[3]);
                }
#pragma unroll
                for (int x = 0; x < 4; ++x) s[x] = g.row_sum(s[x]);
                if (ci == 0) {
                    w[ri] = e[ri] + s[0];
                    w[ri + H] = e[ri + H] + s[1];
                    ac[ri] = s[2];
                    ac[ri + H] = s[3];
                }
            } else if (ci == 0) {
                w[ri] = e[ri];
                w[ri + H] = e[ri + H];
                ac[ri] = ac[ri + H] = R(0);
            }
        }
        g.sync();
        // G = U + L^T JL, Z = L^T JF (row ri); L^T w; J1 + F^T JF (rows 2 ri,
        // 2 ri + 1) and F^T w in registers
        R fw0 = R(0), fw1 = R(0);
        {
            R zz[4] = {R(0), R(0), R(0), R(0)}, gg[2];
            ldrow<M, 2>(U, ri, 2 * ci, gg);
#pragma unroll(team::k_unroll(N))
            for (int kk = 0; kk < N; ++kk) {
                R f[2], l[1], jf[4], jl[2];
                ldrow<N, 2>(F, kk, 2 * ri, f);
                ldrow<M, 1>(L, kk, ri, l);
                ldrow<N, 4>(JF, kk, 4 * ci, jf);
                ldrow<M, 2>(JL, kk, 2 * ci, jl);
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    now.x[0][x] = team::fma_(f[0], jf[x], now.x[0][x]);
                    now.x[1][x] = team::fma_(f[1], jf[x], now.x[1][x]);
                    zz[x] = team::fma_(l[0], jf[x], zz[x]);
                }
                gg[0] = team::fma_(l[0], jl[0], gg[0]);
                gg[1] = team::fma_(l[0], jl[1], gg[1]);
            }
            strow<N, 4>(Z, ri, 4 * ci, zz);
            strow<M, 2>(G, ri, 2 * ci, gg);
            R lw = R(0);
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const int kk = 4 * ci + x;
                const R wx = w[kk];
                R f[2], l[1];
                ldrow<N, 2>(F, kk, 2 * ri, f);
                ldrow<M, 1>(L, kk, ri, l);
                fw0 = team::fma_(f[0], wx, fw0);
                fw1 = team::fma_(f[1], wx, fw1);
                lw = team::fma_(l[0], wx, lw);
            }
            lw = g.row_sum(lw);
            if (ci == 0) om[ri] = lw;
        }
        g.sync();
        // [Zt | Pt | om] = G^{-1} [Z | P2^T | L^T w]
        ok &= team::solve_spd<M, 2 * N + 1>(
            G, g,
            [&](int r, R(&col)[M]) {
                if (r < N) {
#pragma unroll
                    for (int i = 0; i < M; ++i) col[i] = Z[Sw<R, N>::at(i, r)];
                } else if (r < 2 * N) {
#pragma unroll
                    for (int i = 0; i < M; i += 2) {
                        R x[2];
                        ldrow<M, 2>(P2, r - N, i, x);
                        col[i] = x[0];
                        col[i + 1] = x[1];
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < M; ++i) col[i] = om[i];
                }
            },
            [&](int r, const R(&col)[M]) {
                if (r < 2 * N) {
                    R* o = r < N ? ZT : PT;
#pragma unroll
                    for (int i = 0; i < M; ++i) o[Sw<R, N>::at(i, r & (N - 1))] = col[i];
                } else {
#pragma unroll
                    for (int i = 0; i < M; ++i) om[i] = col[i];
                }
            });
        g.sync();
        // A, C (rows ri, ri + H), J (rows 2 ri, 2 ri + 1), b, eta; raw C into JF
        // and raw J into the step's F, which nothing reads any more
        R* rawC = JF;
        R* rawJ = sh + S::IN + I::F + cur * N * N;
        {
            R cc[2][4];
            ldrow<N, 4>(PC, ri, 4 * ci, cc[0]);
            ldrow<N, 4>(PC, ri + H, 4 * ci, cc[1]);
            constexpr int EP = 16 / (int)sizeof(R), EM = EP < M ? EP : M;
#pragma unroll
            for (int kk = 0; kk < M; kk += EM) {
                R p0[EM], p1[EM];
                ldrow<M, EM>(P2, ri, kk, p0);
                ldrow<M, EM>(P2, ri + H, kk, p1);
#pragma unroll
                for (int q = 0; q < EM; ++q) {
                    R zt[4], pt[4], z[2];
                    ldrow<N, 4>(ZT, kk + q, 4 * ci, zt);
                    ldrow<N, 4>(PT, kk + q, 4 * ci, pt);
                    ldrow<N, 2>(Z, kk + q, 2 * ri, z);
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        af[0][x] = team::fma_(-p0[q], zt[x], af[0][x]);
                        af[1][x] = team::fma_(-p1[q], zt[x], af[1][x]);
                        cc[0][x] = team::fma_(p0[q], pt[x], cc[0][x]);
                        cc[1][x] = team::fma_(p1[q], pt[x], cc[1][x]);
                        now.x[0][x] = team::fma_(-z[0], zt[x], now.x[0][x]);
                        now.x[1][x] = team::fma_(-z[1], zt[x], now.x[1][x]);
                    }
                }
            }
            R s0 = R(0), s1 = R(0), p0[2], p1[2];
            ldrow<M, 2>(P2, ri, 2 * ci, p0);
            ldrow<M, 2>(P2, ri + H, 2 * ci, p1);
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                const R o = om[2 * ci + x];
                R z[2];
                ldrow<N, 2>(Z, 2 * ci + x, 2 * ri, z);
                s0 = team::fma_(p0[x], o, s0);
                s1 = team::fma_(p1[x], o, s1);
                fw0 = team::fma_(-z[0], o, fw0);
                fw1 = team::fma_(-z[1], o, fw1);
            }
            s0 = g.row_sum(s0);
            s1 = g.row_sum(s1);
            fw0 = g.row_sum(fw0);
            fw1 = g.row_sum(fw1);
            if (ci == 0) {
                b[ri] += ac[ri] + s0;
                b[ri + H] += ac[ri + H] + s1;
                e[2 * ri] = q0 + fw0;
                e[2 * ri + 1] = q1 + fw1;
            }
            strow<N, 4>(PA, ri, 4 * ci, af[0]);
            strow<N, 4>(PA, ri + H, 4 * ci, af[1]);
            strow<N, 4>(rawC, ri, 4 * ci, cc[0]);
            strow<N, 4>(rawC, ri + H, 4 * ci, cc[1]);
            strow<N, 4>(rawJ, 2 * ri, 4 * ci, now.x[0]);
            strow<N, 4>(rawJ, 2 * ri + 1, 4 * ci, now.x[1]);
        }
        g.sync();
        {
            R cc[2][4];
            ldrow<N, 4>(rawC, 2 * ri, 4 * ci, cc[0]);
            ldrow<N, 4>(rawC, 2 * ri + 1, 4 * ci, cc[1]);
            team::symmetrise<N>(cc, rawC, g);
            team::symmetrise<N>(now.x, rawJ, g);
            strow<N, 4>(PC, 2 * ri, 4 * ci, cc[0]);
            strow<N, 4>(PC, 2 * ri + 1, 4 * ci, cc[1]);
            strow<N, 4>(PJ, 2 * ri, 4 * ci, now.x[0]);
            strow<N, 4>(PJ, 2 * ri + 1, 4 * ci, now.x[1]);
        }
    }
    g.sync();
    RT* out = a.E + c * E::SIZE;
    for (int t = g.lane; t < N * N; t += Team<N>::LG) {
        const int q = Sw<R, N>::at(t / N, t % N);
        out[E::OA + t] = static_cast<RT>(PA[q]);
        out[E::OC + t] = static_cast<RT>(PC[q]);
        out[E::OJ + t] = static_cast<RT>(PJ[q]);
    }
    for (int i = g.lane; i < N; i += Team<N>::LG) {
        out[E::OB + i] = static_cast<RT>(b[i]);
        out[E::OE + i] = static_cast<RT>(e[i]);
    }
    flag(a.status, ok);
}

template <typename R, typename RT, int N, int M, int NT, int MINB>
__global__ void __launch_bounds__(NT * Team<N>::LG, MINB) k_tfold(Args<R, RT> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int gi = threadIdx.x / Team<N>::LG;
    const long long c = (long long)blockIdx.x * NT + gi;
    if (c >= a.C) return;
    b_tfold<R, RT, N, M>(a, c, reinterpret_cast<R*>(smem_raw) +
                                   gi * tstride_of<N, R>(TFoldSmem<N, M>::SIZE));
}

// ---- per-chunk Riccati re-fold with outputs and the chunk affine map -------
template <int N, int M>
struct TRefoldSmem {
    static constexpr int SV = 0, PHI = N * N, IN = 2 * N * N, SL = IN + TeamIn<N, M>::SIZE,
                         FT = SL + N * M, SFT = FT + N * N, W = SFT + N * N, K = W + M * N,
                         G = K + M * N, V = G + M * M, VV = V, EV = VV + N, GM = EV + N,
                         CT = GM + N, DD = CT + N, SIZE = DD + M;
    static_assert(N < 8 || G - SL >= 3 * N * N + 3 * N, "cost_general's scratch");
    static_assert(SL % 4 == 0 && V % 4 == 0, "16-byte matrices");
};

template <typename R, typename RT, int N, int M>
__device__ __forceinline__ void b_trefold(const Args<R, RT>& a, long long c, R* sh) {
    using S = TRefoldSmem<N, M>;
    using I = TeamIn<N, M>;
    constexpr int H = N / 2, LG = Team<N>::LG;
    const Team<N> g;
    const int ri = g.ri, ci = g.ci;
    const Item<R>& it = a.items[find_chunk(a.items, a.count, c)];
    const DescT<R>& D = it.D;
    R *Sm = sh + S::SV, *Phi = sh + S::PHI, *SL = sh + S::SL, *Ft = sh + S::FT, *SFt = sh + S::SFT,
      *W = sh + S::W, *K = sh + S::K, *G = sh + S::G;
    R *v = sh + S::VV, *ev = sh + S::EV, *gm = sh + S::GM, *ct = sh + S::CT, *dd = sh + S::DD;
    const long long T = D.T;
    const long long lc = c - it.c0;
    const long long s0 = lc * it.B < T ? lc * it.B : T;
    const long long e0 = s0 + it.B < T ? s0 + it.B : T;
    const TeamWalk<R, N, M> wk(D, g);
    const bool vS = vec_ok(D.S, 0), vK = vec_ok(D.K, 0);
    CostTile<R> next;
    if (s0 < e0) {
        wk.stage(D, e0 - 1, sh + S::IN, 0, true, g);
        if (wk.hid) cost_prefetch<N, M>(next, D, e0 - 1, wk, g);
    }
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
        CostTile<R> now = next;
        R q0, q1;
        if (k > s0) wk.stage(D, k - 1, sh + S::IN, cur ^ 1, false, g);
        if (wk.hid) {
            if (k > s0) cost_prefetch<N, M>(next, D, k - 1, wk, g);
            cost_q<N>(now, q0, q1, g);
        } else {
            cost_general<N>(now.x, q0, q1, D, k, SL, g);
        }
        if (D.eta) {
            q0 = D.eta[k * D.seta + 2 * ri];
            q1 = D.eta[k * D.seta + 2 * ri + 1];
        }
        // S F in registers, S L to shared memory, ev = v - S c
        R sf[2][4];
        {
            R sl[2][2];
            team::zero(sf);
            team::zero(sl);
            constexpr int EP = 16 / (int)sizeof(R);
#pragma unroll(team::k_unroll(N) / EP)
            for (int kk = 0; kk < N; kk += EP) {
                R x0[EP], x1[EP];
                ldrow<N, EP>(Sm, ri, kk, x0);
                ldrow<N, EP>(Sm, ri + H, kk, x1);
#pragma unroll
                for (int q = 0; q < EP; ++q) {
                    R f[4], l[2];
                    ldrow<N, 4>(F, kk + q, 4 * ci, f);
                    ldrow<M, 2>(L, kk + q, 2 * ci, l);
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        sf[0][x] = team::fma_(x0[q], f[x], sf[0][x]);
                        sf[1][x] = team::fma_(x1[q], f[x], sf[1][x]);
                    }
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
                        sl[0][x] = team::fma_(x0[q], l[x], sl[0][x]);
                        sl[1][x] = team::fma_(x1[q], l[x], sl[1][x]);
                    }
                }
            }
            strow<M, 2>(SL, ri, 2 * ci, sl[0]);
            strow<M, 2>(SL, ri + H, 2 * ci, sl[1]);
            R t0 = R(0), t1 = R(0);
            if (wk.has_c) {
                R x0[4], x1[4];
                ldrow<N, 4>(Sm, ri, 4 * ci, x0);
                ldrow<N, 4>(Sm, ri + H, 4 * ci, x1);
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const R cx = cv[4 * ci + x];
                    t0 = team::fma_(-x0[x], cx, t0);
                    t1 = team::fma_(-x1[x], cx, t1);
                }
                t0 = g.row_sum(t0);
                t1 = g.row_sum(t1);
            }
            if (ci == 0) {
                ev[ri] = v[ri] + t0;
                ev[ri + H] = v[ri + H] + t1;
            }
        }
        g.sync();
        // G = U + L^T SL, W = SL^T F (row ri), L^T ev
        {
            R ww[4] = {R(0), R(0), R(0), R(0)}, gg[2];
            ldrow<M, 2>(U, ri, 2 * ci, gg);
#pragma unroll(team::k_unroll(N))
            for (int kk = 0; kk < N; ++kk) {
                R f[4], l[1], sl[1], s2[2];
                ldrow<N, 4>(F, kk, 4 * ci, f);
                ldrow<M, 1>(L, kk, ri, l);
                ldrow<M, 1>(SL, kk, ri, sl);
                ldrow<M, 2>(SL, kk, 2 * ci, s2);
#pragma unroll
                for (int x = 0; x < 4; ++x) ww[x] = team::fma_(sl[0], f[x], ww[x]);
                gg[0] = team::fma_(l[0], s2[0], gg[0]);
                gg[1] = team::fma_(l[0], s2[1], gg[1]);
            }
            strow<N, 4>(W, ri, 4 * ci, ww);
            strow<M, 2>(G, ri, 2 * ci, gg);
            R lw = R(0);
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                R l[1];
                ldrow<M, 1>(L, 4 * ci + x, ri, l);
                lw = team::fma_(l[0], ev[4 * ci + x], lw);
            }
            lw = g.row_sum(lw);
            if (ci == 0) dd[ri] = lw;
        }
        g.sync();
        ok &= team::solve_spd<M, N + 1>(
            G, g,
            [&](int r, R(&col)[M]) {
                if (r < N) {
#pragma unroll
                    for (int i = 0; i < M; ++i) col[i] = W[Sw<R, N>::at(i, r)];
                } else {
#pragma unroll
                    for (int i = 0; i < M; ++i) col[i] = dd[i];
                }
            },
            [&](int r, const R(&col)[M]) {
                if (r < N) {
#pragma unroll
                    for (int i = 0; i < M; ++i) K[Sw<R, N>::at(i, r)] = col[i];
                } else {
#pragma unroll
                    for (int i = 0; i < M; ++i) dd[i] = col[i];
                }
            });
        g.sync();
        // Ft = F - L K, S Ft = S F - SL K, ct = c + L d; K_k and d_k out
        {
            R ft[2][4];
            ldrow<N, 4>(F, ri, 4 * ci, ft[0]);
            ldrow<N, 4>(F, ri + H, 4 * ci, ft[1]);
            constexpr int EP = 16 / (int)sizeof(R), EM = EP < M ? EP : M;
#pragma unroll
            for (int kk = 0; kk < M; kk += EM) {
                R l0[EM], l1[EM], x0[EM], x1[EM];
                ldrow<M, EM>(L, ri, kk, l0);
                ldrow<M, EM>(L, ri + H, kk, l1);
                ldrow<M, EM>(SL, ri, kk, x0);
                ldrow<M, EM>(SL, ri + H, kk, x1);
#pragma unroll
                for (int q = 0; q < EM; ++q) {
                    R y[4];
                    ldrow<N, 4>(K, kk + q, 4 * ci, y);
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        ft[0][x] = team::fma_(-l0[q], y[x], ft[0][x]);
                        ft[1][x] = team::fma_(-l1[q], y[x], ft[1][x]);
                        sf[0][x] = team::fma_(-x0[q], y[x], sf[0][x]);
                        sf[1][x] = team::fma_(-x1[q], y[x], sf[1][x]);
                    }
                }
            }
            strow<N, 4>(Ft, ri, 4 * ci, ft[0]);
            strow<N, 4>(Ft, ri + H, 4 * ci, ft[1]);
            strow<N, 4>(SFt, ri, 4 * ci, sf[0]);
            strow<N, 4>(SFt, ri + H, 4 * ci, sf[1]);
            R t0 = R(0), t1 = R(0), l0[2], l1[2];
            ldrow<M, 2>(L, ri, 2 * ci, l0);
            ldrow<M, 2>(L, ri + H, 2 * ci, l1);
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                t0 = team::fma_(l0[x], dd[2 * ci + x], t0);
                t1 = team::fma_(l1[x], dd[2 * ci + x], t1);
            }
            t0 = g.row_sum(t0);
            t1 = g.row_sum(t1);
            if (ci == 0) {
                ct[ri] = (wk.has_c ? cv[ri] : R(0)) + t0;
                ct[ri + H] = (wk.has_c ? cv[ri + H] : R(0)) + t1;
                D.u[k * M + ri] = dd[ri];  // feedforward, replaced in the rollout
            }
            if (a.out_mask & 2) {
                R y[4];
                ldrow<N, 4>(K, ri, 4 * ci, y);
                team::stg_row<N, 4>(D.K + k * M * N, ri, 4 * ci, y, vK);
            }
        }
        g.sync();
        // S <- Q + F^T S Ft (raw into [W | K]), v <- q + Ft^T ev; Phi <- Phi Ft,
        // gamma <- gamma + Phi ct
        R ph[2][4];
        R* raw = W;
        {
            team::tn<N, N, N, 2, 4, false>(now.x, F, SFt, 2 * ri, 4 * ci);
            strow<N, 4>(raw, 2 * ri, 4 * ci, now.x[0]);
            strow<N, 4>(raw, 2 * ri + 1, 4 * ci, now.x[1]);
            team::zero(ph);
            team::nn<N, N, N, 4, false>(ph[0], ph[1], Phi, Ft, ri, ri + H, 4 * ci);
            R t0 = R(0), t1 = R(0), g0 = R(0), g1 = R(0), p0[4], p1[4];
            ldrow<N, 4>(Phi, ri, 4 * ci, p0);
            ldrow<N, 4>(Phi, ri + H, 4 * ci, p1);
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                R f[2];
                ldrow<N, 2>(Ft, 4 * ci + x, 2 * ri, f);
                const R ex = ev[4 * ci + x], cx = ct[4 * ci + x];
                t0 = team::fma_(f[0], ex, t0);
                t1 = team::fma_(f[1], ex, t1);
                g0 = team::fma_(p0[x], cx, g0);
                g1 = team::fma_(p1[x], cx, g1);
            }
            t0 = g.row_sum(t0);
            t1 = g.row_sum(t1);
            g0 = g.row_sum(g0);
            g1 = g.row_sum(g1);
            if (ci == 0) {
                v[2 * ri] = q0 + t0;
                v[2 * ri + 1] = q1 + t1;
                gm[ri] += g0;
                gm[ri + H] += g1;
                if (a.out_mask & 4) {
                    D.v[k * N + 2 * ri] = q0 + t0;
                    D.v[k * N + 2 * ri + 1] = q1 + t1;
                }
            }
        }
        g.sync();
        team::symmetrise<N>(now.x, raw, g);
        strow<N, 4>(Sm, 2 * ri, 4 * ci, now.x[0]);
        strow<N, 4>(Sm, 2 * ri + 1, 4 * ci, now.x[1]);
        strow<N, 4>(Phi, ri, 4 * ci, ph[0]);
        strow<N, 4>(Phi, ri + H, 4 * ci, ph[1]);
        if (a.out_mask & 1) {
            team::stg_row<N, 4>(D.S + k * N * N, 2 * ri, 4 * ci, now.x[0], vS);
            team::stg_row<N, 4>(D.S + k * N * N, 2 * ri + 1, 4 * ci, now.x[1], vS);
        }
    }
    g.sync();
    RT* out = a.FE + c * DAffine<N>::SIZE;
    for (int t = g.lane; t < N * N; t += LG)
        out[DAffine<N>::OF + t] = static_cast<RT>(Phi[Sw<R, N>::at(t / N, t % N)]);
    for (int i = g.lane; i < N; i += LG) out[DAffine<N>::OC + i] = static_cast<RT>(gm[i]);
    flag(a.status, ok);
}

template <typename R, typename RT, int N, int M, int NT, int MINB>
__global__ void __launch_bounds__(NT * Team<N>::LG, MINB) k_trefold(Args<R, RT> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int gi = threadIdx.x / Team<N>::LG;
    const long long c = (long long)blockIdx.x * NT + gi;
    if (c >= a.C) return;
    b_trefold<R, RT, N, M>(a, c, reinterpret_cast<R*>(smem_raw) +
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
