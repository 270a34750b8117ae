// Team algebra for the LQT operators at n = 8, 16, 32 (m = n / 2), in the
// arithmetic type R.
//
// A team of LG = N^2 / 8 lanes (8, 32 or 128) owns one element; its matrices
// live in shared memory and every N x N product is cut into 2 x 4 register
// tiles, one per lane: a step of k reads two left entries and four right ones
// for eight FMAs, in 128-bit loads along k (left) and along the columns
// (right).  A lane that owned a whole row would read one shared word per FMA,
// and the shared-memory pipe, not the FMA pipe, was then the limit.  Rows
// are stored in 16-byte chunks, chunk c of row i at c ^ s(i) (Sw): the left
// reads of neighbouring rows, the right reads of one row and the transposed
// reads then fall in distinct banks without padding.
//
// The formulas are those of lqt_lanes.cuh / lqt_lane_step.cuh: eq. lqt_comb
// for the operator, the Riccati step of Sec. II-B with the gains of
// eq. Control_LQT, and the affine maps of Sec. IV-C.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lqt_lane_step.cuh"
#include "lqt_tma.cuh"

namespace lqt {
namespace team {

using lanes::rcp;

template <typename R>
__device__ __forceinline__ R fma_(R a, R b, R c);
template <>
__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
template <>
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }

// Shared-memory layout of a matrix with COLS columns (COLS * sizeof(R) a
// multiple of 16 bytes): row-major, the 16-byte chunks of a row permuted.
template <typename R, int COLS>
struct Sw {
    static constexpr int EPC = 16 / (int)sizeof(R);  // elements per chunk
    static constexpr int RC = COLS / EPC;            // chunks per row
    static constexpr int RPL = RC >= 8 ? 1 : 8 / RC; // rows per 128 bytes
    static constexpr int MASK = (RC < 8 ? RC : 8) - 1;
    static_assert(COLS % EPC == 0, "whole chunks");
    __device__ static __forceinline__ int s(int row) { return (row / RPL) & MASK; }
    __device__ static __forceinline__ int chunk(int row, int c) {
        return row * COLS + ((c ^ s(row)) * EPC);
    }
    __device__ static __forceinline__ int at(int row, int col) {
        return chunk(row, col / EPC) + col % EPC;
    }
};

// CT consecutive values from / to p (aligned to CT values, at most 16 bytes)
template <int CT>
__device__ __forceinline__ void ldv(const float* p, float* o) {
    if constexpr (CT == 4) {
        const float4 t = *reinterpret_cast<const float4*>(p);
        o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
    } else if constexpr (CT == 2) {
        const float2 t = *reinterpret_cast<const float2*>(p);
        o[0] = t.x; o[1] = t.y;
    } else {
        o[0] = *p;
    }
}
template <int CT>
__device__ __forceinline__ void ldv(const double* p, double* o) {
    if constexpr (CT == 2) {
        const double2 t = *reinterpret_cast<const double2*>(p);
        o[0] = t.x; o[1] = t.y;
    } else {
        o[0] = *p;
    }
}
template <int CT>
__device__ __forceinline__ void stv(float* p, const float* o) {
    if constexpr (CT == 4) *reinterpret_cast<float4*>(p) = make_float4(o[0], o[1], o[2], o[3]);
    else if constexpr (CT == 2) *reinterpret_cast<float2*>(p) = make_float2(o[0], o[1]);
    else *p = o[0];
}
template <int CT>
__device__ __forceinline__ void stv(double* p, const double* o) {
    if constexpr (CT == 2) *reinterpret_cast<double2*>(p) = make_double2(o[0], o[1]);
    else *p = o[0];
}

// CT consecutive columns (CT divides col) of a swizzled row
template <int COLS, int CT, typename R>
__device__ __forceinline__ void ldrow(const R* m, int row, int col, R (&o)[CT]) {
    constexpr int E = Sw<R, COLS>::EPC, V = CT < E ? CT : E;
#pragma unroll
    for (int v = 0; v < CT; v += V) ldv<V>(m + Sw<R, COLS>::at(row, col + v), o + v);
}
template <int COLS, int CT, typename R>
__device__ __forceinline__ void strow(R* m, int row, int col, const R (&o)[CT]) {
    constexpr int E = Sw<R, COLS>::EPC, V = CT < E ? CT : E;
#pragma unroll
    for (int v = 0; v < CT; v += V) stv<V>(m + Sw<R, COLS>::at(row, col + v), o + v);
}
// the same in global memory, row stride COLS; vec: the matrix starts on 16 bytes
template <int COLS, int CT, typename R>
__device__ __forceinline__ void ldg_row(const R* m, int row, int col, R (&o)[CT], bool vec) {
    constexpr int E = 16 / (int)sizeof(R), V = CT < E ? CT : E;
    const R* p = m + row * COLS + col;
    if (vec) {
#pragma unroll
        for (int v = 0; v < CT; v += V) ldv<V>(p + v, o + v);
    } else {
#pragma unroll
        for (int v = 0; v < CT; ++v) o[v] = p[v];
    }
}
template <int COLS, int CT, typename R>
__device__ __forceinline__ void stg_row(R* m, int row, int col, const R (&o)[CT], bool vec) {
    constexpr int E = 16 / (int)sizeof(R), V = CT < E ? CT : E;
    R* p = m + row * COLS + col;
    if (vec) {
#pragma unroll
        for (int v = 0; v < CT; v += V) stv<V>(p + v, o + v);
    } else {
#pragma unroll
        for (int v = 0; v < CT; ++v) p[v] = o[v];
    }
}

// One team of LG = N^2 / (4 RT) lanes: lane = tile (ri, ci) of RT x 4 entries,
// ri in [0, N / RT), ci in [0, N / 4).  Left-operand ("NN") tiles hold rows
// ri + i N / RT, transposed-left ("TN") tiles rows RT ri + i, i < RT; both hold
// columns 4 ci .. 4 ci + 3 of N (2 ci, 2 ci + 1 of M).
template <int N, int RT = 2>
struct Team {
    static constexpr int LC = N / 4, LR = N / RT;
    static constexpr int LG = LC * LR;
    static constexpr int LW = LG < 32 ? LG : 32;  // lanes in one warp
    static constexpr int NW = LG / LW;            // warps
    int lane, ri, ci;
    unsigned mask;  // the team's lanes of this warp
    __device__ __forceinline__ Team() {
        lane = threadIdx.x % LG;
        ri = lane / LC;
        ci = lane % LC;
        mask = LG >= 32 ? 0xffffffffu
                        : (((1u << LW) - 1u) << ((threadIdx.x & 31) / LW * LW));
    }
    __device__ __forceinline__ void sync() const {
        if constexpr (LG <= 32)
            __syncwarp(mask);
        else  // one named barrier per team of the CTA (0 is __syncthreads)
            asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)threadIdx.x / LG), "n"(LG) : "memory");
    }
    // whether x holds in every lane of the team
    __device__ __forceinline__ bool all(bool x) const {
        if constexpr (LG <= 32) {
            return __all_sync(mask, x);
        } else {
            int r;
            asm volatile(
                "{\n .reg .pred p, q;\n setp.ne.s32 p, %1, 0;\n"
                " bar.red.and.pred q, %2, %3, p;\n selp.s32 %0, 1, 0, q;\n}"
                : "=r"(r)
                : "r"((int)x), "r"(1 + (int)threadIdx.x / LG), "n"(LG)
                : "memory");
            return r != 0;
        }
    }
    // sum over the LC lanes of a lane row
    template <typename R>
    __device__ __forceinline__ R row_sum(R x) const {
#pragma unroll
        for (int d = 1; d < LC; d <<= 1) x += __shfl_xor_sync(mask, x, d);
        return x;
    }
};

// steps of k unrolled together: whole periods of the swizzle, whole loops up to 16
constexpr int k_unroll(int K) { return K <= 16 ? K : 8; }

// acc[i] += sign * A[r0 + i step][0..K) B[0..K)[c0 .. c0 + CT)
template <int K, int ACOLS, int BCOLS, bool NEG, int RT, int CT, typename R>
__device__ __forceinline__ void nn(R (&acc)[RT][CT], const R* A, const R* B, int r0, int step,
                                   int c0) {
    constexpr int E = 16 / (int)sizeof(R);
#pragma unroll(k_unroll(K) / E)
    for (int k = 0; k < K; k += E) {
        R a[RT][E];
#pragma unroll
        for (int i = 0; i < RT; ++i) ldrow<ACOLS, E>(A, r0 + i * step, k, a[i]);
#pragma unroll
        for (int q = 0; q < E; ++q) {
            R b[CT];
            ldrow<BCOLS, CT>(B, k + q, c0, b);
#pragma unroll
            for (int i = 0; i < RT; ++i)
#pragma unroll
                for (int c = 0; c < CT; ++c)
                    acc[i][c] = fma_(NEG ? -a[i][q] : a[i][q], b[c], acc[i][c]);
        }
    }
}

// acc[i] += sign * sum_k A[k][r0 + i] B[k][c0 ..), i < RT
template <int K, int ACOLS, int BCOLS, bool NEG, int RT, int CT, typename R>
__device__ __forceinline__ void tn(R (&acc)[RT][CT], const R* A, const R* B, int r0, int c0) {
#pragma unroll(k_unroll(K))
    for (int k = 0; k < K; ++k) {
        R a[RT], b[CT];
        ldrow<ACOLS, RT>(A, k, r0, a);
        ldrow<BCOLS, CT>(B, k, c0, b);
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int c = 0; c < CT; ++c) acc[i][c] = fma_(NEG ? -a[i] : a[i], b[c], acc[i][c]);
    }
}

template <int RT, int CT, typename R>
__device__ __forceinline__ void zero(R (&a)[RT][CT]) {
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int c = 0; c < CT; ++c) a[i][c] = R(0);
}

// tile <- (tile + transpose) / 2 for a TN tile whose raw values of all lanes
// are in `raw` (N x N)
template <int N, int RT, typename R>
__device__ __forceinline__ void symmetrise(R (&t)[RT][4], const R* raw, const Team<N, RT>& g) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        R x[RT];
        ldrow<N, RT>(raw, 4 * g.ci + c, RT * g.ri, x);
#pragma unroll
        for (int i = 0; i < RT; ++i) t[i][c] = R(0.5) * (t[i][c] + x[i]);
    }
}

// RT rows r0 + i step of a swizzled matrix, columns c0 .. c0 + CT
template <int COLS, int RT, int CT, typename R>
__device__ __forceinline__ void ldtile(const R* m, int r0, int step, int c0, R (&t)[RT][CT]) {
#pragma unroll
    for (int i = 0; i < RT; ++i) ldrow<COLS, CT>(m, r0 + i * step, c0, t[i]);
}
template <int COLS, int RT, int CT, typename R>
__device__ __forceinline__ void sttile(R* m, int r0, int step, int c0, const R (&t)[RT][CT]) {
#pragma unroll
    for (int i = 0; i < RT; ++i) strow<COLS, CT>(m, r0 + i * step, c0, t[i]);
}

// The system [G | B] of an m x m solve in shared memory: M rows, G's M columns
// and then NR right sides, row stride LD.  A lane reads whole columns, so the
// solve's loads and stores are one uniform sweep over the rows; LD = 4 mod 16
// keeps rows 16-byte aligned for the products that read it and spreads the
// transposed stores of P2 over the banks.
template <int N, int M, int NR>
struct Sys {
    static constexpr int B = M;  // first right side
    static constexpr int LD = N == 8 ? (M + NR + 3) / 4 * 4 : (M + NR - 4 + 15) / 16 * 16 + 4;
    static constexpr int SIZE = M * LD;
    static_assert(LD >= M + NR, "all columns fit");
};
template <int LD, int CT, typename R>
__device__ __forceinline__ void ldsys(const R* t, int row, int col, R (&o)[CT]) {
    constexpr int E = 16 / (int)sizeof(R), V = CT < E ? CT : E;
#pragma unroll
    for (int v = 0; v < CT; v += V) ldv<V>(t + row * LD + col + v, o + v);
}
template <int LD, int CT, typename R>
__device__ __forceinline__ void stsys(R* t, int row, int col, const R (&o)[CT]) {
    constexpr int E = 16 / (int)sizeof(R), V = CT < E ? CT : E;
#pragma unroll
    for (int v = 0; v < CT; v += V) stv<V>(t + row * LD + col + v, o + v);
}

// 1 / sqrt(x) to within an ulp: the hardware's approximation and one Newton
// step (FP32; x > 0 and normal), two correctly rounded steps (FP64)
__device__ __forceinline__ float rsqrt_(float x) {
    const float y = rsqrtf(x);
    return fmaf(0.5f * y, fmaf(-x * y, y, 1.0f), y);
}
__device__ __forceinline__ double rsqrt_(double x) { return 1.0 / sqrt(x); }

// The M x M systems above by elimination without pivoting (stable for SPD G).
// Column-per-lane: every warp of the team holds the M columns of G and its
// share of the right sides in registers; the pivot column's entries come from
// its lane by shuffles, and no sync is needed before the caller's.  FULL: the
// right sides become G^{-1} B (Gauss-Jordan); otherwise Rc^{-1} B with
// G = Rc Rc^T (the forward half of a Cholesky solve, half the work).  With inv
// (FULL) G^{-1} replaces G: a pivot's own column takes its inverse column
// instead of the unit column.
template <bool FULL, int M, int NR, int N, int RT, typename R>
__device__ __forceinline__ bool solve_spd(R* t, const Team<N, RT>& g, bool inv = false) {
    using T = Team<N, RT>;
    using S = Sys<N, M, NR>;
    constexpr int NRW = (NR + T::NW - 1) / T::NW;
    constexpr int COLS = M + NRW, SL = (COLS + T::LW - 1) / T::LW;
    const int lw = g.lane % T::LW, wi = g.lane / T::LW;
    R col[SL][M];
#pragma unroll
    for (int s = 0; s < SL; ++s) {
        const int j = s * T::LW + lw, c = j < M ? j : j + wi * NRW;
        const bool in = j < COLS && c < M + NR;
#pragma unroll
        for (int i = 0; i < M; ++i) col[s][i] = in ? t[i * S::LD + c] : R(0);
    }
    if (FULL && T::NW > 1 && inv) g.sync();  // every warp has read G
    bool ok = true;
#pragma unroll
    for (int k = 0; k < M; ++k) {
        const int ks = k / T::LW, kl = k % T::LW;
        const R piv = __shfl_sync(g.mask, col[ks][k], kl, T::LW);
        ok = ok && piv > R(0) && isfinite(piv);
        const R sc = FULL ? rcp(piv) : rsqrt_(piv);
        R f[M];
#pragma unroll
        for (int i = 0; i < M; ++i)
            if (i > k || (FULL && i < k)) f[i] = __shfl_sync(g.mask, col[ks][i], kl, T::LW);
#pragma unroll
        for (int s = 0; s < SL; ++s) {
            const bool own = FULL && s == ks && inv && lw == kl;
            const R pk = own ? sc : col[s][k] * sc, fk = FULL ? pk : pk * sc;
#pragma unroll
            for (int i = 0; i < M; ++i)
                if (i > k || (FULL && i < k))
                    col[s][i] = fma_(-f[i], fk, own ? R(0) : col[s][i]);
            col[s][k] = pk;
        }
    }
#pragma unroll
    for (int s = 0; s < SL; ++s) {
        const int j = s * T::LW + lw, c = j < M ? j : j + wi * NRW;
        if ((j >= M || (FULL && inv && wi == 0)) && j < COLS && c < M + NR) {
#pragma unroll
            for (int i = 0; i < M; ++i) t[i * S::LD + c] = col[s][i];
        }
    }
    return ok;
}

// Row key of the pivot search: the magnitude's leading bits with the row in
// the low five, 0 for a row already used.  The largest key is the largest
// entry up to a relative 2^-18 (2^-15 for FP64, from its high word).
__device__ __forceinline__ unsigned pivot_key(float x, int row) {
    return (__float_as_uint(fabsf(x)) & ~31u) | (unsigned)row;
}
__device__ __forceinline__ unsigned pivot_key(double x, int row) {
    return ((unsigned)__double2hiint(fabs(x)) & ~31u) | (unsigned)row;
}

// [M | B] by Gauss-Jordan elimination with partial pivoting.  Row-per-lane:
// lane r of each group of N lanes holds row r of M and its group's NR columns
// of B in registers; the LG / N groups repeat M and split B's columns.  The
// pivot row is found by one warp reduction and read by shuffles; rows are not
// swapped: a lane's row ends as the solution row of the pivot it served as,
// which is returned in `krow`.  M's columns shift left by one each step, so
// the loop needs no dynamic register index.
template <int NR, int N, typename R>
__device__ __forceinline__ bool solve_pivoted(R (&m)[N], R (&b)[NR], int& krow,
                                              const Team<N>& g) {
    const int r = g.lane % N;
    bool used = false, ok = true;
#pragma unroll 1
    for (int k = 0; k < N; ++k) {
        const unsigned key = used ? 0u : pivot_key(m[0], r);
        const int p = (int)(__reduce_max_sync(g.mask, key) & 31u);
        const R piv = __shfl_sync(g.mask, m[0], p, N);
        ok = ok && piv != R(0) && isfinite(piv);
        const R inv = rcp(piv);
        const bool me = r == p;
        // other rows subtract f times the pivot row; the pivot row is scaled:
        // x - (1 - inv) x = inv x would lose digits, so it is selected
        const R f = m[0] * inv;
#pragma unroll
        for (int c = 1; c < N; ++c) {
            const R pc = __shfl_sync(g.mask, m[c], p, N);
            m[c - 1] = me ? pc * inv : fma_(-f, pc, m[c]);
        }
#pragma unroll
        for (int c = 0; c < NR; ++c) {
            const R pc = __shfl_sync(g.mask, b[c], p, N);
            b[c] = me ? pc * inv : fma_(-f, pc, b[c]);
        }
        if (me) {
            used = true;
            krow = k;
        }
    }
    return ok;
}

// ---- element, value and affine map in global memory: dense rows -----------
template <int N>
struct DElem {  // A, b, C, eta, J
    static constexpr int OA = 0, OB = N * N, OC = OB + N, OE = OC + N * N, OJ = OE + N,
                         SIZE = OJ + N * N;
};
template <int N>
struct DValue {  // S, v
    static constexpr int OS = 0, OV = N * N, SIZE = N * N + N;
};
template <int N>
struct DAffine {  // F, c
    static constexpr int OF = 0, OC = N * N, SIZE = N * N + N;
};

// dense global matrix (16-byte aligned) -> swizzled shared matrix
template <int N, typename R>
__device__ __forceinline__ void load_mat(R* dst, const R* src, const Team<N>& g) {
    constexpr int E = 16 / (int)sizeof(R), RC = N / E;
#pragma unroll
    for (int t = 0; t < N * RC / Team<N>::LG; ++t) {
        const int q = t * Team<N>::LG + g.lane, row = q / RC, c = q % RC;
        R x[E];
        ldv<E>(src + q * E, x);
        stv<E>(dst + Sw<R, N>::chunk(row, c), x);
    }
}

// Shared memory of combine / value_apply (elements)
template <int N>
struct CombineSmem {
    static constexpr int C1 = 0, J2 = N * N, A1 = 2 * N * N, A2 = 3 * N * N, MX = 4 * N * N,
                         X3 = 5 * N * N, JX = 6 * N * N, T = 7 * N * N, V = 8 * N * N,
                         SIZE = V + 6 * N;
};
template <int N>
struct ApplySmem {
    static constexpr int C = 0, S = N * N, A = 2 * N * N, MX = 3 * N * N, T = 4 * N * N,
                         V = 5 * N * N, SIZE = V + 3 * N;
};

// out = e1 (x) e2 (eq. lqt_comb) for dense elements in global memory (out may
// be e1).  sh: CombineSmem<N>::SIZE elements of the team's shared memory.
template <int N, typename R>
__device__ bool combine(const R* e1, const R* e2, R* out, R* sh, const Team<N>& g) {
    using E = DElem<N>;
    using S = CombineSmem<N>;
    constexpr int H = N / 2, CG = 16;  // matrix right sides per column group
    const int ri = g.ri, ci = g.ci;
    R* b1 = sh + S::V;
    R* h1 = b1 + N;
    R* b2 = h1 + N;
    R* h2 = b2 + N;
    R* be = h2 + N;
    R* w = be + N;
    load_mat<N>(sh + S::C1, e1 + E::OC, g);
    load_mat<N>(sh + S::J2, e2 + E::OJ, g);
    load_mat<N>(sh + S::A1, e1 + E::OA, g);
    load_mat<N>(sh + S::A2, e2 + E::OA, g);
    for (int i = g.lane; i < N; i += Team<N>::LG) {
        b1[i] = e1[E::OB + i];
        h1[i] = e1[E::OE + i];
        b2[i] = e2[E::OB + i];
        h2[i] = e2[E::OE + i];
    }
    // the terms added last (rows 2 ri, 2 ri + 1 of J1; rows ri, ri + H of C2)
    R jj[2][4], cc[2][4];
    ldg_row<N, 4>(e1 + E::OJ, 2 * ri, 4 * ci, jj[0], true);
    ldg_row<N, 4>(e1 + E::OJ, 2 * ri + 1, 4 * ci, jj[1], true);
    ldg_row<N, 4>(e2 + E::OC, ri, 4 * ci, cc[0], true);
    ldg_row<N, 4>(e2 + E::OC, ri + H, 4 * ci, cc[1], true);
    g.sync();
    // M = I + C1 J2 ; be = b1 + C1 eta2 ; w = eta2 - J2 b1
    {
        R a[2][4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            a[0][c] = ri == 4 * ci + c ? R(1) : R(0);
            a[1][c] = ri + H == 4 * ci + c ? R(1) : R(0);
        }
        nn<N, N, N, false>(a, sh + S::C1, sh + S::J2, ri, H, 4 * ci);
        sttile<N>(sh + S::MX, ri, H, 4 * ci, a);
        R s[4] = {R(0), R(0), R(0), R(0)};
        R x0[4], x1[4], y0[4], y1[4];
        ldrow<N, 4>(sh + S::C1, ri, 4 * ci, x0);
        ldrow<N, 4>(sh + S::C1, ri + H, 4 * ci, x1);
        ldrow<N, 4>(sh + S::J2, ri, 4 * ci, y0);
        ldrow<N, 4>(sh + S::J2, ri + H, 4 * ci, y1);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const R h = h2[4 * ci + c], b = b1[4 * ci + c];
            s[0] = fma_(x0[c], h, s[0]);
            s[1] = fma_(x1[c], h, s[1]);
            s[2] = fma_(-y0[c], b, s[2]);
            s[3] = fma_(-y1[c], b, s[3]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) s[i] = g.row_sum(s[i]);
        if (ci == 0) {
            be[ri] = b1[ri] + s[0];
            be[ri + H] = b1[ri + H] + s[1];
            w[ri] = h2[ri] + s[2];
            w[ri + H] = h2[ri + H] + s[3];
        }
    }
    g.sync();
    // X1 = M^{-1} A1, X3 = M^{-1} C1 (16 columns of [A1 | C1] per group of N
    // lanes), x2 = M^{-1} be
    bool ok;
    {
        const int r = g.lane % N, grp = g.lane / N;
        R m[N], b[CG + 1];
#pragma unroll
        for (int c = 0; c < N; c += 2) {
            R x[2];
            ldrow<N, 2>(sh + S::MX, r, c, x);
            m[c] = x[0];
            m[c + 1] = x[1];
        }
#pragma unroll
        for (int c = 0; c < CG; c += 2) {
            const int q = grp * CG + c;  // column of [A1 | C1]
            R x[2];
            ldrow<N, 2>(sh + (q < N ? S::A1 : S::C1), r, q & (N - 1), x);
            b[c] = x[0];
            b[c + 1] = x[1];
        }
        b[CG] = be[r];
        int kr = 0;
        ok = solve_pivoted<CG + 1, N>(m, b, kr, g);
        g.sync();  // MX and be are read
#pragma unroll
        for (int c = 0; c < CG; c += 2) {
            const int q = grp * CG + c;
            const R x[2] = {b[c], b[c + 1]};
            strow<N, 2>(sh + (q < N ? S::MX : S::X3), kr, q & (N - 1), x);
        }
        if (grp == 0) be[kr] = b[CG];
    }
    g.sync();
    // JX = J2 X1, A = A2 X1, T = A2 X3 ; b = b2 + A2 x2 ; eta = eta1 + X1^T w
    R aa[2][4];
    {
        R jx[2][4], t[2][4];
        zero(aa);
        zero(jx);
        zero(t);
        nn<N, N, N, false>(jx, sh + S::J2, sh + S::MX, ri, H, 4 * ci);
        nn<N, N, N, false>(aa, sh + S::A2, sh + S::MX, ri, H, 4 * ci);
        nn<N, N, N, false>(t, sh + S::A2, sh + S::X3, ri, H, 4 * ci);
        strow<N, 4>(sh + S::JX, ri, 4 * ci, jx[0]);
        strow<N, 4>(sh + S::JX, ri + H, 4 * ci, jx[1]);
        strow<N, 4>(sh + S::T, ri, 4 * ci, t[0]);
        strow<N, 4>(sh + S::T, ri + H, 4 * ci, t[1]);
        R s[4] = {R(0), R(0), R(0), R(0)};
        R x0[4], x1[4];
        ldrow<N, 4>(sh + S::A2, ri, 4 * ci, x0);
        ldrow<N, 4>(sh + S::A2, ri + H, 4 * ci, x1);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int k = 4 * ci + c;
            s[0] = fma_(x0[c], be[k], s[0]);
            s[1] = fma_(x1[c], be[k], s[1]);
            R x[2];
            ldrow<N, 2>(sh + S::MX, k, 2 * ri, x);
            s[2] = fma_(x[0], w[k], s[2]);
            s[3] = fma_(x[1], w[k], s[3]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) s[i] = g.row_sum(s[i]);
        if (ci == 0) {
            out[E::OB + ri] = b2[ri] + s[0];
            out[E::OB + ri + H] = b2[ri + H] + s[1];
            out[E::OE + 2 * ri] = h1[2 * ri] + s[2];
            out[E::OE + 2 * ri + 1] = h1[2 * ri + 1] + s[3];
        }
    }
    g.sync();
    // J = J1 + A1^T JX ; C = C2 + T A2^T
    tn<N, N, N, false>(jj, sh + S::A1, sh + S::JX, 2 * ri, 4 * ci);
    {
        constexpr int EP = 16 / (int)sizeof(R);
#pragma unroll 1
        for (int k = 0; k < N; k += EP) {
            R t0[EP], t1[EP];
            ldrow<N, EP>(sh + S::T, ri, k, t0);
            ldrow<N, EP>(sh + S::T, ri + H, k, t1);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                R a[EP];
                ldrow<N, EP>(sh + S::A2, 4 * ci + c, k, a);
#pragma unroll
                for (int q = 0; q < EP; ++q) {
                    cc[0][c] = fma_(t0[q], a[q], cc[0][c]);
                    cc[1][c] = fma_(t1[q], a[q], cc[1][c]);
                }
            }
        }
    }
    // raw C into C1 (no longer read), raw J into J2
    strow<N, 4>(sh + S::C1, ri, 4 * ci, cc[0]);
    strow<N, 4>(sh + S::C1, ri + H, 4 * ci, cc[1]);
    strow<N, 4>(sh + S::J2, 2 * ri, 4 * ci, jj[0]);
    strow<N, 4>(sh + S::J2, 2 * ri + 1, 4 * ci, jj[1]);
    stg_row<N, 4>(out + E::OA, ri, 4 * ci, aa[0], true);
    stg_row<N, 4>(out + E::OA, ri + H, 4 * ci, aa[1], true);
    g.sync();
    ldrow<N, 4>(sh + S::C1, 2 * ri, 4 * ci, cc[0]);
    ldrow<N, 4>(sh + S::C1, 2 * ri + 1, 4 * ci, cc[1]);
    symmetrise<N>(cc, sh + S::C1, g);
    symmetrise<N>(jj, sh + S::J2, g);
    stg_row<N, 4>(out + E::OC, 2 * ri, 4 * ci, cc[0], true);
    stg_row<N, 4>(out + E::OC, 2 * ri + 1, 4 * ci, cc[1], true);
    stg_row<N, 4>(out + E::OJ, 2 * ri, 4 * ci, jj[0], true);
    stg_row<N, 4>(out + E::OJ, 2 * ri + 1, 4 * ci, jj[1], true);
    return ok;
}

// out = P (x) val for a value val = (0, 0, 0, v, S) (dense, global; out may be
// val): S <- A^T S X + J, v <- X^T (v - S b) + eta, X = (I + C S)^{-1} A.
template <int N, typename R>
__device__ bool value_apply(const R* P, const R* val, R* out, R* sh, const Team<N>& g) {
    using E = DElem<N>;
    using V = DValue<N>;
    using S = ApplySmem<N>;
    constexpr int H = N / 2, CG = 8;
    const int ri = g.ri, ci = g.ci;
    R* v = sh + S::V;
    R* b = v + N;
    R* e = b + N;
    load_mat<N>(sh + S::C, P + E::OC, g);
    load_mat<N>(sh + S::S, val + V::OS, g);
    load_mat<N>(sh + S::A, P + E::OA, g);
    for (int i = g.lane; i < N; i += Team<N>::LG) {
        v[i] = val[V::OV + i];
        b[i] = P[E::OB + i];
    }
    R jj[2][4];
    ldg_row<N, 4>(P + E::OJ, 2 * ri, 4 * ci, jj[0], true);
    ldg_row<N, 4>(P + E::OJ, 2 * ri + 1, 4 * ci, jj[1], true);
    const R h0 = P[E::OE + 2 * ri], h1 = P[E::OE + 2 * ri + 1];
    g.sync();
    {
        R a[2][4], x0[4], x1[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            a[0][c] = ri == 4 * ci + c ? R(1) : R(0);
            a[1][c] = ri + H == 4 * ci + c ? R(1) : R(0);
        }
        nn<N, N, N, false>(a, sh + S::C, sh + S::S, ri, H, 4 * ci);
        sttile<N>(sh + S::MX, ri, H, 4 * ci, a);
        ldrow<N, 4>(sh + S::S, ri, 4 * ci, x0);
        ldrow<N, 4>(sh + S::S, ri + H, 4 * ci, x1);
        R s0 = R(0), s1 = R(0);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            s0 = fma_(-x0[c], b[4 * ci + c], s0);
            s1 = fma_(-x1[c], b[4 * ci + c], s1);
        }
        s0 = g.row_sum(s0);
        s1 = g.row_sum(s1);
        if (ci == 0) {
            e[ri] = v[ri] + s0;
            e[ri + H] = v[ri + H] + s1;
        }
    }
    g.sync();
    bool ok;
    {
        const int r = g.lane % N, grp = g.lane / N;
        R m[N], x[CG];
#pragma unroll
        for (int c = 0; c < N; c += 2) {
            R t[2];
            ldrow<N, 2>(sh + S::MX, r, c, t);
            m[c] = t[0];
            m[c + 1] = t[1];
        }
#pragma unroll
        for (int c = 0; c < CG; c += 2) {
            R t[2];
            ldrow<N, 2>(sh + S::A, r, grp * CG + c, t);
            x[c] = t[0];
            x[c + 1] = t[1];
        }
        int kr = 0;
        ok = solve_pivoted<CG, N>(m, x, kr, g);
        g.sync();
#pragma unroll
        for (int c = 0; c < CG; c += 2) {
            const R t[2] = {x[c], x[c + 1]};
            strow<N, 2>(sh + S::MX, kr, grp * CG + c, t);
        }
    }
    g.sync();
    {
        R t[2][4];
        zero(t);
        nn<N, N, N, false>(t, sh + S::S, sh + S::MX, ri, H, 4 * ci);
        strow<N, 4>(sh + S::T, ri, 4 * ci, t[0]);
        strow<N, 4>(sh + S::T, ri + H, 4 * ci, t[1]);
        R s0 = R(0), s1 = R(0);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            R x[2];
            ldrow<N, 2>(sh + S::MX, 4 * ci + c, 2 * ri, x);
            s0 = fma_(x[0], e[4 * ci + c], s0);
            s1 = fma_(x[1], e[4 * ci + c], s1);
        }
        s0 = g.row_sum(s0);
        s1 = g.row_sum(s1);
        if (ci == 0) {
            out[V::OV + 2 * ri] = h0 + s0;
            out[V::OV + 2 * ri + 1] = h1 + s1;
        }
    }
    g.sync();
    tn<N, N, N, false>(jj, sh + S::A, sh + S::T, 2 * ri, 4 * ci);
    strow<N, 4>(sh + S::C, 2 * ri, 4 * ci, jj[0]);  // C is no longer read
    strow<N, 4>(sh + S::C, 2 * ri + 1, 4 * ci, jj[1]);
    g.sync();
    symmetrise<N>(jj, sh + S::C, g);
    stg_row<N, 4>(out + V::OS, 2 * ri, 4 * ci, jj[0], true);
    stg_row<N, 4>(out + V::OS, 2 * ri + 1, 4 * ci, jj[1], true);
    return ok;
}

// f2 after f1: (F2 F1, F2 c1 + c2) into out (may be f1 or f2).  sh: 2 N^2.
template <int N, typename R>
__device__ void affine_compose(const R* f1, const R* f2, R* out, R* sh, const Team<N>& g) {
    using A = DAffine<N>;
    constexpr int H = N / 2;
    const int ri = g.ri, ci = g.ci;
    load_mat<N>(sh, f2 + A::OF, g);
    load_mat<N>(sh + N * N, f1 + A::OF, g);
    R c1[4];
    ldg_row<N, 4>(f1 + A::OC, 0, 4 * ci, c1, true);
    const R c20 = f2[A::OC + ri], c21 = f2[A::OC + ri + H];
    g.sync();
    R t[2][4], x0[4], x1[4];
    zero(t);
    nn<N, N, N, false>(t, sh, sh + N * N, ri, H, 4 * ci);
    ldrow<N, 4>(sh, ri, 4 * ci, x0);
    ldrow<N, 4>(sh, ri + H, 4 * ci, x1);
    R s0 = R(0), s1 = R(0);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        s0 = fma_(x0[c], c1[c], s0);
        s1 = fma_(x1[c], c1[c], s1);
    }
    s0 = g.row_sum(s0);
    s1 = g.row_sum(s1);
    g.sync();  // every lane has read f1 and f2
    stg_row<N, 4>(out + A::OF, ri, 4 * ci, t[0], true);
    stg_row<N, 4>(out + A::OF, ri + H, 4 * ci, t[1], true);
    if (ci == 0) {
        out[A::OC + ri] = c20 + s0;
        out[A::OC + ri + H] = c21 + s1;
    }
}

// y = F x + c for a dense global map and global vectors (y must not be x
// unless the caller syncs between; both rows are returned to ci == 0 lanes)
template <int N, typename R>
__device__ __forceinline__ void affine_apply(const R* f, const R* x, R& y0, R& y1,
                                             const Team<N>& g) {
    using A = DAffine<N>;
    constexpr int H = N / 2;
    const int ri = g.ri, ci = g.ci;
    R a0[4], a1[4], xv[4];
    ldg_row<N, 4>(f + A::OF, ri, 4 * ci, a0, true);
    ldg_row<N, 4>(f + A::OF, ri + H, 4 * ci, a1, true);
    ldg_row<N, 4>(x, 0, 4 * ci, xv, true);
    R s0 = R(0), s1 = R(0);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        s0 = fma_(a0[c], xv[c], s0);
        s1 = fma_(a1[c], xv[c], s1);
    }
    y0 = f[A::OC + ri] + g.row_sum(s0);
    y1 = f[A::OC + ri + H] + g.row_sum(s1);
}

}  // namespace team
}  // namespace lqt
