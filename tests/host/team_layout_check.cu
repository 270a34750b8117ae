// Host-side checks of the shared-memory layouts of the team kernels and vector
// walks (n = 8, 16, 32) and of the n <= 4 vector pass (built and run by
// tests/test_team_layouts.py; no GPU needed):
//   Sw               the swizzle permutes the 16-byte chunks of each row, and the
//                    reads of a product fall in distinct banks
//   Sys, TFoldSmem, TRefoldSmem, VWalk, VResid, CombineSmem, ApplySmem, VecSmem
//                    parts that are read 16 bytes at a time start on 16 bytes, no
//                    part reaches into the next, the general cost's scratch holds
//                    p = 2n outputs
//   Launcher         every CTA's dynamic shared memory fits the opt-in limit
#include <cstdio>

#include "lqt_chain_impl.cuh"
#include "lqt_kernels.cuh"
#include "lqt_variants.h"

using namespace lqt;
using namespace lqt::chain;

static int fails = 0;
#define CHECK(c, ...)                                \
    do {                                             \
        if (!(c)) {                                  \
            std::printf("FAIL line %d: ", __LINE__); \
            std::printf(__VA_ARGS__);                \
            std::printf("\n");                       \
            ++fails;                                 \
        }                                            \
    } while (0)

constexpr int kLimit = 227 * 1024;

// The address in elements, as Sw::at computes it (device functions; restated).
template <typename R, int COLS>
static int at(int row, int col) {
    constexpr int E = 16 / (int)sizeof(R), RC = COLS / E, RPL = RC >= 8 ? 1 : 8 / RC;
    return row * COLS + (((col / E) ^ ((row / RPL) & ((RC < 8 ? RC : 8) - 1))) * E) + col % E;
}

template <typename R, int ROWS, int COLS>
static void swizzle_checks() {
    using S = team::Sw<R, COLS>;
    constexpr int E = 16 / (int)sizeof(R);
    CHECK(S::EPC == E && S::RC == COLS / E && S::RPL == (S::RC >= 8 ? 1 : 8 / S::RC) &&
              S::MASK == (S::RC < 8 ? S::RC : 8) - 1,
          "constants of Sw<%d, %d>", (int)sizeof(R), COLS);
    bool seen[ROWS * COLS] = {};
    for (int i = 0; i < ROWS; ++i)
        for (int j = 0; j < COLS; ++j) {
            const int q = at<R, COLS>(i, j);
            CHECK(q >= i * COLS && q < (i + 1) * COLS && !seen[q], "element (%d, %d) at %d", i, j, q);
            seen[q] = true;
            CHECK((q % E == j % E && at<R, COLS>(i, j / E * E) % E == 0), "chunk of (%d, %d)", i, j);
        }
    // a column of 16-byte chunks over 8 neighbouring rows covers all 32 banks
    if (S::RC >= 8)
        for (int c = 0; c < S::RC; ++c) {
            unsigned banks = 0;
            for (int i = 0; i < 8; ++i) banks |= 1u << (at<R, COLS>(i, c * E) * (int)sizeof(R) / 16 % 8);
            CHECK(banks == 0xffu, "column %d of %d", c, COLS);
        }
}

// parts[i]: offset and size in elements, ascending
struct Part {
    int at, size;
};
template <typename R, int K>
static void parts_check(const char* name, const Part (&p)[K], int size, bool vec = true) {
    for (int i = 0; i < K; ++i) {
        CHECK(!vec || p[i].at * (int)sizeof(R) % 16 == 0, "%s: part %d at %d", name, i, p[i].at);
        const int next = i + 1 < K ? p[i + 1].at : size;
        CHECK(p[i].at + p[i].size <= next, "%s: part %d [%d, %d) reaches into %d", name, i, p[i].at,
              p[i].at + p[i].size, next);
    }
}

template <typename R, typename RT, int N, int M>
static void team_checks() {
    swizzle_checks<R, N, N>();
    swizzle_checks<R, N, M>();
    swizzle_checks<R, M, N>();
    {
        using S = TFoldSmem<N, M>;
        using Y = typename S::Sy;
        const Part p[] = {{S::PA, N * N}, {S::PC, N * N}, {S::PJ, N * N},
                          {S::IN, TeamIn<N, M>::SIZE}, {S::JF, N * N}, {S::JL, N * M},
                          {S::SY, Y::SIZE}};
        parts_check<R>("fold", p, S::V);
        CHECK(Y::LD >= M + 2 * N + 1 && Y::LD * (int)sizeof(R) % 16 == 0, "fold system stride");
        // cost_general: Y (p x N), H and X staged for p <= N, or Y alone up to p = 2N
        const int staged = N * N + N * N + N * (N | 1), wide = 2 * N * N;
        CHECK(S::JF + (staged > wide ? staged : wide) <= S::V, "fold: general cost's scratch");
        CHECK(S::AC == S::W + N && S::DESC >= S::AC + N, "fold: its 2N outputs");
        CHECK(S::DESC * (int)sizeof(R) % 8 == 0 &&
                  S::SIZE - S::DESC >= (int)(sizeof(DescT<R>) / sizeof(R)),
              "fold: descriptor");
    }
    {
        using S = TRefoldSmem<N, M>;
        using Y = typename S::Sy;
        const Part p[] = {{S::SV, N * N}, {S::PHI, N * N}, {S::IN, TeamIn<N, M>::SIZE},
                          {S::SL, N * M}, {S::SY, Y::SIZE}, {S::FT, N * N}, {S::SFT, N * N}};
        parts_check<R>("re-fold", p, S::V);
        CHECK(Y::LD >= M + N + 1 && Y::LD * (int)sizeof(R) % 16 == 0, "re-fold system stride");
        CHECK(S::SL + N * N <= S::FT, "re-fold: raw S over S L and the system");
        const int staged = N * N + N * N + N * (N | 1), wide = 2 * N * N;
        CHECK(S::SL + (staged > wide ? staged : wide) <= S::V, "re-fold: general cost's scratch");
        CHECK(S::CT == S::EV + N && S::DESC >= S::CT + N, "re-fold: its 2N outputs");
        CHECK(S::DESC * (int)sizeof(R) % 8 == 0 &&
                  S::SIZE - S::DESC >= (int)(sizeof(DescT<R>) / sizeof(R)),
              "re-fold: descriptor");
    }
    {
        using I = TeamIn<N, M>;
        const Part p[] = {{I::F, 2 * N * N}, {I::L, 2 * N * M}, {I::U, 2 * M * M}, {I::C, 2 * N}};
        parts_check<R>("staged inputs", p, I::SIZE);
    }
    {
        using W = VWalk<N, M>;
        const Part f[] = {{W::F, N * N}, {W::L, N * M}, {W::K, M * N}, {W::C, N}, {W::D, M},
                          {W::XH, N}, {W::UH, M}, {W::QH, M}};
        parts_check<R>("forward walk", f, W::FWD);
        const Part b[] = {{W::F, N * N}, {W::L, N * M}, {W::K, M * N}, {W::C, N}, {W::S, N * N},
                          {W::GI, M * M}, {W::E, N}};
        parts_check<R>("backward walk", b, W::BACK);
        CHECK(W::FWD * (int)sizeof(R) % 16 == 0 && W::BACK * (int)sizeof(R) % 16 == 0 &&
                  W::FWD_SIZE * (int)sizeof(R) % 16 == 0 && W::BACK_SIZE * (int)sizeof(R) % 16 == 0,
              "stages and warps of the walks");
    }
    {
        using V = VResid<N, M>;
        const Part p[] = {{V::F, N * N}, {V::L, N * M}, {V::U, M * M}, {V::S, N * N}, {V::X, N * N},
                          {V::XV, N}, {V::UV, M}, {V::VV, N}, {V::CV, N}, {V::RV, N}};
        parts_check<R>("residual stage", p, V::STAGE);
        const Part q[] = {{V::L1, N}, {V::X1, N}, {V::HH, 2 * N}, {V::HL, 2 * N}, {V::YH, 2 * N},
                          {V::YL, 2 * N}, {V::Q, M}};
        parts_check<R>("residual vectors", q, V::SIZE, false);
        CHECK(V::STAGE * (int)sizeof(R) % 16 == 0 && V::SIZE * (int)sizeof(R) % 16 == 0,
              "stages and warps of the residuals");
    }
    {
        using C = team::CombineSmem<N>;
        const Part p[] = {{C::C1, N * N}, {C::J2, N * N}, {C::A1, N * N}, {C::A2, N * N},
                          {C::MX, N * N}, {C::X3, N * N}, {C::JX, N * N}, {C::T, N * N},
                          {C::V, 6 * N}};
        parts_check<RT>("combine", p, C::SIZE);
        using A = team::ApplySmem<N>;
        const Part q[] = {{A::C, N * N}, {A::S, N * N}, {A::A, N * N}, {A::MX, N * N},
                          {A::T, N * N}, {A::V, 3 * N}};
        parts_check<RT>("apply", q, A::SIZE);
    }
    using Lc = Launcher<R, RT, N, M>;
    const long long ctas[] = {(long long)Lc::NT_WALK * Lc::TFOLD_B,
                              (long long)Lc::NT_WALK * Lc::TREFOLD_B,
                              (long long)Lc::TT * Lc::TUP_B, (long long)Lc::TT * Lc::TDOWN_B,
                              (long long)Lc::TT * Lc::TFUP_B, Lc::VFWD_B, Lc::VBACK_B,
                              Lc::VRESID_B};
    for (long long b : ctas) CHECK(b > 0 && b <= kLimit, "N=%d: a CTA of %lld bytes", N, b);
    const int es = (int)sizeof(R), et = (int)sizeof(RT);
    const int blocks[][2] = {{Lc::TFOLD_B, TFoldSmem<N, M>::SIZE * es},
                             {Lc::TREFOLD_B, TRefoldSmem<N, M>::SIZE * es},
                             {Lc::TUP_B, team::CombineSmem<N>::SIZE * et},
                             {Lc::TDOWN_B, team::ApplySmem<N>::SIZE * et},
                             {Lc::TFUP_B, 2 * N * N * et}};
    for (const auto& b : blocks)
        CHECK(b[0] >= b[1] && b[0] % 16 == 0, "N=%d: teams %d bytes apart hold %d", N, b[0], b[1]);
    // named barriers of the teams wider than a warp: 0 is __syncthreads, 15 the last
    CHECK(Lc::LGW <= 32 || Lc::NT_WALK <= 15, "N=%d: barriers of the walks", N);
    CHECK(Lc::LG <= 32 || Lc::TT <= 15, "N=%d: barriers of the tree levels", N);
    if (Lc::kPersistFits) {
        const int warp_teams = Lc::LG < 32 ? 32 / Lc::LG : 1;
        CHECK((long long)Lc::NT_PERSIST * Lc::PERSIST_B <= kLimit && Lc::PERSIST_B % 16 == 0,
              "N=%d: persistent CTA", N);
        const int ring = VWalk<N, M>::FWD_SIZE * es;
        CHECK(ring <= warp_teams * Lc::PERSIST_B,
              "N=%d: a rollout's ring in the blocks of a warp's teams", N);
    }
}

// n <= 4: the vector pass's tree and values, and the first pass's maps behind the
// value tree of a tile's block
template <typename R, int N, int M>
static void vec_checks() {
    constexpr int W = tile_threads<R, N, M>();
    using V = VecSmem<R, N, M, W>;
    constexpr int WS = tstride(W, (int)sizeof(R));
    CHECK(V::XS == Dims<N>::AFFINE * WS && V::MODEL == V::XS + N * WS &&
              (kSmemHead + V::MODEL * (int)sizeof(R)) % 16 == 0,
          "N=%d M=%d: vector pass", N, M);
    for (int p = 0; p <= 2 * N; ++p)
        CHECK(V::bytes(p) <= (size_t)kLimit, "N=%d M=%d p=%d: vector pass", N, M, p);
    CHECK((Dims<N>::ELEM - Dims<N>::AFFINE) * WS >= N * N * W, "N=%d M=%d: kept maps", N, M);
    constexpr int big = SoloSmem<R, N, M, W>::BIG;
    CHECK(V::MODEL <= big, "N=%d M=%d: one tile", N, M);
}
#define VEC_CHECK(R, N, M) vec_checks<R, N, M>();

int main() {
    team_checks<float, float, 8, 4>();
    team_checks<float, float, 16, 8>();
    team_checks<float, float, 32, 16>();
    team_checks<float, double, 8, 4>();
    team_checks<float, double, 16, 8>();
    team_checks<float, double, 32, 16>();
    team_checks<double, double, 8, 4>();
    team_checks<double, double, 16, 8>();
    team_checks<double, double, 32, 16>();
    LQT_VARIANTS_F32_SMALL(VEC_CHECK)
    LQT_VARIANTS_F32_N4(VEC_CHECK)
    LQT_VARIANTS_F64(VEC_CHECK)
    std::printf("%s (%d failures)\n", fails ? "layout checks FAILED" : "layout checks ok", fails);
    return fails ? 1 : 0;
}
