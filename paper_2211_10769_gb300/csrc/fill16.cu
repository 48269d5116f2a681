// fill16.cu -- launches of the packed 16-bit pair fill (wavefront16.cuh) and
// the test of whether a scoring scheme and tile shape keep it exact.
#include "sw.h"
#include "sw_ctx.h"
#include "fill16_launch.cuh"

#include <algorithm>

using namespace swgb;


namespace {

// Steps by which a warp trails the one above, and clocks of a step over the sweep (one strip, measured with the pair
// profile of DNA at the shapes below, and at 4 and 6 rows, which are not built).  The int16 profile's steps are some 5%
// longer at every shape, which leaves the order of the shapes as it is.
constexpr double kP16ChainSteps = 105;
constexpr double kP16TileClocks = 464;
constexpr double p16_step_clocks(int R) { return R <= 8 ? 70 + 3.3 * R : (R <= 16 ? 53 + 5.4 * R : 46 + 6.1 * R); }

// W = 2 (score mode only): blocks of two compute warps for batches, whose
// pairs' last strips are partly empty (a strip of four warps runs its pair's
// width with one to four of them busy).
template <int R>
int launch16_mode(sw_ctx *c, int mode, bool left, int W, const FillLaunch &L, int K, long long tickets, int B) {
    if constexpr (R == 8 || R == 12 || R == 16)
        if (W == 2) return mode == kModeScore && !left ? launch16_pk<R, kModeScore, false, 2>(c, L, K, tickets, B) : SW_EINVAL;
    if (W != 4) return SW_EINVAL;
    return launch16_mode4<R, true>(c, mode, left, L, K, tickets, B);
}

// shapes with a pair profile only, for pairs of small alphabets
#define SWGB_P16_PAIR_SHAPES(X) X(10) X(14) X(20) X(26)
#define SWGB_P16_SHAPES(X) X(8) X(12) X(16) SWGB_P16_PAIR_SHAPES(X)

}  // namespace

bool swgb::p16_fits(const DevScoring &s, int R) {
    switch (R) {
        case 8: case 12: case 16: break;
#define SWGB_P16_CASE(R) case R: if (!pair_profile_fits<R, 4>(s.K)) return false; break;
        SWGB_P16_PAIR_SHAPES(SWGB_P16_CASE)
#undef SWGB_P16_CASE
        default: return false;
    }
    if (s.alg != kAlgLocal && R != 8 && R != 12 && R != 16) return false;   // the shapes of fill16_variants.cu
    int lo = 127, hi = -128;
    for (int k = 0; k < s.K * s.K; ++k) { lo = std::min(lo, (int)s.mat[k]); hi = std::max(hi, (int)s.mat[k]); }
    return p16_spread(R, s.go, s.ge, hi, lo) <= kP16Span;
}

bool swgb::p16_pair_profile(int K) { return pair_profile_fits<8, 4>(K); }

int swgb::launch_fill16(sw_ctx *c, const FillConfig &cfg, int mode, bool fold, const FillLaunch &L, int K,
                        long long tickets) {
    if (tickets <= 0) return SW_OK;
    if (cfg.alg != kAlgLocal) return launch_fill16_variant(c, cfg, mode, L, K, tickets);
    if (cfg.P16 == 2 && fold && mode == kModeScore) return launch_fill16_batch(c, cfg, L, K, tickets);
    switch (cfg.R) {
#define SWGB_P16_CASE(R) case R: return launch16_mode<R>(c, mode, cfg.left != 0, cfg.W, L, K, tickets, cfg.B);
        SWGB_P16_SHAPES(SWGB_P16_CASE)
#undef SWGB_P16_CASE
        default: return SW_EINVAL;
    }
}

int swgb::launch_straighten(sw_ctx *c, int R, bool local, const FillTask *tasks, int ntasks, int max_rows,
                            const DevScoring *sc) {
    if (ntasks <= 0) return SW_OK;
    if (!local) return launch_straighten_variant(c, R, tasks, ntasks, max_rows, sc);
    switch (R) {
#define SWGB_P16_CASE(R) case R: return launch_straighten_r<R, true>(c, tasks, ntasks, max_rows, sc);
        SWGB_P16_SHAPES(SWGB_P16_CASE)
#undef SWGB_P16_CASE
        default: return SW_EINVAL;
    }
}

// Rows a lane of the packed fill of one m x n pair, 0 where no shape is exact
// for the scoring.  A pair's strips (128 R rows each) form one chain: each warp
// trails the one above by kP16ChainSteps steps (64 positions and a chunk of
// 32, and per strip of four warps the hand-off through global memory), and
// strips beyond one per SM follow in waves.  So the fill takes about
//   (columns x whole waves before the last strip + its place in the chain + columns) x step(R),
// with step(R) the measured clocks of a step of one strip (GB300): few rows a
// lane leave a long chain of short steps, many leave SMs idle.  Measured, score
// fills: 30 kbp R = 8 / 10: 2.17 / 2.18 ms; 200 kbp R = 12 / 14: 15.3 / 16.0;
// 1 Mbp R = 14 / 16 / 20 / 26: 257 / 270 / 260 / 214 ms.  (4 and 6 rows a lane were tried
// and not kept: 8 kbp R = 4 / 6 / 8 0.69 / 0.65 / 0.63 ms, 30 kbp R = 6 2.25.)
// tiles: an alignment's forward fill.  Its traceback tiles are as high as a strip (128 R rows), and the
// first round of them runs after the whole fill, kP16TileClocks a row of the side (R = 8 / 12 / 16: 230 / 350 /
// 458 us at 2,070 MHz).
int swgb::p16_rows_per_lane(const sw_ctx *c, int64_t m, int64_t n, const DevScoring &s, bool tiles) {
    static constexpr struct { int R; double clk; } kShapes[] = {
#define SWGB_P16_ROW(R) {R, p16_step_clocks(R)},
        SWGB_P16_SHAPES(SWGB_P16_ROW)
#undef SWGB_P16_ROW
    };
    int best = 0;
    double best_cost = 1e300;
    for (const auto &q : kShapes) {
        if (!p16_fits(s, q.R)) continue;
        const int64_t last = (m + 128LL * q.R - 1) / (128LL * q.R) - 1;      // the last strip
        const double wave = std::max((double)n, c->nsm * kP16ChainSteps * 4);
        const double steps = (double)(last / c->nsm) * wave + (double)(last % c->nsm) * kP16ChainSteps * 4 + (double)n +
                             kP16ChainSteps * std::min<double>(4.0, (double)m / (32.0 * q.R));
        const double cost = steps * q.clk + (tiles ? kP16TileClocks * std::min<double>(128.0 * q.R, (double)std::min(m, n)) : 0);
        if (cost < best_cost) { best_cost = cost; best = q.R; }
    }
    return best;
}
