// fill16_variants.cu -- launches of the packed 16-bit pair fill for the
// global, semi-global and overlap algorithms of paper Section 2.1 (no zero
// floor, the algorithm's borders and end cells), in their own translation unit
// so that they compile in parallel with the local fill.
#include "sw.h"
#include "fill16_launch.cuh"

using namespace swgb;

int swgb::launch_fill16_variant(sw_ctx *c, const FillConfig &cfg, int mode, const FillLaunch &L, int K, long long tickets) {
    if (cfg.W != 4) return SW_EINVAL;
    switch (cfg.R) {
        case 8: return launch16_mode4<8, false>(c, mode, cfg.left != 0, L, K, tickets, cfg.B);
        case 12: return launch16_mode4<12, false>(c, mode, cfg.left != 0, L, K, tickets, cfg.B);
        case 16: return launch16_mode4<16, false>(c, mode, cfg.left != 0, L, K, tickets, cfg.B);
        default: return SW_EINVAL;
    }
}

int swgb::launch_straighten_variant(sw_ctx *c, int R, const FillTask *tasks, int ntasks, int max_rows,
                                    const DevScoring *sc) {
    switch (R) {
        case 8: return launch_straighten_r<8, false>(c, tasks, ntasks, max_rows, sc);
        case 12: return launch_straighten_r<12, false>(c, tasks, ntasks, max_rows, sc);
        case 16: return launch_straighten_r<16, false>(c, tasks, ntasks, max_rows, sc);
        default: return SW_EINVAL;
    }
}
