// fill16_batch.cu -- the packed 16-bit pair fill for batches: an int8 query
// profile, so that three to five blocks fit an SM.  A batch's strips are
// independent enough to fill several blocks an SM, where the ALU pipe is the
// bound: 79% busy with the pair profile in two blocks of four warps at 8 rows a lane, 89%
// with three blocks at 12 rows and the int8 profile.  1,500 pairs of
// 3,072 x 4,000: DNA 3,280 GCUPS with the pair profile at its best shape (8 rows,
// two blocks), 3,530 with 12 rows, int8 and three blocks; protein 3,050 and 3,350.
#include "sw.h"
#include "fill16_launch.cuh"

using namespace swgb;

int swgb::launch_fill16_batch(sw_ctx *c, const FillConfig &cfg, const FillLaunch &L, int K, long long tickets) {
    switch (cfg.R * 16 + cfg.W) {
        case 8 * 16 + 4: return launch16<8, 4, kModeScore, kP16Int8, false, true, 3>(c, L, K, tickets, cfg.B);
        case 12 * 16 + 4: return launch16<12, 4, kModeScore, kP16Int8, false, true, 3>(c, L, K, tickets, cfg.B);
        case 8 * 16 + 2: return launch16<8, 2, kModeScore, kP16Int8, false, true, 5>(c, L, K, tickets, cfg.B);
        case 12 * 16 + 2: return launch16<12, 2, kModeScore, kP16Int8, false, true, 4>(c, L, K, tickets, cfg.B);
        default: return SW_EINVAL;
    }
}
