// db_launch.cuh -- launches of the packed database search for one tile
// shape (rows a lane R, warps a block W, lanes a wavefront G), instantiated in
// several translation units (db_shapes_*.cu) that compile in parallel.
#pragma once
#include "sw_ctx.h"
#include "dbsearch.cuh"

#include <algorithm>

#ifndef CU
#define CU(x) do { if ((x) != cudaSuccess) { cudaGetLastError(); return SW_ECUDA; } } while (0)
#define RC(x) do { int rc_ = (x); if (rc_) return rc_; } while (0)
#endif

namespace swgb {

inline constexpr long long kMaxProfileSmem = 200 * 1024;

// Profile bytes of a query of m residues for tile shape (R, G) (whole passes
// of G lane slots of db_lane_slot(R) bytes, per residue code and padding).
template <int R, int G>
size_t db_profile_bytes(int codes, int m) {
    constexpr int ROWS = G * R;
    const long long mpad = (long long)((m + ROWS - 1) / ROWS) * G * db_lane_slot(R);
    return (size_t)(codes + 1) * (size_t)mpad;
}

// Scratch of one launch: boundary rows, one per wavefront (32 / G of them a
// warp) of every block that can be resident at once, and the slot pool's words.
template <int R, int W, int G>
int db_scratch(sw_ctx *c, int codes, int m, int maxlen, int *nslots, size_t *row_bytes, size_t *slot_bytes) {
    const size_t smem = db_profile_bytes<R, G>(codes, m);
    int occ = 0;
    CU(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, db_s16x2_kernel<R, W, false, G>, W * 32, smem));
    int occ2 = 0;
    CU(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ2, db_s16x2_kernel<R, W, true, G>, W * 32, smem));
    occ = std::min(occ, occ2);
    if (occ < 1) return SW_ECUDA;
    *nslots = occ * c->nsm;
    *row_bytes = (size_t)*nslots * W * (32 / G) * (size_t)(maxlen + 1) * sizeof(uint2);
    *slot_bytes = (size_t)((*nslots + 31) / 32) * sizeof(unsigned);
    return SW_OK;
}

template <int R, int W, int G>
int launch_db(sw_ctx *c, const DbJob *jobs, int njobs, int nblocks, const DbView &D0, int codes, int m,
              const DbBufs &B) {
    const size_t smem = db_profile_bytes<R, G>(codes, m);
    // boundary rows: one per warp of every block that can be resident at once; a grid larger
    // than that (the server's steps) takes the kernel whose later blocks share the slots
    DbView D = D0;
    size_t row_bytes = 0, slot_bytes = 0;
    RC((db_scratch<R, W, G>(c, codes, m, D.maxlen, &D.nslots, &row_bytes, &slot_bytes)));
    D.slot_words = (D.nslots + 31) / 32;
    const bool over = nblocks > D.nslots;
    RC(B.rows->ensure(row_bytes));
    RC(B.slots->ensure(slot_bytes));
    D.slot_pool = static_cast<unsigned *>(B.slots->p);
    D.err = B.err;
    D.spin_limit = c->spin_limit;
    if (over) {
        init_slot_pool_kernel<<<1, 64, 0, c->stream>>>(D.slot_pool, D.slot_words, D.nslots, D.nslots);
        CU(cudaGetLastError());
        ++c->launches;
    }
    auto kern = over ? db_s16x2_kernel<R, W, true, G> : db_s16x2_kernel<R, W, false, G>;
    const int kp = kt_begin(c, SW_KT_DB16);
    kern<<<(unsigned)nblocks, W * 32, smem, c->stream>>>(jobs, njobs, D, B.scorings,
                                                         static_cast<uint2 *>(B.rows->p));
    kt_end(c, kp);
    CU(cudaGetLastError());
    ++c->launches;
    return SW_OK;
}

template <int R, int W, int G>
int resident_blocks(sw_ctx *c, int codes, int m, int *out) {
    const size_t smem = db_profile_bytes<R, G>(codes, m);
    if ((long long)smem > kMaxProfileSmem) return SW_ERANGE;
    static int attr_set[64] = {0};
    if (c->device < 64 && !attr_set[c->device]) {
        CU(cudaFuncSetAttribute(db_s16x2_kernel<R, W, false, G>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kMaxProfileSmem));
        CU(cudaFuncSetAttribute(db_s16x2_kernel<R, W, true, G>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kMaxProfileSmem));
        attr_set[c->device] = 1;
    }
    int occ = 0;
    CU(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, db_s16x2_kernel<R, W, false, G>, W * 32, smem));
    if (occ < 1) return SW_ECUDA;
    *out = occ * c->nsm;
    return SW_OK;
}

// A tile shape, what it measures and what can be done with it; `codes`: the database's residue codes (DbView::pad).
//   gcups: 10^9 cells a second, padding rows included, all SMs full (60,000 subjects of 360 residues);
//   clk1, clk: clocks of a step of a warp that has its SM for itself (subjects of 40,000 columns), for
//   queries of one pass and of several, whose boundary row goes through memory.
// (GB300, 152 SMs, 2,070 MHz.)
struct DbShape {
    int R, W, G;
    double gcups, clk1, clk;
    size_t (*profile_bytes)(int codes, int m);
    int (*scratch)(sw_ctx *c, int codes, int m, int maxlen, int *nslots, size_t *row_bytes, size_t *slot_bytes);
    int (*launch)(sw_ctx *c, const DbJob *jobs, int njobs, int nblocks, const DbView &D, int codes, int m, const DbBufs &B);
    int (*resident)(sw_ctx *c, int codes, int m, int *out);
};

template <int R, int W, int G>
DbShape db_shape_ops(double gcups, double clk1, double clk) {
    return DbShape{R, W, G, gcups, clk1, clk, db_profile_bytes<R, G>, db_scratch<R, W, G>, launch_db<R, W, G>, resident_blocks<R, W, G>};
}

DbShape db_shape_a(int k);      // the shapes of each translation unit
DbShape db_shape_b(int k);
DbShape db_shape_c(int k);
DbShape db_shape_d(int k);

}  // namespace swgb
