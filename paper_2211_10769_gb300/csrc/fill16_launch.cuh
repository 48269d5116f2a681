// fill16_launch.cuh -- launches of the packed 16-bit pair fill and of the
// straightening of its checkpoint columns, shared by the translation units of
// the local algorithm (fill16.cu) and of the others (fill16_variants.cu).
#pragma once
#include "sw_ctx.h"
#include "straighten.cuh"
#include "wavefront16.cuh"

#include <algorithm>

#ifndef CU
#define CU(x) do { if ((x) != cudaSuccess) { cudaGetLastError(); return SW_ECUDA; } } while (0)
#endif

namespace swgb {

// largest pair profile (small alphabets); larger alphabets take the int16 profile
inline constexpr size_t kPairProfileMax = 170 * 1024;
inline constexpr size_t kSharedMax = 227 * 1024;          // shared memory a block can have

template <int R, int W, int MODE, int PK, bool LEFT, bool LOCAL, int MINB = 1>
int launch16(sw_ctx *c, const FillLaunch &L, int K, long long tickets, int max_blocks) {
    auto kern = wavefront16_kernel<R, W, MODE, PK, LEFT, LOCAL, MINB>;
    const size_t smem = p16_shared_bytes<R, W>() + p16_profile_bytes(R, W, K, PK);
    static int attr_set[64] = {0};
    if (c->device >= 64 || !attr_set[c->device]) {
        const size_t cap = p16_shared_bytes<R, W>() + (PK == kP16Pair ? kPairProfileMax : p16_profile_bytes(R, W, kMaxAlphabet, PK));
        CU(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)std::min(cap, kSharedMax)));
        if (c->device < 64) attr_set[c->device] = 1;
    }
    int occ = 0;
    CU(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, (W + 2) * 32, smem));
    if (occ < 1) return SW_ECUDA;
    if (max_blocks > 0) occ = std::min(occ, max_blocks);
    const long long grid = std::min<long long>(tickets, (long long)occ * c->nsm);
    const int kp = kt_begin(c, SW_KT_FILL);
    kern<<<(unsigned)grid, (W + 2) * 32, smem, c->stream>>>(L);
    kt_end(c, kp);
    CU(cudaGetLastError());
    ++c->launches;
    return SW_OK;
}

// Whether a block of W compute warps at R rows a lane takes the pair profile for K residue codes (it has to fit).
template <int R, int W>
bool pair_profile_fits(int K) {
    const size_t p = p16_profile_bytes(R, W, K, kP16Pair);
    return p <= kPairProfileMax && p16_shared_bytes<R, W>() + p <= kSharedMax;
}

template <int R, int MODE, bool LEFT = false, int W = 4, bool LOCAL = true>
int launch16_pk(sw_ctx *c, const FillLaunch &L, int K, long long tickets, int B) {
    if (pair_profile_fits<R, W>(K)) return launch16<R, W, MODE, kP16Pair, LEFT, LOCAL>(c, L, K, tickets, B);
    if constexpr (R == 8 || R == 12 || R == 16) return launch16<R, W, MODE, kP16Int16, LEFT, LOCAL>(c, L, K, tickets, B);
    else return SW_EINVAL;                          // (p16_fits keeps other shapes to small alphabets)
}

template <int R, bool LOCAL>
int launch_straighten_r(sw_ctx *c, const FillTask *tasks, int ntasks, int max_rows, const DevScoring *sc) {
    const int wpt = (max_rows + 32 * R - 1) / (32 * R);
    const long long threads = 32LL * wpt * ntasks;
    straighten_kernel<R, LOCAL><<<(unsigned)((threads + kStraightThreads - 1) / kStraightThreads), kStraightThreads, 0,
                            c->stream>>>(tasks, ntasks, wpt, sc);
    CU(cudaGetLastError());
    ++c->launches;
    return SW_OK;
}

// Modes of one shape: left = the coarse-tile refills (checkpoint mode only), whose tasks enter the fill at a
// checkpoint column.
template <int R, bool LOCAL>
int launch16_mode4(sw_ctx *c, int mode, bool left, const FillLaunch &L, int K, long long tickets, int B) {
    if (left) return mode == kModeScoreCk ? launch16_pk<R, kModeScoreCk, true, 4, LOCAL>(c, L, K, tickets, B) : SW_EINVAL;
    switch (mode) {
        case kModeScore: return launch16_pk<R, kModeScore, false, 4, LOCAL>(c, L, K, tickets, B);
        case kModeScoreCk: return launch16_pk<R, kModeScoreCk, false, 4, LOCAL>(c, L, K, tickets, B);
        default: return SW_EINVAL;
    }
}

}  // namespace swgb
