// straighten.cuh -- checkpoint columns of the packed pair fill brought to one
// column, so that traceback tiles may have any number of rows a lane.
//
// The packed fill (wavefront16.cuh) stores a checkpoint column at one step of
// its sweep, when lane l's top half (R/2 rows) is at column c - 2l and its
// bottom half at c - 2l - 1.  Here one warp takes the R * 32 rows of one such
// warp and runs the remaining triangle: position v = 2l (top half) or 2l + 1
// (bottom) advances v columns, in step with its neighbours -- the top half's
// k-th column needs lane l-1's bottom half after its (k-1)-th, the bottom
// half's needs this lane's top half after its (k-1)-th -- so that every row
// ends at column c: a 63-step wavefront inside the warp.
//
// Apart from the tiles, because the fill's rows a lane are chosen for the
// length of its strip chain and the tiles' for their own: 200 kbp runs 12 and
// 8, 1 Mbp 26 and 8.
#pragma once
#include "wavefront.cuh"

namespace swgb {

constexpr int kStraightThreads = 128;

// One warp per R * 32 rows of every task with left_split == R; tasks [0, ntasks), wpt warps each (the most any needs).
template <int R, bool LOCAL>
__global__ void __launch_bounds__(kStraightThreads)
straighten_kernel(const FillTask *tasks, int ntasks, int wpt, const DevScoring *scorings)
{
    constexpr int H = R / 2;
    __shared__ int8_t mat[kMaxAlphabet * (kMaxAlphabet + 1)];
    __shared__ uint8_t res[kStraightThreads / 32][64];   // per warp: the columns c - 63 .. c
    const int lane = threadIdx.x & 31;
    const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const DevScoring &SC = scorings[tasks[0].scoring];   // one scoring a launch
    const int K = SC.K, go = SC.go, ge = SC.ge;
    // score of a row's residue against a column's; residue K (padding rows) at kPadScore
    for (int k = threadIdx.x; k < K * (K + 1); k += blockDim.x) {
        const int x = k % (K + 1), y = k / (K + 1);
        mat[k] = x < K ? SC.mat[x * K + y] : (int8_t)kPadScore;
    }
    __syncthreads();
    if (w >= ntasks * wpt) return;
    const FillTask &T = tasks[w / wpt];
    const int base = (w % wpt) * 32 * R;                 // first row of the warp within the task
    const int rows = T.rows;
    if (!T.straight || T.left_split != R || base >= rows) return;
    uint8_t *const col = res[threadIdx.x >> 5];
    for (int k = lane; k < 64; k += 32) col[k] = (uint8_t)min((int)T.b[k - 64], K - 1);
    __syncwarp();
    const int grow = base + lane * R;
    int U[R], E[R], code[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        int2 v = make_int2(-go, kNeg);
        code[r] = K;
        if (grow + r < rows) {
            v = __ldcg(T.left + grow + r);
            code[r] = min((int)T.a[grow + r], K - 1);
        }
        U[r] = v.x; E[r] = v.y;
    }
    const bool in = grow < rows;
    const int2 at = in ? __ldcg(T.left_aux + grow / H) : make_int2(-go, kNeg);       // top half
    const int2 ab = in ? __ldcg(T.left_aux + grow / H + 1) : make_int2(-go, kNeg);   // bottom half
    int udT = at.x, fT = at.y;        // row above the top half at its column; F of its last row
    int udB = ab.x, fB = ab.y;        // the same for the bottom half
#pragma unroll 1
    for (int k = 1; k < 64; ++k) {
        // lane l-1's bottom half after its (k-1)-th column: the row above this lane's top half
        const int uupT = __shfl_up_sync(kFull, U[R - 1], 1);
        const int fupT = __shfl_up_sync(kFull, fB, 1);
        if (k <= 2 * lane + 1) {
            // both halves side by side (two independent chains); the top half stops one column earlier
            const bool top = k <= 2 * lane;
            const int8_t *mt = mat + col[min(63, 64 + k - 2 * lane - 1)] * (K + 1);   // column c - 2l + k
            const int8_t *mb = mat + col[64 + k - 2 * lane - 2] * (K + 1);            // column c - 2l - 1 + k
            const int uupB = U[H - 1];
            int f = __viaddmax_s32(fupT, -ge, uupT), g = __viaddmax_s32(fT, -ge, uupB);
            int dt = udT, db = udB;
#pragma unroll
            for (int x = 0; x < H; ++x) {
                const int ut = U[x], ub = U[H + x];
                const int et = __viaddmax_s32(E[x], -ge, ut), eb = __viaddmax_s32(E[H + x], -ge, ub);
                const int xt = (LOCAL ? __viaddmax_s32_relu(dt, mt[code[x]] + go, et) : __viaddmax_s32(dt, mt[code[x]] + go, et)) - go;
                const int xb = (LOCAL ? __viaddmax_s32_relu(db, mb[code[H + x]] + go, eb) : __viaddmax_s32(db, mb[code[H + x]] + go, eb)) - go;
                if (top) { U[x] = __viaddmax_s32(f, -go, xt); E[x] = et; }
                U[H + x] = __viaddmax_s32(g, -go, xb);
                E[H + x] = eb;
                dt = ut;
                db = ub;
                if (x + 1 < H) {
                    f = __viaddmax_s32(f, -ge, xt);
                    g = __viaddmax_s32(g, -ge, xb);
                }
            }
            if (top) { fT = f; udT = uupT; }
            fB = g;
            udB = uupB;
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (grow + r < rows) T.straight[grow + r] = make_int2(U[r], E[r]);
}

}  // namespace swgb
