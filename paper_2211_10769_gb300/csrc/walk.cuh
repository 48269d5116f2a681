// walk.cuh -- the traceback walk over recomputed decision bits (paper
// Section 2.2, reconstruction phase).
//
// The matrix is cut into square tiles of BT x BT cells.  A round of the
// reconstruction recomputes the decision bits of a set of tiles (a band
// around the path) and this kernel walks the canonical path through them:
//
//   state H: stop if the H source is zero; diagonal -> emit M, go up-left;
//            source E -> state E; source F -> state F;
//   state E: emit I, go left; back to H if the E-opened bit is set;
//   state F: emit D, go up; back to H if the F-opened bit is set.
//
// The bits come in words of R nibbles along the diagonal (wavefront.cuh): word
// q of row group g holds row g R + x's nibble of column q + x.  The walk is one
// warp's chain of dependent lookups, so what bounds it is the number of
// lookups and the latency of each:
//   * it reads words from shared memory: a window of row groups by diagonals
//     around the walk's (kWinRows rows, kWinDiags diagonals; word q of group g lies
//     on diagonal q - g R, so the window is a rectangle).  Warp 0 walks while the
//     other warps stage the same diagonals of the groups above into a second
//     buffer;
//   * in state H lane l reads the word of the walk's diagonal l groups up: 32 R
//     cells at once, in which one vote and one shuffle find the cell that ends the
//     run and its whole nibble, which settles a gap of one cell.  In states E and F
//     the lanes read the next 32 cells of the row or column.
// (Before, the words were columns of a row group: a lane read one or two cells, 64
// a turn at about 780 clocks, and windows met at most 2 x 2 tiles.  200 kbp:
// 1.65 ms, 100 kbp global with unrelated ends 2.9 ms, 3 kbp on 256-row tiles 129 us.)
// The walk stops when it reaches a zero cell or the border (done = 1), or
// when its next cell lies in a tile that was not recomputed this round
// (done = 0, the host computes that tile next).
#pragma once
#include <type_traits>

#include "sw_device.cuh"

namespace swgb {

struct WalkState {
    int32_t i, j;          // current cell (1-based rows / columns; 0 = border)
    int32_t state;         // 0 = H, 1 = E, 2 = F
    int32_t done;          // 0 running / needs tiles, 1 finished, 2 inconsistent bits
    int64_t nruns;         // run records written so far
    int32_t cur_op;        // op of the open run (0 = M, 1 = I, 2 = D, -1 = none)
    int32_t cur_len;
};

// The tiles recomputed in one round: for each tile row I in [I0, I0 + nI), a
// window of nJ tile columns that follows the diagonal, [J0 + (I - I0),
// J0 + (I - I0) + nJ); a null entry means the tile was not computed.  Words of
// a tile: [local row / R][ld], word q (local) at index q + R - 1.
template <typename Word>
struct TileTable {
    const Word *const *bits;   // nI * nJ entries
    int32_t I0, J0, nI, nJ;
    int32_t BT;                // tile side
    int32_t ld;                // words per row group
};

constexpr int kWalkTableMax = 4096;   // tile-table entries cached in shared memory
constexpr int kWinRows = 768;         // rows of a window (a multiple of every R)
constexpr int kWinDiags = 128;        // diagonals of a window, the walk's in the middle
constexpr int kWinMargin = 16;        // diagonals a staged window must leave either side of the walk's
constexpr int kStageThreads = 512;    // threads staging a window (warps 1..16)
constexpr int kWalkThreads = 32 + kStageThreads;   // warp 0 walks
constexpr int kStage = 8;             // window words a thread loads at once
constexpr int kWalkMinBT = 256;       // tiles at least this side

__device__ __forceinline__ int leading_zeros(unsigned v) { return __clz((int)v); }
__device__ __forceinline__ int leading_zeros(unsigned long long v) { return __clzll((long long)v); }

template <int R>
constexpr size_t walk_window_bytes(size_t word_bytes) { return 2 * (size_t)(kWinRows / R) * kWinDiags * word_bytes; }

// Row groups [g_lo, g_lo + ng), diagonals (column - row, 0-based) [dlo, dlo + kWinDiags).
struct WalkWindow {
    int g_lo, ng, dlo;
};

template <typename Word>
__device__ __forceinline__ const Word *tile_ptr(const TileTable<Word> &T, const Word *const *tiles, int I, int J) {
    const int ti = I - T.I0, tj = J - (T.J0 + ti);
    return (ti >= 0 && tj >= 0 && ti < T.nI && tj < T.nJ) ? tiles[ti * T.nJ + tj] : nullptr;
}

// The window whose last row group is ghi.
template <int R>
__device__ __forceinline__ WalkWindow make_window(int ghi, int dlo) {
    constexpr int RG = kWinRows / R;
    const int glo = max(0, ghi - (RG - 1));
    return WalkWindow{glo, ghi - glo + 1, dlo};
}

// Whether window m holds the cell (r0, c0) at least kWinMargin diagonals from either side.
template <int R>
__device__ __forceinline__ bool window_holds(const WalkWindow &m, int r0, int c0) {
    const int g = r0 / R - m.g_lo, d = c0 - r0 - m.dlo;
    return r0 >= 0 && g >= 0 && g < m.ng && d >= kWinMargin && d < kWinDiags - kWinMargin;
}

// Stage window m into win: staging thread t (of kStageThreads) takes diagonal
// t % kWinDiags of every kStageThreads / kWinDiags-th row group, kStage
// independent words in flight at a time.  A word that reaches over a tile's right
// edge is the union of the two tiles' words.  Missing tiles and columns left of
// the matrix read as 0.
template <typename Word, int R>
__device__ __forceinline__ void stage_window(const TileTable<Word> &T, const Word *const *tiles, const WalkWindow &m,
                                             Word *win, int t) {
    constexpr int kStep = kStageThreads / kWinDiags;       // row groups a thread advances
    static_assert(kStageThreads % kWinDiags == 0, "whole row groups per pass");
    const int k = t % kWinDiags, BT = T.BT;
    int g = t / kWinDiags;
    // the thread's tile and its place in it, advanced with the groups (BT is a multiple of R)
    const int r = (m.g_lo + g) * R, q = m.dlo + k + r;
    int I = r / BT, lr = r - I * BT;
    int J = q >= 0 ? q / BT : -((-q + BT - 1) / BT), lq = q - J * BT;
    while (g < m.ng) {
        Word v[kStage], x[kStage];
#pragma unroll
        for (int u = 0; u < kStage; ++u) {
            v[u] = 0; x[u] = 0;
            if (g + u * kStep < m.ng) {
                const size_t row = (size_t)(lr / R) * (size_t)T.ld;
                const Word *a = tile_ptr(T, tiles, I, J);
                if (a) v[u] = __ldcg(a + row + lq + R - 1);
                if (lq > BT - R) {
                    const Word *b = tile_ptr(T, tiles, I, J + 1);
                    if (b) x[u] = __ldcg(b + row + lq - BT + R - 1);
                }
            }
            lr += kStep * R; lq += kStep * R;
            while (lr >= BT) { lr -= BT; ++I; }
            while (lq >= BT) { lq -= BT; ++J; }
        }
#pragma unroll
        for (int u = 0; u < kStage; ++u)
            if (g + u * kStep < m.ng) win[(g + u * kStep) * kWinDiags + k] = v[u] | x[u];
        g += kStage * kStep;
    }
}

// The walk's start taken from the end cell reduced on the device (res: score,
// row, column), for an alignment done in one round without a round trip to
// the host: the end cell in state H, or nothing to walk (done = 3, parked at
// cell (1, 1), a cell every window can hold) when the local score is 0 or the
// end cell lies on the border.
static __global__ void walk_start_kernel(const int4 *res, int local, WalkState *st) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const int4 r = *res;
    WalkState w{r.y, r.z, 0, 0, 0, -1, 0};
    if ((local && r.x <= 0) || r.y <= 0 || r.z <= 0) { w.i = 1; w.j = 1; w.done = 3; }
    *st = w;
}

template <typename Word, int R>
__global__ void __launch_bounds__(kWalkThreads, 1) walk_kernel(const TileTable<Word> T, WalkState *st, int2 *runs,
                                                          long long max_iters)
{
    static_assert(kWinRows % R == 0, "a window holds whole row groups");
    constexpr int kWinWords = (kWinRows / R) * kWinDiags;
    using Wide = typename std::conditional<(R > 8), unsigned long long, unsigned>::type;   // a word, registers whole
    constexpr int kTop = 8 * (int)sizeof(Wide) - 4;        // shift of a Wide's top nibble
    constexpr Wide kOnes = (Wide)(0x1111111111111111ull >> (64 - 4 * R));
    extern __shared__ __align__(16) unsigned char walk_smem[];
    Word *s_buf = reinterpret_cast<Word *>(walk_smem);   // two windows
    __shared__ const Word *s_tiles[kWalkTableMax];
    __shared__ WalkState s_w;
    __shared__ WalkWindow s_mw[2];
    __shared__ int s_stop, s_redo;
    if (blockIdx.x != 0) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ntab = T.nI * T.nJ;
    if (ntab > kWalkTableMax || T.BT < kWalkMinBT || T.BT % R != 0 || T.ld < T.BT + R - 1) {   // the host keeps within these
        if (threadIdx.x == 0) st->done = 2;
        return;
    }
    for (int k = threadIdx.x; k < ntab; k += blockDim.x) s_tiles[k] = T.bits[k];
    if (threadIdx.x == 0) {
        s_w = *st;
        s_stop = s_w.done != 0;
        const int r0 = max(s_w.i - 1, 0), c0 = max(s_w.j - 1, 0);
        s_mw[0] = make_window<R>(r0 / R, c0 - r0 - kWinDiags / 2);
    }
    __syncthreads();
    if (warp > 0 && !s_stop) stage_window<Word, R>(T, s_tiles, s_mw[0], s_buf, threadIdx.x - 32);
    __syncthreads();
    long long it = 0;                                    // walk turns (warp 0)
    int cur = 0;
    while (!s_stop) {
        const int nxt = cur ^ 1;
        const WalkWindow m = s_mw[cur];
        // the same diagonals above the current window (none above the first row)
        const WalkWindow up = m.g_lo > 0 ? make_window<R>(m.g_lo - 1, m.dlo) : WalkWindow{0, 0, 0};
        if (warp > 0) {
            if (threadIdx.x == 32) s_mw[nxt] = up;
            if (up.ng > 0) stage_window<Word, R>(T, s_tiles, up, s_buf + nxt * kWinWords, threadIdx.x - 32);
        } else {
            const Word *s_win = s_buf + cur * kWinWords;
            WalkState w = s_w;
            int nr = 0;                                  // run records written in this window
            int2 *out = runs + w.nruns;
            // every lane keeps the same (uniform) run state; lane 0 stores the records
            auto emit = [&](int op, int cnt) {
                if (op == w.cur_op) { w.cur_len += cnt; return; }
                if (w.cur_len > 0) {
                    if (lane == 0) out[nr] = make_int2(w.cur_op, w.cur_len);
                    ++nr;
                }
                w.cur_op = op;
                w.cur_len = cnt;
            };
            bool stop = false;                           // back to the host (or finished)
            while (true) {                               // (w.done is 0 here: every exit that sets it breaks)
                if (++it >= max_iters) { w.done = 2; stop = true; break; }
                const int r = w.i - 1, c = w.j - 1;
                const int g0 = (int)((unsigned)max(r, 0) / R), x0 = r - g0 * R, gl = g0 - m.g_lo, dd = c - r - m.dlo;
                if (w.state == 0) {
                    if (w.i == 0 || w.j == 0) { w.done = 1; stop = true; break; }
                    if (dd < 0 || dd >= kWinDiags) break;   // a gap ran out of the window
                    // lane l: the walk's diagonal in the l-th group up, from row x0 (lane 0) or the group's last row
                    const int g = gl - lane, top = lane == 0 ? x0 : R - 1;
                    const Word wd = s_win[max(g, 0) * kWinDiags + dd];
                    // a nibble is nonzero here where the H source is not "diagonal"; the top one first
                    const Wide bad = (((Wide)wd ^ kOnes) & (3 * kOnes)) << (kTop - 4 * top);
                    const bool in = g >= 0;
                    const int cnt = bad ? leading_zeros(bad) >> 2 : top + 1;   // leading cells that go on
                    const bool end = !in || bad != 0;
                    const unsigned ends = __ballot_sync(kFull, end);
                    const int before = lane == 0 ? 0 : x0 + 1 + (lane - 1) * R;
                    const int nib = in ? (int)((Wide)wd >> (4 * max(top - cnt, 0))) & 15 : 16;
                    const int lim = min(r, c) + 1;       // cells up to the border
                    if (ends == 0) {                     // all 32 groups go on
                        const int pos = min(x0 + 1 + 31 * R, lim);
                        emit(0, pos);
                        w.i -= pos;
                        w.j -= pos;
                        continue;
                    }
                    const int val = __shfl_sync(kFull, (before + (in ? cnt : 0)) | (nib << 16), __ffs(ends) - 1);
                    const int pos = min(val & 0xffff, lim), nbk = val >> 16;
                    if (pos > 0) emit(0, pos);
                    w.i -= pos;
                    w.j -= pos;
                    if (pos == lim) continue;            // the border
                    if (nbk == 16) break;                // the window's first row: the next window starts here
                    const int src = nbk & 3;
                    if (src == 0) {                      // a zero cell, or a tile that was not recomputed
                        if (tile_ptr(T, s_tiles, (r - pos) / T.BT, (c - pos) / T.BT)) w.done = 1;
                        stop = true;
                        break;
                    }
                    w.state = src == 2 ? 1 : 2;
                    if (nbk & (src == 2 ? 4 : 8)) {      // opened here: a gap of one cell
                        emit(w.state, 1);
                        if (src == 2) --w.j; else --w.i;
                        w.state = 0;
                    }
                } else {
                    // lane p: the cell p columns to the left (E) or p rows up (F); a cell of the path in a gap state
                    // has a nonzero nibble (its H source is not "zero"), so 0 is a tile that was not recomputed
                    const bool inE = w.state == 1;
                    const int rp = inE ? r : r - lane, d = inE ? dd - lane : dd + lane;
                    const int gp = (int)((unsigned)max(rp, 0) / R), gw = gp - m.g_lo;
                    const bool out_m = rp < 0 || (inE && c - lane < 0);
                    const bool in = gw >= 0 && d >= 0 && d < kWinDiags;
                    const Word wd = s_win[max(gw, 0) * kWinDiags + min(max(d, 0), kWinDiags - 1)];
                    int nib = (int)((Wide)wd >> (4 * max(rp - gp * R, 0))) & 15;
                    nib = out_m ? 17 : (in ? nib : 16);
                    const bool end = nib >= 16 || nib == 0 || (nib & (inE ? 4 : 8)) != 0;
                    const unsigned ends = __ballot_sync(kFull, end);
                    const int pos = ends ? __ffs(ends) - 1 : 32;
                    const int nbk = __shfl_sync(kFull, nib, pos & 31);
                    const bool opened = ends != 0 && nbk != 0 && nbk < 16;
                    const int step = pos + (opened ? 1 : 0);   // the extensions, and the opening cell
                    if (ends != 0 && nbk == 17) { w.done = 2; stop = true; break; }   // a gap cannot reach the border
                    if (step > 0) emit(w.state, step);
                    if (inE) w.j -= step; else w.i -= step;
                    if (opened) { w.state = 0; continue; }
                    if (ends == 0) continue;
                    if (nbk == 0) stop = true;           // missing tile: ask the host
                    break;                               // (nbk 16: the window's edge)
                }
            }
            if (lane == 0) {
                w.nruns += nr;
                s_w = w;
                s_stop = stop;
            }
        }
        __syncthreads();
        if (s_stop) break;
        // the staged window serves if it holds the walk's cell with room to both sides
        if (threadIdx.x == 0) {
            const int r0 = max(s_w.i - 1, 0), c0 = max(s_w.j - 1, 0);
            s_redo = !window_holds<R>(s_mw[nxt], r0, c0);
            if (s_redo) s_mw[nxt] = make_window<R>(r0 / R, c0 - r0 - kWinDiags / 2);
        }
        __syncthreads();
        if (s_redo) {
            if (warp > 0) stage_window<Word, R>(T, s_tiles, s_mw[nxt], s_buf + nxt * kWinWords, threadIdx.x - 32);
            __syncthreads();
        }
        cur = nxt;
    }
    if (threadIdx.x == 0) {
        WalkState w = s_w;
        if (w.done == 1 && w.cur_len > 0) {
            runs[w.nruns++] = make_int2(w.cur_op, w.cur_len);
            w.cur_len = 0;
            w.cur_op = -1;
        }
        *st = w;
    }
}

}  // namespace swgb
