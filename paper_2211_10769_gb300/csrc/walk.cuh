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

#include "wavefront.cuh"

namespace swgb {

struct WalkState {
    int32_t i, j;          // current cell (1-based rows / columns; 0 = border)
    int32_t state;         // 0 = H, 1 = E, 2 = F
    int32_t done;          // 0 running / needs tiles, 1 finished, 2 inconsistent bits
    int64_t nruns;         // run records {op: 0 = M, 1 = I, 2 = D; cells > 0} written so far;
                           // consecutive records may have the same op
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
constexpr int kWalkMinBT = 256;       // tiles at least this side

__device__ __forceinline__ int leading_zeros(unsigned v) { return __clz((int)v); }
__device__ __forceinline__ int leading_zeros(unsigned long long v) { return __clzll((long long)v); }

template <int R>
constexpr size_t walk_window_bytes(size_t word_bytes) {   // two windows, each below a group of zero words
    return 2 * (size_t)(kWinRows / R + 1) * kWinDiags * word_bytes;
}

// Four consecutive words of a row group, loaded and stored as vectors.
template <typename Word>
struct alignas(sizeof(Word) == 2 ? 8 : 16) Quad {
    unsigned v[sizeof(Word)];
};

template <typename Word>
__device__ __forceinline__ Quad<Word> load_quad(const Word *p) {
    Quad<Word> q;
    if constexpr (sizeof(Word) == 2) {
        const uint2 x = __ldcg(reinterpret_cast<const uint2 *>(p));
        q.v[0] = x.x; q.v[1] = x.y;
    } else {
#pragma unroll
        for (int k = 0; k < (int)sizeof(Word) / 4; ++k) {
            const uint4 x = __ldcg(reinterpret_cast<const uint4 *>(p) + k);
            q.v[4 * k] = x.x; q.v[4 * k + 1] = x.y; q.v[4 * k + 2] = x.z; q.v[4 * k + 3] = x.w;
        }
    }
    return q;
}

// Row groups [g_lo, g_lo + ng), diagonals (column - row, 0-based) [dlo, dlo + kWinDiags), dlo = 1 (mod 4), which
// puts a quad of diagonals at a multiple of four words of a tile's row group.
struct WalkWindow {
    int g_lo, ng, dlo;
};

template <typename Word>
__device__ __forceinline__ const Word *tile_ptr(const TileTable<Word> &T, const Word *const *tiles, int I, int J) {
    const int ti = I - T.I0, tj = J - (T.J0 + ti);
    return (ti >= 0 && tj >= 0 && ti < T.nI && tj < T.nJ) ? tiles[ti * T.nJ + tj] : nullptr;
}

// The window whose last row group is ghi; the first diagonal around the walk's.
template <int R>
__device__ __forceinline__ WalkWindow make_window(int ghi, int dlo) {
    constexpr int RG = kWinRows / R;
    const int glo = max(0, ghi - (RG - 1));
    return WalkWindow{glo, ghi - glo + 1, dlo};
}

__device__ __forceinline__ int window_diag(int d) { return ((d - kWinDiags / 2 - 1) & ~3) + 1; }

// Whether window m holds the cell (r0, c0) at least kWinMargin diagonals from either side.
template <int R>
__device__ __forceinline__ bool window_holds(const WalkWindow &m, int r0, int c0) {
    const int g = r0 / R - m.g_lo, d = c0 - r0 - m.dlo;
    return r0 >= 0 && g >= 0 && g < m.ng && d >= kWinMargin && d < kWinDiags - kWinMargin;
}

// Stage window m into win: a warp takes every (kStageThreads / 32)-th row group,
// four diagonals a lane, kStage independent quads in flight at a time.  A word that reaches
// over a tile's right edge is the union of the two tiles' words.  Missing tiles and
// columns left of the matrix read as 0.
template <typename Word, int R>
__device__ __forceinline__ void stage_window(const TileTable<Word> &T, const Word *const *tiles, const WalkWindow &m,
                                             Word *win, int t) {
    constexpr int kStep = kStageThreads / 32;              // row groups a thread advances
    constexpr int kStage = kWinRows / R / kStep < 6 ? kWinRows / R / kStep : 6;   // quads a thread loads at once
    static_assert(kWinDiags == 128, "a warp takes a row group");
    static_assert(R % 4 == 0 && kStep * R <= kWalkMinBT, "quads are aligned; a step leaves at most one tile");
    const int k = 4 * (t & 31), BT = T.BT;
    int g = t >> 5;
    // the thread's tile and its place in it, advanced with the groups (BT is a multiple of R)
    const int r = (m.g_lo + g) * R, q = m.dlo + k + r;
    int I = r / BT, lr = r - I * BT;
    int J = q >= 0 ? q / BT : -((-q + BT - 1) / BT), lq = q - J * BT;
    while (g < m.ng) {
        Quad<Word> v[kStage];
#pragma unroll
        for (int u = 0; u < kStage; ++u) {
            Quad<Word> x{};
            v[u] = Quad<Word>{};
            if (g + u * kStep < m.ng) {
                const size_t row = (size_t)(lr / R) * (size_t)T.ld;
                const Word *a = tile_ptr(T, tiles, I, J);
                if (a) v[u] = load_quad(a + row + lq + R - 1);
                if (lq > BT - R) {
                    const Word *b = tile_ptr(T, tiles, I, J + 1);
                    if (b) x = load_quad(b + row + lq - BT + R - 1);
#pragma unroll
                    for (int y = 0; y < (int)sizeof(Word); ++y) v[u].v[y] |= x.v[y];
                }
            }
            lr += kStep * R; lq += kStep * R;
            if (lr >= BT) { lr -= BT; ++I; }
            if (lq >= BT) { lq -= BT; ++J; }
        }
#pragma unroll
        for (int u = 0; u < kStage; ++u)
            if (g + u * kStep < m.ng) *reinterpret_cast<Quad<Word> *>(win + (g + u * kStep) * kWinDiags + k) = v[u];
        g += kStage * kStep;
    }
}

// Where a walk starts, for an alignment done in one round without a round trip to the
// host: at the end cell of the forward fill, reduced from its candidates by the walk's own
// warp 0 into *result, in state H, or nothing to walk (done = 3, parked at cell (1, 1), a
// cell every window can hold) when the local score is 0 or the end cell lies on the
// border, or when the error word is set: the fill then stopped early, and what stands in place
// of its candidates and decision words (an earlier call's) may lead anywhere, past the
// rows + columns run records there is room for.  A null task: the walk goes on from its state.
struct WalkStart {
    const FillTask *task;
    const int4 *cand;
    const DevScoring *scorings;
    int4 *result;
    const int *err;
};

__host__ __device__ __forceinline__ WalkState walk_start(int4 end, bool local, int err) {
    if (err != 0 || (local && end.x <= 0) || end.y <= 0 || end.z <= 0) return WalkState{1, 1, 0, 3, 0};
    return WalkState{end.y, end.z, 0, 0, 0};
}

template <typename Word, int R>
__global__ void __launch_bounds__(kWalkThreads, 1) walk_kernel(const TileTable<Word> T, const WalkStart start,
                                                          WalkState *st, int2 *runs,
                                                          int max_iters)
{
    static_assert(kWinRows % R == 0, "a window holds whole row groups");
    constexpr int kWinWords = (kWinRows / R + 1) * kWinDiags;   // a group of zero words, then the window's
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
    int4 end;
    if (start.task && warp == 0)
        end = reduce_candidates(*start.task, start.cand, start.scorings[start.task->scoring], lane);
    if (threadIdx.x == 0) {
        if (start.task) {
            *start.result = end;
            s_w = walk_start(end, start.scorings[start.task->scoring].alg == kAlgLocal, *start.err);
        } else {
            s_w = *st;
        }
        s_stop = s_w.done != 0;
        const int r0 = max(s_w.i - 1, 0), c0 = max(s_w.j - 1, 0);
        s_mw[0] = make_window<R>(r0 / R, window_diag(c0 - r0));
    }
    if (threadIdx.x < kWinDiags) { s_buf[threadIdx.x] = 0; s_buf[kWinWords + threadIdx.x] = 0; }
    s_buf += kWinDiags;
    __syncthreads();
    if (warp > 0 && !s_stop) stage_window<Word, R>(T, s_tiles, s_mw[0], s_buf, threadIdx.x - 32);
    __syncthreads();
    int it = 0;                                          // walk turns (warp 0)
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
            auto emit = [&](int op, int cnt) {
                if (lane == 0) out[nr] = make_int2(op, cnt);
                ++nr;
            };
            // the cell, relative to the window
            int rw = w.i - 1 - m.g_lo * R, dd = w.j - w.i - m.dlo, state = w.state;
            bool stop = false;                           // back to the host (or finished)
            while (true) {                               // (w.done is 0 here: every exit that sets it breaks)
                if (++it >= max_iters) { w.done = 2; stop = true; break; }
                if (rw < 0 || (unsigned)dd >= (unsigned)kWinDiags) break;   // out of the window
                const int g0 = (int)((unsigned)rw / R), x0 = rw - g0 * R;
                if (state == 0) {
                    // lane l: the walk's diagonal in the l-th group up, from row x0 (lane 0) or the group's last
                    // row; above the window's first group the words are 0, and columns left of the matrix read as 0
                    const int top = lane == 0 ? x0 : R - 1;
                    const Word wd = s_win[max(g0 - lane, -1) * kWinDiags + dd];
                    // a nibble is nonzero here where the H source is not "diagonal"; the top one first
                    const Wide bad = (((Wide)wd ^ kOnes) & (3 * kOnes)) << (kTop - 4 * top);
                    const unsigned ends = __ballot_sync(kFull, bad != 0);
                    if (ends == 0) {                     // all 32 groups go on
                        const int pos = x0 + 1 + 31 * R;
                        emit(0, pos);
                        rw -= pos;
                        continue;
                    }
                    const int cnt = leading_zeros(bad) >> 2;   // leading cells that go on
                    const int nib = (int)((Wide)wd >> (4 * max(top - cnt, 0))) & 15;
                    const int before = max(0, x0 + 1 - R + lane * R);
                    const int val = __shfl_sync(kFull, (before + cnt) | (nib << 16), __ffs(ends) - 1);
                    const int pos = val & 0xffff, nbk = val >> 16, src = nbk & 3;
                    if (pos > 0) emit(0, pos);
                    rw -= pos;
                    if (src == 0) {                      // a zero cell, a tile that was not recomputed, or an edge
                        const int r = rw + m.g_lo * R, c = r + m.dlo + dd;
                        if (rw < 0 || c < 0) break;
                        if (tile_ptr(T, s_tiles, r / T.BT, c / T.BT)) w.done = 1;
                        stop = true;
                        break;
                    }
                    if (src == 2) {
                        if (nbk & 4) { emit(1, 1); --dd; }   // opened here: a gap of one cell
                        else state = 1;
                    } else {
                        if (nbk & 8) { emit(2, 1); --rw; ++dd; }
                        else state = 2;
                    }
                } else {
                    // lane p: the cell p columns to the left (E) or p rows up (F); a cell of the path in a gap state
                    // has a nonzero nibble (its H source is not "zero"), so 0 is a tile that was not recomputed
                    const bool inE = state == 1;
                    const int rp = inE ? rw : rw - lane, d = inE ? dd - lane : dd + lane;
                    const int gp = (int)((unsigned)max(rp, 0) / R);
                    const bool in = rp >= 0 && d >= 0 && d < kWinDiags;
                    const Word wd = s_win[gp * kWinDiags + min(max(d, 0), kWinDiags - 1)];
                    const int nib = in ? (int)((Wide)wd >> (4 * max(rp - gp * R, 0))) & 15 : 16;
                    const bool end = nib >= 16 || nib == 0 || (nib & (inE ? 4 : 8)) != 0;
                    const unsigned ends = __ballot_sync(kFull, end);
                    const int pos = ends ? __ffs(ends) - 1 : 32;
                    const int nbk = __shfl_sync(kFull, nib, pos & 31);
                    const bool opened = ends != 0 && nbk != 0 && nbk < 16;
                    const int step = pos + (opened ? 1 : 0);   // the extensions, and the opening cell
                    if (step > 0) emit(state, step);
                    if (inE) dd -= step; else { rw -= step; dd += step; }
                    if (opened) { state = 0; continue; }
                    if (ends == 0) continue;
                    // the window's edge (nbk 16), a column left of the matrix, or a missing tile: ask the host
                    if (nbk == 0 && rw + m.g_lo * R + m.dlo + dd >= 0) stop = true;
                    break;
                }
            }
            w.i = rw + m.g_lo * R + 1;
            w.j = w.i + m.dlo + dd;
            w.state = state;
            if (w.done == 0 && (w.i <= 0 || w.j <= 0)) {   // the border; a gap cannot reach it
                w.done = state == 0 ? 1 : 2;
                stop = true;
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
            if (s_redo) s_mw[nxt] = make_window<R>(r0 / R, window_diag(c0 - r0));
        }
        __syncthreads();
        if (s_redo) {
            if (warp > 0) stage_window<Word, R>(T, s_tiles, s_mw[nxt], s_buf + nxt * kWinWords, threadIdx.x - 32);
            __syncthreads();
        }
        cur = nxt;
    }
    if (threadIdx.x == 0) *st = s_w;
}

}  // namespace swgb
