// wavefront16.cuh -- intra-task Smith-Waterman/Gotoh fill of one pair in
// packed 16-bit lanes (paper Section 2.1: one matrix, all processing
// elements cooperate and pass border elements to their neighbours).
//
// The block layout is the one of wavefront.cuh (W compute warps per strip of
// W*32*R rows, an input and an output warp, strips chained through a global
// boundary-row ring), but every lane holds two wavefront positions, packed
// into the two 16-bit halves of its registers:
//
//   * lane t owns rows [tR, tR + R) of its warp; the top half, rows
//     [tR, tR + R/2), lives in the low 16 bits and at step s computes column
//     s - 2t; the bottom half, rows [tR + R/2, tR + R), lives in the high
//     16 bits and computes column s - 2t - 1;
//   * the bottom half's row above is this lane's top half one step earlier
//     (a register); the top half's is lane t-1's bottom half one step
//     earlier (a shuffle), or the strip's boundary row for lane 0;
//   * so one __viaddmax_s16x2 advances two cells, and the vertical
//     dependency chain of a step is R/2 packed operations long.
//
// What bounds it.  A pair's strips form one chain of warps, at 200 kbp one
// compute warp per SM sub-partition, so a step runs at the pace of a single
// warp: its dependent chain (the shuffle, then the F chain through R/2 rows)
// and the instructions around it, which a lone warp issues at 0.73 a clock at
// most (measured with all SMs busy, loops longer than about 100
// instructions).  So the step is kept short; everything that can be done once
// per chunk of 32 steps, or once per sweep, is:
//
//   * one base per warp and no scaling (below): a shuffled value needs no
//     conversion;
//   * the bottom half's (H - open, F) go to the next lane, and to the next
//     warp's ring, as one packed word: one shuffle, one select, one store;
//   * the end cell's row and column are not tracked; a chunk only keeps its
//     largest value per half-lane (half a vimax3 a row), and the place is
//     looked up once, at the end of the sweep (p16_locate);
//   * the columns past the last one have profile offsets too (padding), so
//     that every chunk runs the same unrolled loop.
//
// 45 instructions a step at 12 rows a lane (77 before), 91 clocks in the
// loop.  200 kbp score fill 18.85 -> 15.2 ms, 1 Mbp (16 rows a lane) 332 ->
// 276 ms (GB300, 2,070 MHz).  Tried on the same code: four ALU operations a
// cell pair and two plain subtractions, as in the database search (26 rows a lane
// 207 -> 229 clocks a step, 12 rows 115.5 -> 117.6: a lone warp has no issue slots
// for the extra instruction); a third step of skew per lane to take the
// shuffle off the chain (the longer fill eats the gain); unrolling 8 (16.4
// ms) and 32 steps (18.4 ms) instead of 16.
//
// Exact 16-bit values.  A warp keeps one base B: absolute value = B + stored
// value.  H cannot change faster than
//   |H(p) - H(q)| <= D (max S + extend) + 2 open,   D = row + column distance
// (a path through p or q bends to the other cell for one gap each way; a row
// or column more earns max S at most and saves an extension).  U = H - open,
// E, F, X and the sums the instructions form lie within 3 open + extend +
// |S| + max S of a neighbouring H.  All cells a warp touches in one chunk lie
// within 32R rows and kP16Pos + kP16CH columns of each other, so all its
// values lie within p16_spread of lane 0's first row (the reference).  At each
// chunk start the warp moves its base if the reference has left kP16Center
// +- kP16Slack (never below 0).  With the spread at most kP16Span:
//   * B = 0: values are absolute, the 0 floor of H is the hardware relu;
//   * B > 0: every value of the warp lies in (0, 32767), so the relu never
//     fires -- as in the true recurrence, where every such H is above B > 0.
// The strips exchange absolute rows (plain int32 in global memory); a warp's
// ring entries are relative to its base of that chunk, which it stores beside
// them.  The result does not depend on the bases.
//
// End cell: the first cell in row-major order that holds the largest H.  A
// half-lane (R/2 rows of a lane) is a row range, ordered by 2 lane + half.  At a
// chunk's end the warp compares the largest value of the chunk with its best:
// larger, or equal in an earlier half-lane, makes this chunk the best's, and
// the chunk's snapshot (the lane states at its start, written to shared memory
// every chunk) is kept; equal in the same half-lane, the snapshot is kept
// beside the first one, because that chunk may hold an earlier row.  At the
// end of the sweep the kept chunks are run again with a test per cell
// (p16_locate).  A third equal chunk makes the warp look the kept ones up at
// once.  Cells outside the task never decide: a padding cell is below every
// real one, or (gaps that cost nothing) equal to a real one in the same or an
// earlier row of an earlier step, and p16_locate tests real cells only.
//
// Query profile: for small alphabets a pair profile, one packed word per
// (residue of the top half, residue of the bottom half) and packed row; else
// an int16 profile whose two words per packed row are merged with one prmt;
// batches, which want several blocks an SM, an int8 one a quarter its size.
//
// Modes: score (end-cell candidate per strip) and score with checkpoints
// (strip bottom rows, and staircase checkpoint columns in the two-positions
// form that FillTask::left_split describes).
#pragma once
#include "wavefront.cuh"

namespace swgb {

constexpr int kNeg16p = -16384;     // -infinity of a packed 16-bit lane
constexpr int kP16Center = 16384;   // stored value of a warp's reference once B > 0
constexpr int kP16Slack = 1024;     // drift of the reference from kP16Center before the base moves
constexpr int kP16Span = 15000;     // largest value spread (p16_spread) the packed fill accepts
constexpr int kP16QS = 512;         // columns of the strip's boundary ring (channel 0)
constexpr int kP16RS = 256;         // steps of the rings between the warps
constexpr int kP16Pos = 64;         // wavefront positions per warp (two per lane)
constexpr int kP16CH = 32;          // steps per chunk (hand-off, base change; 16 measured slower)
constexpr int kP16Lag = kP16Pos - 1;   // lane 31's bottom half trails lane 0's top half
// Columns left of the last warp's published count whose profile offsets may still be read: lane 31's, one more for
// the words of the step before, and the chunk left of the task that a block's first strip starts with, when
// nothing is published yet.
constexpr int kP16Back = kP16Pos + kP16CH + 2;
// Columns that may have their profile offset in the ring once the last warp has published `done` columns.
__host__ __device__ constexpr int p16_offset_room(int done) { return done + kQB - kP16Back; }
// steps per unrolled body (12 rows a lane at 200 kbp: 8, 16, 32 steps 16.4, 15.2, 18.4 ms; 26 rows: 8 and 16 steps
// 212 and 205 clocks a step)
constexpr int kP16Unroll = 16;
// An I/O warp with nothing to move sleeps this long: polling takes issue slots from the compute warp
// beside it (200 kbp: 48 ns 15.5 ms, 128 ns 15.25 ms, 256 ns 15.15 ms)
constexpr int kP16IdleNs = 256;

// Profile kinds of the packed fill.
enum P16Prof { kP16Pair = 0, kP16Int16 = 1, kP16Int8 = 2 };

// Profile words a lane loads per step, and the bytes of its slot in an int8 profile row.
__host__ __device__ constexpr int p16_words(int R, int PK) { return PK == kP16Int8 ? R / 4 : R / 2; }
__host__ __device__ constexpr int p16_slot8(int R) { return R <= 8 ? 8 : 16; }

// Bound on the spread of all values a warp touches during one chunk (see the header); the packed
// fill is exact when it is at most kP16Span.
inline long long p16_spread(int R, int go, int ge, int max_s, int min_s) {
    const long long L = (long long)ge + (max_s > 0 ? max_s : 0);
    const long long D = 32LL * R + kP16Pos + kP16CH + 4;
    const long long neg = -min_s > 128 ? -min_s : 128;          // padding residues score -128
    return D * L + 3LL * go + ge + neg + (max_s > 0 ? max_s : 0);
}

// Bytes of the packed fill's query profile for K residue codes.
inline size_t p16_profile_bytes(int R, int W, int K, int pk) {
    const size_t HC = (size_t)W * 32 * R;
    if (pk == kP16Int8) return (size_t)(K + 1) * W * 32 * p16_slot8(R);
    return pk == kP16Pair ? (size_t)(K + 1) * (K + 1) * (HC / 2) * 4 : (size_t)(K + 1) * HC * 2;
}

// Words of a lane's state in a snapshot: U, E, fb, udiag0, rounded up to whole 16-byte stores.
__host__ __device__ constexpr int p16_snap_words(int R) { return (R + 2 + 3) / 4 * 4; }

__device__ __forceinline__ unsigned p16_pack(int lo, int hi) {
    return (unsigned)(lo & 0xffff) | ((unsigned)hi << 16);
}
__device__ __forceinline__ int p16_lo(unsigned v) { return (int)(short)(v & 0xffffu); }
__device__ __forceinline__ int p16_hi(unsigned v) { return (int)v >> 16; }

template <unsigned sel>
__device__ __forceinline__ unsigned prmt_c(unsigned a, unsigned b) {
    unsigned d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "n"(sel));
    return d;
}

__device__ __forceinline__ unsigned prmt_v(unsigned a, unsigned b, unsigned sel) {
    unsigned d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}

// low half = 16-bit half ha of a, high half = 16-bit half hb of b
template <int ha, int hb>
__device__ __forceinline__ unsigned p16_halves(uint32_t a, uint32_t b) {
    return prmt_c<(2 * ha) | ((2 * ha + 1) << 4) | ((4 + 2 * hb) << 8) | ((5 + 2 * hb) << 12)>(a, b);
}

// pair profile: a lane's H words of one residue pair in chunks of 4, 2 and 1 words, each kind
// [chunk][lane] so that a warp's load is conflict-free
template <int H> struct P16Chunks {
    static constexpr int N4 = H == 6 ? 0 : H / 4, N2 = H == 6 ? 3 : (H % 4) / 2, N1 = H % 2;
};
// word index of packed row k of lane g (of NL) within one residue pair's H * NL words
template <int H>
__device__ __forceinline__ int p16_pair_word(int k, int g, int NL) {
    using C = P16Chunks<H>;
    if (k < 4 * C::N4) return ((k >> 2) * NL + g) * 4 + (k & 3);
    k -= 4 * C::N4;
    if (k < 2 * C::N2) return 4 * C::N4 * NL + ((k >> 1) * NL + g) * 2 + (k & 1);
    return (4 * C::N4 + 2 * C::N2) * NL + g;
}

// Profile words of one step (H per lane) for the column whose profile offset is off.
template <int R, int PK, int NL>
__device__ __forceinline__ void p16_load(const int8_t *prof, int g, int off, uint32_t (&w)[p16_words(R, PK)]) {
    constexpr int H = R / 2;
    if constexpr (PK == kP16Int8) {
        static_assert(R == 8 || R == 12 || R == 16, "int8 profile loads");
        const int8_t *p = prof + off + g * p16_slot8(R);
        if constexpr (R == 8) {
            const uint2 v = *reinterpret_cast<const uint2 *>(p);
            w[0] = v.x; w[1] = v.y;
        } else {
            const uint4 v = *reinterpret_cast<const uint4 *>(p);
            w[0] = v.x; w[1] = v.y; w[2] = v.z;
            if constexpr (R == 16) w[3] = v.w;
        }
    } else if constexpr (PK == kP16Pair) {
        using C = P16Chunks<H>;
        const int8_t *p = prof + off;
#pragma unroll
        for (int q = 0; q < C::N4; ++q) {
            const uint4 v = *reinterpret_cast<const uint4 *>(p + g * 16 + (size_t)q * NL * 16);
            w[4 * q] = v.x; w[4 * q + 1] = v.y; w[4 * q + 2] = v.z; w[4 * q + 3] = v.w;
        }
#pragma unroll
        for (int q = 0; q < C::N2; ++q) {
            const uint2 v = *reinterpret_cast<const uint2 *>(p + g * 8 + (size_t)(C::N4 * 16 + q * 8) * NL);
            w[4 * C::N4 + 2 * q] = v.x; w[4 * C::N4 + 2 * q + 1] = v.y;
        }
        if constexpr (C::N1 == 1)
            w[H - 1] = *reinterpret_cast<const uint32_t *>(p + g * 4 + (size_t)(C::N4 * 16 + C::N2 * 8) * NL);
    } else if constexpr (R == 8 || R == 16) {
        const int8_t *p = prof + off + 2 * g * R;
#pragma unroll
        for (int q = 0; q < R / 8; ++q) {
            const uint4 v = *reinterpret_cast<const uint4 *>(p + 16 * q);
            w[4 * q] = v.x; w[4 * q + 1] = v.y; w[4 * q + 2] = v.z; w[4 * q + 3] = v.w;
        }
    } else {
        const int8_t *p = prof + off + 2 * g * R;
#pragma unroll
        for (int q = 0; q < R / 4; ++q) {
            const uint2 v = *reinterpret_cast<const uint2 *>(p + 8 * q);
            w[2 * q] = v.x; w[2 * q + 1] = v.y;
        }
    }
}

// Score pair S + open of packed row k.
template <int R, int PK>
__device__ __forceinline__ unsigned p16_score(const uint32_t (&cur)[p16_words(R, PK)],
                                              const uint32_t (&prev)[p16_words(R, PK)], int k) {
    if constexpr (PK == kP16Pair) {
        return cur[k];
    } else if constexpr (PK == kP16Int8) {
        const int kb = R / 2 + k;    // constants after unrolling: one prmt, both bytes sign-extended
        const unsigned x = k & 3, y = 4 + (kb & 3);
        return prmt_v(cur[k >> 2], prev[kb >> 2], x | ((8 | x) << 4) | (y << 8) | ((8 | y) << 12));
    } else {
        constexpr int H = R / 2;
        const int kb = H + k;        // bottom half's row k is lane row R/2 + k
        switch ((k & 1) * 2 + (kb & 1)) {   // constants after unrolling: one prmt
            case 0: return p16_halves<0, 0>(cur[k >> 1], prev[kb >> 1]);
            case 1: return p16_halves<0, 1>(cur[k >> 1], prev[kb >> 1]);
            case 2: return p16_halves<1, 0>(cur[k >> 1], prev[kb >> 1]);
            default: return p16_halves<1, 1>(cur[k >> 1], prev[kb >> 1]);
        }
    }
}

// Per-lane state: U = H - open and E of the lane's R/2 packed rows relative to the warp's base;
// fb the F of the row below each half's last row; flast the F of that last row; udiag0 the packed
// row above the two halves at their previous columns; w the bottom half's (U, F below) for the
// next lane; cmx the largest U of the chunk per half.
template <int R>
struct P16Lane {
    unsigned U[R / 2], E[R / 2];
    unsigned fb, flast, udiag0, w, cmx;
};

// -extend, -open and -infinity in both halves.
struct P16Consts { unsigned nge2, ngo2, neg2; };

// One step of one lane: column s - 2 lane (top half) and the one before (bottom half); top = lane 0's row
// above for this step, (H - open, F of the first row).
// LOCAL = false: no zero floor, and cmx is kept by the caller (the largest U only matters in the last row).
// EDGE: a half whose bits are set in hold keeps its state (its column lies outside the task).
template <int R, int PK, bool LOCAL = true, bool EDGE = false>
__device__ __forceinline__ void p16_step(P16Lane<R> &st, const uint32_t (&pw)[p16_words(R, PK)],
                                         const uint32_t (&pwp)[p16_words(R, PK)],
                                         unsigned top, bool lane0, const P16Consts &c, unsigned hold = 0)
{
    constexpr int H = R / 2;
    [[maybe_unused]] auto held = [&](unsigned now, unsigned before) { return EDGE ? (now & ~hold) | (before & hold) : now; };
    unsigned r = __shfl_up_sync(kFull, st.w, 1);
    r = lane0 ? top : r;
    // low half: the row above the top half (lane t-1's bottom half one step earlier); high half: this
    // lane's own top half one step earlier
    const unsigned uup = prmt_c<0x5410>(r, st.U[H - 1]);
    unsigned f = prmt_c<0x5432>(r, st.fb);
    unsigned udiag = st.udiag0;
    st.udiag0 = held(uup, udiag);
#pragma unroll
    for (int k = 0; k < H; ++k) {
        const unsigned sp = p16_score<R, PK>(pw, pwp, k);
        const unsigned uold = st.U[k];
        const unsigned e = __viaddmax_s16x2(st.E[k], c.nge2, uold);
        const unsigned x = LOCAL ? __viaddmax_s16x2_relu(udiag, sp, e)   // max(H(i-1,j-1) + S, E, 0)
                                 : __viaddmax_s16x2(udiag, sp, e);
        const unsigned xgo = __viaddmax_s16x2(x, c.ngo2, c.neg2);  // x - open
        const unsigned u = __viaddmax_s16x2(f, c.ngo2, xgo);       // H - open
        st.E[k] = held(e, st.E[k]);
        udiag = uold;
        st.U[k] = held(u, uold);
        if (k + 1 < H) f = __viaddmax_s16x2(f, c.nge2, xgo);       // F of the next row
        else st.fb = held(__viaddmax_s16x2(f, c.nge2, xgo), st.fb);   // F of the row below the half
    }
    st.flast = held(f, st.flast);
    st.w = prmt_c<0x7632>(st.U[H - 1], st.fb);
    if constexpr (LOCAL) {
#pragma unroll
        for (int k = 0; k + 1 < H; k += 2) st.cmx = __vimax3_s16x2(st.cmx, st.U[k], st.U[k + 1]);
        if constexpr (H % 2 == 1) st.cmx = __vmaxs2(st.cmx, st.U[H - 1]);
    }
}

// The halves of a lane whose columns j (top) and j - 1 (bottom) lie outside [lo, n).
__device__ __forceinline__ unsigned p16_hold(int j, int lo, int n) {
    return ((j >= lo && j < n) ? 0u : 0xffffu) | ((j - 1 >= lo && j - 1 < n) ? 0u : 0xffff0000u);
}

__device__ __forceinline__ int ld_relaxed(const int *p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Input warp of a packed fill block, ahead of the first compute warp: every column's profile offset into the
// offset ring (published in *res; it goes on past the last column with the padding residue) and the strip's top
// boundary row (H - open, F; absolute) into channel 0 (published in prod[0]).
template <int QS, int QB, int PK, bool LOCAL>
__device__ __forceinline__ void p16_input_warp(const FillTask &T, const FillLaunch &L, int strip, long long slot,
                                               int n, int n_ext, int go, int K, int Wa, int2 *ring0, int *poff,
                                               int pstride, int *prod, int *res, const int *cons, volatile int *s_abort,
                                               int lane, int alg, int ge)
{
    constexpr int kBatch = 64;                 // columns of either stream per turn
    const uint8_t *const b = T.b;
    const bool left = T.left != nullptr;
    const int2 *const src = strip == 0 ? T.top : T.bnd + (size_t)((strip - 1) % T.nslot) * n;
    const int *const pprev = L.prog + (slot - 1);
    const long long spin_limit = L.spin_limit;
    const int col0 = T.col0;
    int next = 0, rnext = 0, avail = strip == 0 ? n : 0;
    long long idle = 0;
    bool warm = true;                          // the first turn runs the boundary code with nothing to move (instruction cache)
    while (next < n || rnext < n_ext) {
        bool moved = false;
        if (next < n) {
            const int room = lds_acquire(&cons[0]) + QS;
            int target = min(n, min(next + kBatch, room));
            if (target > next) {
                if (avail < target) {
                    const int seen = ld_relaxed(pprev);
                    if (seen > avail) {
                        asm volatile("fence.acq_rel.gpu;" ::: "memory");   // the row up to `seen` is visible now
                        avail = seen;
                    }
                }
                target = max(next, min(target, avail));
            }
            target = max(target, next);
            if (target > next || warm) {
                const int c0 = next + lane, c1 = c0 + 32;
                // the matrix's top border: H(0, j) of the algorithm, F = -infinity
                int2 v0 = make_int2(LOCAL ? 0 : (int)top_border_h(alg, (long long)col0 + c0 + 1, go, ge), kNeg);
                int2 v1 = make_int2(LOCAL ? 0 : (int)top_border_h(alg, (long long)col0 + c1 + 1, go, ge), kNeg);
                if (src && c0 < target) v0 = __ldcg(src + c0);
                if (src && c1 < target) v1 = __ldcg(src + c1);
                if (c0 < target) ring0[c0 & (QS - 1)] = make_int2(v0.x - go, v0.y);
                if (c1 < target) ring0[c1 & (QS - 1)] = make_int2(v1.x - go, v1.y);
                __syncwarp();
                if (lane == 0) sts_release(&prod[0], target);
                moved = target > next;
                next = target;
                warm = false;
            }
        }
        // the offsets run ahead: in idle turns, and whenever they are less than two batches ahead
        if (rnext < n_ext && (!moved || rnext < next + 2 * kBatch)) {
            const int target = min(n_ext, min(rnext + kBatch, p16_offset_room(lds_acquire(&prod[Wa]))));
            if (target > rnext) {
                for (int col = rnext + lane; col < target; col += 32) {
                    const int c = col < n ? min((int)__ldg(b + col), K) : K;
                    if constexpr (PK == kP16Pair) {
                        const int cm = (col > 0 || left) && col <= n ? min((int)__ldg(b + col - 1), K) : K;
                        poff[col & (QB - 1)] = (c * (K + 1) + cm) * pstride;
                    } else {
                        poff[col & (QB - 1)] = c * pstride;
                    }
                }
                __syncwarp();
                if (lane == 0) sts_release(res, target);
                rnext = target;
                moved = true;
            }
        }
        if (moved) {
            idle = 0;
        } else {
            if (*s_abort) break;
            if (++idle > spin_limit) {
                if (lane == 0) atomicCAS(L.err, 0, kErrTimeout);
                *s_abort = 1;
                break;
            }
            __nanosleep(kP16IdleNs);
        }
    }
}

// Output warp: the strip's bottom row from the last active warp's channel to global memory as
// (H, F), absolute; publishes the stored column count with a release store.
__device__ __forceinline__ void p16_output_warp(const FillTask &T, const FillLaunch &L, int strip, long long slot,
                                                int n, int go, int SH, int Wa, const uint2 *ringW, const int *baseW,
                                                const int *prod, int *cons, volatile int *s_abort, int lane)
{
    int out_next = 0;
    long long idle = 0;
    const bool ck = T.ckpt_every > 0 && ((strip + 1) % T.ckpt_every) == 0 &&
                    (long long)(strip + 1) * SH <= (long long)T.rows;
    int2 *const cdst = ck ? T.ckpt + (size_t)((strip + 1) / T.ckpt_every - 1) * n : nullptr;
    const bool store = strip + 1 < T.nstrips;
    int2 *const dst = store ? T.bnd + (size_t)(strip % T.nslot) * n : nullptr;
    int *const prog = L.prog + slot;
    const long long spin_limit = L.spin_limit;
    bool warm = true;                          // the first turn runs with nothing to move (instruction cache)
    while (out_next < n) {
        const int avail_out = min(lds_acquire(&prod[Wa]), out_next + 64);
        if (avail_out > out_next || warm) {
            if (store || ck) {
                const int c0 = out_next + lane, c1 = c0 + 32;
                const bool p0 = c0 < avail_out, p1 = c1 < avail_out;
                const int l0 = c0 + kP16Lag, l1 = c1 + kP16Lag;
                const uint2 v0 = ringW[l0 & (kP16RS - 1)], v1 = ringW[l1 & (kP16RS - 1)];
                const int B0 = baseW[(l0 / kP16CH) & (kP16RS / kP16CH - 1)], B1 = baseW[(l1 / kP16CH) & (kP16RS / kP16CH - 1)];
                const int2 o0 = make_int2(p16_lo(v0.x) + B0 + go, p16_hi(v0.y) + B0);
                const int2 o1 = make_int2(p16_lo(v1.x) + B1 + go, p16_hi(v1.y) + B1);
                if (store && p0) __stcg(dst + c0, o0);
                if (store && p1) __stcg(dst + c1, o1);
                if (ck && p0) __stcg(cdst + c0, o0);
                if (ck && p1) __stcg(cdst + c1, o1);
            }
            warm = false;
            __syncwarp();
            if (lane == 0) {
                if (store) st_release(prog, avail_out);
                sts_release(&cons[Wa], avail_out);
            }
            out_next = avail_out;
            idle = 0;
        } else {
            if (*s_abort) break;
            if (++idle > spin_limit) {
                if (lane == 0) atomicCAS(L.err, 0, kErrTimeout);
                *s_abort = 1;
                break;
            }
            __nanosleep(kP16IdleNs);
        }
    }
}

// The warp waits until *a >= wa, *b >= wb and *c >= wc (bounded); false on timeout or when the block is aborting.
__device__ __forceinline__ bool p16_wait3(const int *a, int wa, const int *b, int wb, const int *c, int wc,
                                          const volatile int *abort_flag, long long limit, int *err) {
    for (long long it = 0;; ++it) {
        const int va = *(const volatile int *)a, vb = *(const volatile int *)b, vc = *(const volatile int *)c;
        if (va >= wa && vb >= wb && vc >= wc) break;
        if (*abort_flag) return false;
        if (it > limit) { atomicCAS(err, 0, kErrTimeout); return false; }
        if (it > 1) __nanosleep(64);
    }
    __threadfence_block();
    return true;
}

// The first half-lane (2 lane + half) whose chunk maximum is v.
__device__ __forceinline__ int p16_first_pos(unsigned cmx, int v) {
    const unsigned b0 = __ballot_sync(kFull, p16_lo(cmx) == v), b1 = __ballot_sync(kFull, p16_hi(cmx) == v);
    const int p0 = b0 ? 2 * (__ffs(b0) - 1) : 64, p1 = b1 ? 2 * (__ffs(b1) - 1) + 1 : 64;
    return min(p0, p1);
}

// Snapshot of a warp's state at a chunk's start, for finding the end cell's row and column later.
template <int R>
struct P16Snap {
    uint4 st[p16_snap_words(R) / 4][32];   // U, E, fb, udiag0 of every lane
    unsigned top[kP16CH];                  // lane 0's rows above
    int s0, B;
};

// The first cell in row-major order, among the valid cells of half-lane pos of the chunk in snapshot S,
// whose H - open equals u: (row of the half, column), or (R, 0).  Valid: rows [row_lo, row_hi) of the half, real columns.
template <int R, int PK, int NL, bool LOCAL>
__device__ __noinline__ int2 p16_locate(const P16Snap<R> &S, const int8_t *prof, int g, int pstride, const FillTask &T,
                                        int n, int K, int go, int ge, int pos, int u, int row_lo, int row_hi)
{
    constexpr int H = R / 2;
    const int lane = threadIdx.x & 31;
    unsigned q[p16_snap_words(R)];
#pragma unroll
    for (int k = 0; k < p16_snap_words(R) / 4; ++k) {
        const uint4 v = S.st[k][lane];
        q[4 * k] = v.x; q[4 * k + 1] = v.y; q[4 * k + 2] = v.z; q[4 * k + 3] = v.w;
    }
    P16Lane<R> st;
#pragma unroll
    for (int k = 0; k < H; ++k) { st.U[k] = q[k]; st.E[k] = q[H + k]; }
    st.fb = q[2 * H]; st.udiag0 = q[2 * H + 1];
    st.flast = 0;
    st.w = prmt_c<0x7632>(st.U[H - 1], st.fb);
    st.cmx = 0x80008000u;
    const P16Consts c{p16_pack(-ge, -ge), p16_pack(-go, -go), p16_pack(kNeg16p, kNeg16p)};
    const int want = u - S.B;
    const bool mine = lane == (pos >> 1);
    const int h = pos & 1;
    int row = R, col = 0;
    const uint8_t *const b = T.b;
    const int first = T.left ? -(1 << 30) : 0;
    auto code = [&](int j) { return (j >= first && j < n) ? min((int)__ldg(b + j), K) : K; };
#pragma unroll 1
    for (int k0 = 0; k0 < kP16CH; k0 += 4) {
        int cc[5];                                         // residues of columns j - 1 .. j + 3, loaded together
#pragma unroll
        for (int x = 0; x < 5; ++x) cc[x] = code(S.s0 + k0 + x - 1 - 2 * lane);
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int j = S.s0 + k0 + x - 2 * lane;
            uint32_t pw[p16_words(R, PK)], pwp[p16_words(R, PK)];
            if constexpr (PK == kP16Pair) {
                p16_load<R, PK, NL>(prof, g, (cc[x + 1] * (K + 1) + cc[x]) * pstride, pw);
#pragma unroll
                for (int y = 0; y < p16_words(R, PK); ++y) pwp[y] = 0;
            } else {
                p16_load<R, PK, NL>(prof, g, cc[x + 1] * pstride, pw);
                p16_load<R, PK, NL>(prof, g, cc[x] * pstride, pwp);
            }
            p16_step<R, PK, LOCAL, !LOCAL>(st, pw, pwp, S.top[k0 + x], lane == 0, c, LOCAL ? 0u : p16_hold(j, first, n));
            const int jj = j - h;
            if (mine && jj >= 0 && jj < n) {
#pragma unroll
                for (int y = H - 1; y >= 0; --y)
                    if (y < row && y >= row_lo && y < row_hi && (h ? p16_hi(st.U[y]) : p16_lo(st.U[y])) == want) { row = y; col = jj; }
            }
        }
    }
    row = __shfl_sync(kFull, row, pos >> 1);
    col = __shfl_sync(kFull, col, pos >> 1);
    return make_int2(row, col);
}

// A task that starts right of a checkpoint column written by this fill (the
// two-positions staircase of the checkpoint mode, FillTask::left_split):
// lane l's top half holds its rows at column -1 - 2l and its bottom half at
// -2 - 2l (task columns), which is exactly the wavefront's state after step
// -1.  The lane takes that state (relative to a base taken from lane 0) and the
// sweep goes on from step 0; its first steps recompute real columns left of
// the task from real residues (the offset ring's slots left of column 0).
template <int R, bool LOCAL>
__device__ __forceinline__ void p16_enter_staircase(const FillTask &T, P16Lane<R> &st, int &B, int grow, int lane, int go,
                                                    int ge) {
    constexpr int H = R / 2;
    int vU[R], vE[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        int2 v = make_int2(-go, kNeg);
        if (grow + r < T.rows) v = __ldcg(T.left + grow + r);
        vU[r] = v.x;
        vE[r] = v.y;
    }
    const bool in = grow < T.rows;
    const int2 at = in ? __ldcg(T.left_aux + grow / H) : make_int2(-go, kNeg);       // top half
    const int2 ab = in ? __ldcg(T.left_aux + grow / H + 1) : make_int2(-go, kNeg);   // bottom half
    B = __shfl_sync(kFull, vU[0], 0) - kP16Center;
    if (LOCAL) B = max(B, 0);
    auto rel = [&](int v) { return max(min(v - B, 32767), kNeg16p); };
#pragma unroll
    for (int k = 0; k < H; ++k) {
        st.U[k] = p16_pack(rel(vU[k]), rel(vU[H + k]));
        st.E[k] = p16_pack(rel(vE[k]), rel(vE[H + k]));
    }
    st.udiag0 = p16_pack(rel(at.x), rel(ab.x));
    st.flast = p16_pack(rel(at.y), rel(ab.y));
    st.fb = __viaddmax_s16x2(st.flast, p16_pack(-ge, -ge), st.U[H - 1]);
    st.w = prmt_c<0x7632>(st.U[H - 1], st.fb);
}


// A compile-time integer as an argument.
template <int V> struct P16Int { static constexpr int v = V; };

// Shared memory of a block ahead of its query profile.
template <int R, int W>
struct P16Shared {
    P16Snap<R> snap[W][3];
    int poff[kQB];                         // profile offset per column
    int2 ring0[kP16QS];                    // (H - open, F), absolute: the strip's boundary row
    uint2 ring[W][kP16RS];                 // channel w + 1: after step s of warp w, at slot s, (w, F of the bottom row)
    int base[W][kP16RS / kP16CH];          // base of warp w per chunk
    int4 cand[W];
    long long tk;
    int prod[W + 1];                       // columns available in channel k
    int cons[W + 1];                       // columns consumed from channel k
    int res;                               // columns with a profile offset
    int task, strip;
    int abort;
};

template <int R, int W>
constexpr size_t p16_shared_bytes() { return (sizeof(P16Shared<R, W>) + 15) / 16 * 16; }

// LEFT: the tasks may start right of a checkpoint column written by this fill
// (p16_enter_staircase; the coarse-tile refills of a two-level reconstruction).
// A separate instantiation, so that the others compile exactly without it.
// LOCAL = false: the global, semi-global and overlap algorithms (DevScoring::alg).
// MINB: blocks an SM to compile for.
template <int R, int W, int MODE, int PK, bool LEFT = false, bool LOCAL = true, int MINB = 1>
__global__ void __launch_bounds__((W + 2) * 32, MINB)
wavefront16_kernel(const FillLaunch L)
{
    static_assert(R % 2 == 0 && R >= 4, "two halves");
    static_assert(PK == kP16Pair || R == 8 || R == 12 || R == 16, "int16 and int8 profile loads");
    constexpr int NWD = p16_words(R, PK);
    static_assert(MODE == kModeScore || MODE == kModeScoreCk, "score modes only");
    constexpr int H = R / 2;
    constexpr int HC = W * 32 * R;
    constexpr int NL = W * 32;
    constexpr int CH = kP16CH, QS = kP16QS, RS = kP16RS, QB = kQB, LAG = kP16Lag;
    static_assert(QS >= 2 * 64 + 2 * CH && RS >= 2 * CH + 2 * kP16Pos, "ring too small");
    static_assert(QB >= W * (kP16Pos + CH) + kP16Back + 128, "the first warp's offsets must fit beside those the last warp still reads");
    constexpr int UNR = kP16Unroll;
    static_assert(CH % UNR == 0 && UNR % 4 == 0, "chunks are whole unrolled groups of four steps");
    static_assert(CH == 32, "one boundary entry a lane");

    extern __shared__ __align__(16) int8_t p16_smem[];   // P16Shared, then p16_profile_bytes
    P16Shared<R, W> &S = *reinterpret_cast<P16Shared<R, W> *>(p16_smem);
    int8_t *const prof = p16_smem + p16_shared_bytes<R, W>();
    int2 *const ring0 = S.ring0;
    uint2 (*const ring)[kP16RS] = S.ring;
    int (*const s_base)[kP16RS / kP16CH] = S.base;
    int *const s_poff = S.poff, *const prod = S.prod, *const cons = S.cons;
    P16Snap<R> (*const s_snap)[3] = S.snap;
    int4 *const s_cand = S.cand;
    volatile int *const s_abort = &S.abort;

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;

    for (bool first = true;; first = false) {
        if (threadIdx.x == 0) {
            claim_strip(L, &S.tk, &S.task, &S.strip);
            *s_abort = 0;
        }
        if (threadIdx.x <= W) { prod[threadIdx.x] = 0; cons[threadIdx.x] = 0; }
        if (threadIdx.x == 0) S.res = 0;
        __syncthreads();
        const long long tk = S.tk;
        if (tk >= L.total) return;
        const FillTask &T = L.tasks[S.task];
        const DevScoring &SC = L.scorings[T.scoring];
        const int K = SC.K, go = SC.go, ge = SC.ge;
        const int strip = S.strip;
        const long long slot = T.ticket0 + strip;        // progress and candidate of (task, strip)
        const int SW = (T.strip_warps > 0 && T.strip_warps < W) ? T.strip_warps : W;
        const int SH = SW * 32 * R;
        const int rbase = strip * SH;
        const int n = T.ncols;
        const int Wa = min(SW, (T.rows - rbase + 32 * R - 1) / (32 * R));
        const int n_ext = (n + LAG + CH - 1) / CH * CH + 2;

        const int pstride = PK == kP16Pair ? H * NL * 4 : (PK == kP16Int8 ? NL * p16_slot8(R) : 2 * HC);   // bytes per profile entry
        // query profile of the strip's rows, S(a_r, c) + open, padding rows and columns at kPadScore: a thread takes a
        // row (pair profile: the packed row of a lane) and runs over the residues, so that a row's residue is read
        // once and no index is divided (464 x 503 protein: the fill 69 -> 55 us)
        if constexpr (PK == kP16Pair) {
            uint32_t *pw32 = reinterpret_cast<uint32_t *>(prof);
            for (int idx = threadIdx.x; idx < SW * 32 * H; idx += blockDim.x) {
                const int k = idx % H, pg = idx / H;
                const int rt = rbase + pg * R + k, rb = rt + H;
                const int8_t *mt = rt < T.rows ? SC.mat + min((int)T.a[rt], K - 1) * K : nullptr;
                const int8_t *mb = rb < T.rows ? SC.mat + min((int)T.a[rb], K - 1) * K : nullptr;
                uint32_t *dst = pw32 + p16_pair_word<H>(k, pg, NL);
                for (int ct = 0; ct <= K; ++ct) {
                    const int vt = mt && ct < K ? mt[ct] + go : kPadScore;
                    for (int cb = 0; cb <= K; ++cb)
                        dst[(ct * (K + 1) + cb) * (NL * H)] = p16_pack(vt, mb && cb < K ? mb[cb] + go : kPadScore);
                }
            }
        } else if constexpr (PK == kP16Int8) {
            for (int lr = threadIdx.x; lr < SH; lr += blockDim.x) {
                const int8_t *m = rbase + lr < T.rows ? SC.mat + min((int)T.a[rbase + lr], K - 1) * K : nullptr;
                int8_t *dst = prof + lr / R * p16_slot8(R) + lr % R;
                for (int c = 0; c <= K; ++c) dst[c * (NL * p16_slot8(R))] = (int8_t)(m && c < K ? m[c] + go : kPadScore);
            }
        } else {
            int16_t *p16 = reinterpret_cast<int16_t *>(prof);
            for (int lr = threadIdx.x; lr < SH; lr += blockDim.x) {
                const int8_t *m = rbase + lr < T.rows ? SC.mat + min((int)T.a[rbase + lr], K - 1) * K : nullptr;
                for (int c = 0; c <= K; ++c) p16[c * HC + lr] = (int16_t)(m && c < K ? m[c] + go : kPadScore);
            }
        }
        // the offset ring starts as padding (the warm-up chunk below reads columns down to -96); its last kP16Pos
        // slots hold the columns left of the task: padding at the matrix border, real residues for a task entered from
        // a checkpoint column.  The input warp stays kP16Back slots short of a full ring until the last warp has published
        // a column, i.e. left all of these behind
        if (first) {
            for (int k = threadIdx.x; k < QB; k += blockDim.x) s_poff[k] = (PK == kP16Pair ? K * (K + 1) + K : K) * pstride;
            __syncthreads();
        }
        if (threadIdx.x < kP16Pos) {
            const int j = (int)threadIdx.x - kP16Pos;                       // column -64 .. -1
            const bool real = LEFT && T.left;
            const int cj = real ? min((int)T.b[j], K) : K;
            const int cjm = real ? min((int)T.b[j - 1], K) : K;
            s_poff[QB - kP16Pos + threadIdx.x] = PK == kP16Pair ? (cj * (K + 1) + cjm) * pstride : cj * pstride;
        }
        __syncthreads();

        if (warp == W) {
            p16_input_warp<QS, QB, PK, LOCAL>(T, L, strip, slot, n, n_ext, go, K, Wa, ring0, s_poff, pstride, prod, &S.res, cons,
                                            s_abort, lane, SC.alg, ge);
        } else if (warp == W + 1) {
            p16_output_warp(T, L, strip, slot, n, go, SH, Wa, ring[Wa - 1], s_base[Wa - 1], prod, cons, s_abort,
                                lane);
        } else if (warp >= Wa) {
            if (lane == 0) s_cand[warp] = make_int4(LOCAL ? 0 : kNoScore, 0x7fffffff, 0x7fffffff, 0);
        } else {
            // ================= compute warp =================
            const int g = warp * 32 + lane;
            const int grow = rbase + g * R;
            const bool lane0 = lane == 0;
            const P16Consts cst{p16_pack(-ge, -ge), p16_pack(-go, -go), p16_pack(kNeg16p, kNeg16p)};
            P16Lane<R> st;
            int B = 0;
#pragma unroll
            for (int k = 0; k < H; ++k) { st.U[k] = cst.ngo2; st.E[k] = cst.neg2; }
            st.fb = cst.ngo2; st.flast = cst.neg2; st.udiag0 = cst.ngo2; st.w = cst.ngo2;   // matrix border: H = 0
            if constexpr (LEFT)
                if (T.left) p16_enter_staircase<R, LOCAL>(T, st, B, grow, lane, go, ge);
            // the other algorithms: the matrix's left border H(i, 0) as state, held until a half's column 0; the task's
            // last row (where it is an end row at every column: semi-global, overlap) as a mask over the packed rows
            [[maybe_unused]] unsigned tmask[LOCAL ? 1 : H];
            [[maybe_unused]] int rlast = -1;               // the lane's row that is the task's last one
            [[maybe_unused]] bool track = false;           // this warp holds the last row and it is an end row
            if constexpr (!LOCAL) {
                if (!(LEFT && T.left)) {
                    auto border = [&](long long i) { return (int)left_border_h(SC.alg, i, go, ge) - go; };
                    const long long i0 = (long long)T.row0 + grow;
                    B = border((long long)T.row0 + rbase + warp * 32 * R + 1) - kP16Center;
#pragma unroll
                    for (int k = 0; k < H; ++k)
                        st.U[k] = p16_pack(max(border(i0 + k + 1) - B, kNeg16p), max(border(i0 + H + k + 1) - B, kNeg16p));
                    st.udiag0 = p16_pack(max(border(i0) - B, kNeg16p), max(border(i0 + H) - B, kNeg16p));
                    st.fb = cst.neg2;
                    st.w = prmt_c<0x7632>(st.U[H - 1], st.fb);
                }
                const int rl = T.rows - 1 - grow;
                rlast = rl >= 0 && rl < R ? rl : -1;
#pragma unroll
                for (int k = 0; k < H; ++k) tmask[k] = rl == k ? 0xffffu : (rl == H + k ? 0xffff0000u : 0u);
                track = (SC.alg == kAlgSemiGlobal || SC.alg == kAlgOverlap) && __any_sync(kFull, rlast >= 0);
            }
            // the warp's best: H - open, half-lane (2 lane + half), and where: snapshot, or row and column once located
            int bu = LOCAL ? 1 - go : -(1 << 30), brow = R, bcol = 0, bcb = 0;
            int pa = 0, pb = 0, npend = 0;      // snapshots that hold the best (the second: the same half-lane again)

            unsigned bcm = 0x80008000u;
            bool held = false;
            int cur = 0;                        // snapshot buffer of the running chunk; the other holds the best's chunk
            int next_ck = (MODE == kModeScoreCk && T.colck && T.colck_every > 0) ? T.colck_every - 1 : 0x7fffffff;
            uint2 *rout = ring[warp];
            // rows and columns of the best in the pending snapshots: the smallest row, then the earlier chunk's column
            auto resolve = [&](int pos) {
                const int nr = T.rows - (rbase + (warp * 32 + (pos >> 1)) * R + (pos & 1) * H);
                for (int q = 0; q < npend; ++q) {
                    const int2 c = p16_locate<R, PK, NL, LOCAL>(s_snap[warp][q ? pb : pa], prof, g, pstride, T, n, K, go, ge, pos,
                                                                bu, LOCAL ? 0 : nr - 1, nr);
                    if (c.x < brow) { brow = c.x; bcol = c.y; }
                }
            };
            const long long spin_limit = L.spin_limit;
            int *const err = L.err;
            uint32_t pw[NWD], pwp[NWD];
            int2 off;                           // profile offsets of the next two steps to load
            bool ok = true;
            // the block's first strip runs one chunk left of the task, which keeps the border state: it brings the
            // loop into the instruction cache while the strip above has not produced its first columns yet
            const int sbeg = first && !(LEFT && T.left) ? -CH : 0;
            for (int s0 = sbeg; s0 < n + LAG; s0 += CH) {
                // the chunk's rows above, the profile offsets one step ahead, and room in the ring below
                const int ring_hi = s0 + CH - LAG, out_hi = min(n, ring_hi);
                if (!p16_wait3(&prod[warp], min(n, s0 + CH), &S.res, s0 + CH + 2, &cons[warp + 1], ring_hi - RS, s_abort,
                               spin_limit, err)) {
                    *s_abort = 1;
                    ok = false;
                    break;
                }
                if (s0 == sbeg) {
                    if constexpr (PK == kP16Pair) {
#pragma unroll
                        for (int q = 0; q < NWD; ++q) pwp[q] = 0;
                    } else {
                        p16_load<R, PK, NL>(prof, g, s_poff[(sbeg - 1 - 2 * lane) & (QB - 1)], pwp);
                    }
                    off = *reinterpret_cast<const int2 *>(&s_poff[(sbeg - 2 * lane) & (QB - 1)]);
                    p16_load<R, PK, NL>(prof, g, off.x, pw);
                }
                // lane 0's rows above for the chunk's steps (one entry a lane); -infinity at and past n
                const int tcol = s0 + lane;
                const bool treal = tcol >= 0 && tcol < n;
                int2 tv = make_int2(0, 0);
                int tB = 0;
                if (treal) {
                    if (warp == 0) {
                        tv = ring0[tcol & (QS - 1)];
                    } else {
                        tv.x = (int)ring[warp - 1][(tcol + LAG) & (RS - 1)].x;
                        tB = s_base[warp - 1][((tcol + LAG) / CH) & (RS / CH - 1)];
                    }
                }
                {   // the warp's base follows lane 0's first row
                    const int ref = p16_lo(__shfl_sync(kFull, st.U[0], 0));
                    if (ref > kP16Center + kP16Slack || ((!LOCAL || B > 0) && ref < kP16Center - kP16Slack)) {
                        const int Bn = LOCAL ? max(0, ref + B - kP16Center) : ref + B - kP16Center;
                        const unsigned d2 = p16_pack(B - Bn, B - Bn);
#pragma unroll
                        for (int k = 0; k < H; ++k) {
                            st.U[k] = __viaddmax_s16x2(st.U[k], d2, cst.neg2);
                            st.E[k] = __viaddmax_s16x2(st.E[k], d2, cst.neg2);
                        }
                        st.fb = __viaddmax_s16x2(st.fb, d2, cst.neg2);
                        st.flast = __viaddmax_s16x2(st.flast, d2, cst.neg2);
                        st.udiag0 = __viaddmax_s16x2(st.udiag0, d2, cst.neg2);
                        st.w = prmt_c<0x7632>(st.U[H - 1], st.fb);
                        B = Bn;
                    }
                }
                P16Snap<R> &snap = s_snap[warp][cur];
                {
                    unsigned q[p16_snap_words(R)];
#pragma unroll
                    for (int k = 0; k < H; ++k) { q[k] = st.U[k]; q[H + k] = st.E[k]; }
                    q[2 * H] = st.fb; q[2 * H + 1] = st.udiag0;
#pragma unroll
                    for (int k = 2 * H + 2; k < p16_snap_words(R); ++k) q[k] = 0;
#pragma unroll
                    for (int k = 0; k < p16_snap_words(R) / 4; ++k)
                        snap.st[k][lane] = make_uint4(q[4 * k], q[4 * k + 1], q[4 * k + 2], q[4 * k + 3]);
                    if (lane0) {
                        s_base[warp][(s0 / CH) & (RS / CH - 1)] = B;
                        snap.s0 = s0; snap.B = B;
                    }
                    unsigned t = tcol < 0 ? cst.ngo2 : cst.neg2;
                    if (treal) {
                        if (warp == 0) t = p16_pack(max(tv.x - B, kNeg16p), max(max(tv.y - ge, tv.x) - B, kNeg16p));
                        else t = __viaddmax_s16x2((unsigned)tv.x, p16_pack(tB - B, tB - B), cst.neg2);
                    }
                    snap.top[lane] = t;
                    __syncwarp();
                }
                if constexpr (MODE == kModeScoreCk) {
                    // the checkpoint column before this chunk, out of the snapshot by a small loop: unrolled from the
                    // registers at the chunk's end it slowed every step of the long bodies down (26 rows a lane,
                    // 505,856 x 500,000: 62.8 against the score fill's 58.5 ms, 62.0 with the store compiled in but
                    // never reached; this way 59.4).  Bodies of 8 to 16 rows: the same either way
                    if (s0 - 1 == next_ck && next_ck < n) {   // the same for every lane
                        const long long kk = (next_ck + 1) / T.colck_every - 1;
                        int2 *cc = T.colck + kk * T.colck_ld + (T.row0 + grow);
                        const unsigned *q = reinterpret_cast<const unsigned *>(&snap.st[0][lane]);
                        auto word = [&](int k) { return q[(k >> 2) * 128 + (k & 3)]; };
#pragma unroll 1
                        for (int k = 0; k < H; ++k) {
                            const unsigned u = word(k), e = word(H + k);
                            cc[k] = make_int2(p16_lo(u) + B, p16_lo(e) + B);
                            cc[H + k] = make_int2(p16_hi(u) + B, p16_hi(e) + B);
                        }
                        int2 *ca = T.colck_aux + kk * (T.colck_ld / H) + (T.row0 + grow) / H;
                        ca[0] = make_int2(p16_lo(st.udiag0) + B, p16_lo(st.flast) + B);
                        ca[1] = make_int2(p16_hi(st.udiag0) + B, p16_hi(st.flast) + B);
                        next_ck += T.colck_every;
                    }
                }
                st.cmx = 0x80008000u;
                uint2 *rc = rout + (s0 & (RS - 1));
                // the chunk's steps; NS: steps an unrolled body, EDGE: halves outside the task hold (the other algorithms)
                auto sweep = [&](auto ns, auto edge) {
                    constexpr int NS = decltype(ns)::v;
                    constexpr bool EDGE = decltype(edge)::v != 0;
                    [[maybe_unused]] const int lo = LEFT && T.left ? -(1 << 30) : 0;
                    auto step = [&](const uint32_t (&w)[NWD], const uint32_t (&wp)[NWD], unsigned top, int s) {
                        p16_step<R, PK, LOCAL, EDGE>(st, w, wp, top, lane0, cst, EDGE ? p16_hold(s - 2 * lane, lo, n) : 0u);
                        if (lane == 31) rc[s - s0] = make_uint2(st.w, st.flast);
                        if constexpr (!LOCAL) {
                            if (track) {                   // (one warp of the pair)
                                unsigned v = 0;
#pragma unroll
                                for (int k = 0; k < H; ++k) v |= st.U[k] & tmask[k];
                                st.cmx = __vmaxs2(st.cmx, v);
                            }
                        }
                    };
#pragma unroll 1
                    for (int gs = 0; gs < CH; gs += NS) {
#pragma unroll
                        for (int k4 = 0; k4 < NS; k4 += 4) {
                            const uint4 tops = *reinterpret_cast<const uint4 *>(&snap.top[gs + k4]);
#pragma unroll
                            for (int k2 = 0; k2 < 4; k2 += 2) {
                                const int s = s0 + gs + k4 + k2;
                                // offsets of steps s + 2, s + 3 (slots an even distance apart from lane to lane)
                                const int2 offn = *reinterpret_cast<const int2 *>(&s_poff[(s + 2 - 2 * lane) & (QB - 1)]);
                                uint32_t pwn[NWD];
                                p16_load<R, PK, NL>(prof, g, off.y, pwn);
                                step(pw, pwp, k2 == 0 ? tops.x : tops.z, s);
                                p16_load<R, PK, NL>(prof, g, offn.x, PK == kP16Pair ? pw : pwp);
                                if constexpr (PK == kP16Pair) {
                                    step(pwn, pwp, k2 == 0 ? tops.y : tops.w, s + 1);
                                } else {
                                    uint32_t t2[NWD];
#pragma unroll
                                    for (int q = 0; q < NWD; ++q) t2[q] = pwp[q];      // words of step s + 2
                                    step(pwn, pw, k2 == 0 ? tops.y : tops.w, s + 1);
#pragma unroll
                                    for (int q = 0; q < NWD; ++q) { pwp[q] = pwn[q]; pw[q] = t2[q]; }
                                }
                                off = offn;
                            }
                        }
                    }
                };
                if constexpr (LOCAL) {
                    sweep(P16Int<UNR>{}, P16Int<0>{});     // (a lane past the task's columns steps over padding)
                } else {
                    if ((s0 >= kP16Pos || (LEFT && T.left)) && s0 + CH <= n) sweep(P16Int<UNR>{}, P16Int<0>{});
                    else sweep(P16Int<4>{}, P16Int<1>{});
                }
                if constexpr (!LOCAL) {
                    if (track) {                           // the last row's best of the chunk; the first column that holds it wins
                        const unsigned who = __ballot_sync(kFull, rlast >= 0);
                        const int v = __shfl_sync(kFull, rlast >= H ? p16_hi(st.cmx) : p16_lo(st.cmx), __ffs(who) - 1) + B;
                        if (v > bu) {
                            bu = v; held = true; brow = R;
                            pa = cur; npend = 1;
                            cur = (cur + 1) % 3;
                        }
                    }
                } else {   // a best cell in this chunk?
                    const int lo = p16_lo(st.cmx), hi = p16_hi(st.cmx);
                    const int thr = min(bu - B, 32767);
                    if (__any_sync(kFull, max(lo, hi) >= thr)) {
                        const int wm = __reduce_max_sync(kFull, max(lo, hi)) + B;
                        bool take = wm > bu || !held;          // a larger score
                        if (!take) {
                            // the same score again: the earlier half-lane holds the earlier rows; within one half-lane the
                            // rows decide, which are found later
                            const int bpos = p16_first_pos(bcm, bu - bcb), pos = p16_first_pos(st.cmx, bu - B);
                            take = pos < bpos;
                            if (pos == bpos && brow != 0) {
                                if (npend == 2) {
                                    resolve(bpos);
                                    npend = 0;
                                }
                                if (brow != 0) {
                                    if (npend++ == 0) pa = cur; else pb = cur;
                                    cur = npend == 1 ? (pa + 1) % 3 : 3 - pa - pb;
                                }
                            }
                        }
                        if (take) {
                            bu = wm; held = true; brow = R; bcm = st.cmx; bcb = B;
                            pa = cur; npend = 1;
                            cur = (cur + 1) % 3;
                        }
                    }
                }
                __syncwarp();
                if (lane == 0) {
                    __threadfence_block();
                    *(volatile int *)&cons[warp] = s0 + CH;
                    if (out_hi > 0) *(volatile int *)&prod[warp + 1] = out_hi;
                }
            }
            int cs = LOCAL ? 0 : kNoScore, cj = 0x7fffffff, ci = 0x7fffffff;
            if constexpr (LOCAL) {
                if (ok && held) {
                    const int bpos = p16_first_pos(bcm, bu - bcb);
                    resolve(bpos);
                    if (brow < H) {
                        cs = bu + go; cj = bcol + 1;
                        ci = T.row0 + rbase + (warp * 32 + (bpos >> 1)) * R + (bpos & 1) * H + brow + 1;
                    }
                }
            } else {
                if (ok && held) {                          // the best of the last row (semi-global, overlap)
                    const int l = __ffs(__ballot_sync(kFull, rlast >= 0)) - 1, r = __shfl_sync(kFull, rlast, l);
                    resolve(2 * l + (r >= H ? 1 : 0));
                    if (brow < H) { cs = bu + go; cj = bcol + 1; ci = T.row0 + T.rows; }
                }
                // the last column: every row for the overlap algorithm, the last row for the global one
                if (ok && n > 0 && (SC.alg == kAlgOverlap || SC.alg == kAlgGlobal)) {
#pragma unroll
                    for (int k = 0; k < R; ++k) {
                        const int sc = (k < H ? p16_lo(st.U[k % H]) : p16_hi(st.U[k % H])) + B + go;
                        const int ii = T.row0 + grow + k + 1;
                        const bool end = SC.alg == kAlgOverlap ? grow + k < T.rows : k == rlast;
                        if (end && cand_better(sc, n, ii, cs, cj, ci)) { cs = sc; cj = n; ci = ii; }
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const int os = __shfl_xor_sync(kFull, cs, o);
                    const int oj = __shfl_xor_sync(kFull, cj, o);
                    const int oi = __shfl_xor_sync(kFull, ci, o);
                    if (cand_better(os, oj, oi, cs, cj, ci)) { cs = os; cj = oj; ci = oi; }
                }
            }
            if (lane == 0) s_cand[warp] = make_int4(cs, ci, cj, 0);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            int4 b = s_cand[0];
            for (int w = 1; w < W; ++w) {
                const int4 o = s_cand[w];
                if (cand_better(o.x, o.z, o.y, b.x, b.z, b.y)) b = o;
            }
            b.w = LOCAL ? (b.x > 0 ? 1 : 0) : (b.x != kNoScore ? 1 : 0);
            L.cand[slot] = b;
        }
        __syncthreads();
    }
}

}  // namespace swgb
