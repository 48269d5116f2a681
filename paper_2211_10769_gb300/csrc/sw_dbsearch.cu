// sw_dbsearch.cu -- database search (paper Section 2.1, one-to-many,
// inter-task): device-resident database, packed 16-bit search with exact
// 32-bit rescoring of saturating subjects, top-k hits.
#include "sw.h"
#include "sw_ctx.h"
#include "db_launch.cuh"
#include "wavefront.cuh"
#include "aux_kernels.cuh"

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <numeric>
#include <vector>

using namespace swgb;


struct sw_db {
    int device = 0;
    int64_t nseq = 0;
    int32_t npairs = 0;
    int32_t maxlen = 0;
    int32_t max_code = -1;
    int64_t pcols = 0;                  // columns of all pairs
    std::vector<int64_t> off;           // host copy of the offsets
    std::vector<int32_t> hpairs;        // host copy of the length-sorted pairs
    DevBuf res, doff, pairs, pres, poff;   // pres / poff: interleaved residues of every pair
};

namespace {

static __global__ void max_code_kernel(const uint8_t *s, long long len, int *out) {
    int mx = 0;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < len; k += stride)
        mx = max(mx, (int)s[k]);
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(kFull, mx, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, mx);
}

// Tile shapes of the packed search: rows a lane, warps a block and lanes a
// wavefront (16: two wavefronts a warp).  A query is padded to whole passes of
// G R rows.  A lane's fixed per-step work (two shuffles, lane 0's row above,
// the next residues) is shared by its R rows, so a large database wants the most rows a
// lane whose passes the query fills: 144 residues take one pass at R = 9, 464 one at
// R = 29, 1,000 two at R = 32.  32 lanes a wavefront (1,000: one pass of 32 x 32
// rows, 5,690 against 5,820 GCUPS) pay more for their skew there than a second pass
// costs; four wavefronts of 8 lanes (144: 4,190 against 4,960) lose to their bank
// conflicts and uneven pairs.  Blocks of 8 warps, two (above 16 rows a lane: 128
// registers) to four an SM; long queries, whose profile would not leave room for two
// blocks, take blocks of 16 warps, one an SM, with 32 lanes a wavefront (5,478
// residues: 5,760 GCUPS at R = 29, against 5,270 in two wavefronts a warp, whose
// twice as many boundary rows outgrow the L1 cache that the profile leaves).
// A small database is bound by its longest subject, whose steps follow one another:
// there 32 lanes a wavefront win, whose steps are shorter (a warp of two wavefronts loads two
// pairs' profile rows, in conflict) and which need half the passes: 8,000 subjects (the longest of
// 3,574) x 1,000: 2,632 us at 32 rows in 16 lanes, 1,295 in 32; one subject x 4,000: 772 and 336 us.
constexpr int kDbA = 6, kDbB = 5, kDbC = 6, kDbD = 8;   // shapes per translation unit
constexpr int kDbShapeCount = kDbA + kDbB + kDbC + kDbD;
constexpr int kDbCompact = kDbA + kDbB + kDbC - 1;      // 16 rows a lane in 32 lanes, 16 warps: the last resort
constexpr size_t kDbNarrowProfileMax = 100 * 1024;      // profile bytes of a two-blocks-an-SM shape at most

const DbShape &shape_at(int s) {
    static const auto all = [] {
        std::vector<DbShape> v;
        for (int k = 0; k < kDbA; ++k) v.push_back(db_shape_a(k));
        for (int k = 0; k < kDbB; ++k) v.push_back(db_shape_b(k));
        for (int k = 0; k < kDbC; ++k) v.push_back(db_shape_c(k));
        for (int k = 0; k < kDbD; ++k) v.push_back(db_shape_d(k));
        return v;
    }();
    return all[(size_t)s];
}

// Seconds a shape takes for a query of m residues, by its measured rate and step (DbShape): the work over the chip's
// rate and the longest pair's chain, in a norm close to their larger one.  Blocks of 16 warps have twice the
// chains on an SM.  The exponent and the small factors are fitted to every shape's times for 25 query lengths from
// 30 to 8,000 against eight databases of 1 to 500,000 subjects: the choice is on average 0.1% and at most 6%
// above the fastest shape (by the work alone 30%, and 2.6 times the time at worst).
double db_shape_time(const DbShape &q, int m, const DbLoad &ld, int nsm) {
    const int rows = q.G * q.R, passes = (m + rows - 1) / rows;
    const double blocks = std::min<double>((double)db_blocks_per_sm(q.R, q.W) * nsm, std::ceil(ld.pairs / q.W));
    const double used = std::max(1.0, std::min<double>(nsm, blocks));
    const double work = (double)passes * rows * 2.0 * ld.cols / (q.gcups * 1e9) * (nsm / used) *
                        (q.G == 16 ? 1.0 : (q.W >= 16 ? 1.02 : 0.98));
    const double chains = std::min<double>(q.W, ld.pairs * q.G / 32.0);     // at once in a block
    // (two wavefronts a warp: the longest pair goes on without its neighbour at the end, at a checked step)
    const double clk = (passes == 1 ? q.clk1 : q.clk) + (q.G == 16 ? 15 : 0);
    const double chain = (double)passes * (ld.maxlen + q.G) * clk / 2.07e9 * std::max(1.0, 1.25 * chains / 8);
    return std::sqrt(std::sqrt(work * work * work * work + chain * chain * chain * chain));
}

}  // namespace

// The shape for a query of m residues against a database of `codes` residue codes, of which the launch sweeps
// ld: the fastest by db_shape_time among the shapes whose profile fits.
int swgb::db_shape(const sw_ctx *c, int codes, int m, const DbLoad &ld) {
    auto fits = [&](int s) {
        const size_t p = shape_at(s).profile_bytes(codes, m);
        return shape_at(s).W < 16 ? p <= kDbNarrowProfileMax : (long long)p <= kMaxProfileSmem;
    };
    // tuning override: SWGB_DB_SHAPE=<index of a shape>, where its profile fits
    if (c->db_forced >= 0 && c->db_forced < kDbShapeCount && fits(c->db_forced)) return c->db_forced;
    int best = kDbCompact;
    double best_time = 1e300;
    for (int s = 0; s < kDbShapeCount; ++s) {
        if (!fits(s)) continue;
        const double t = db_shape_time(shape_at(s), m, ld, c->nsm);
        if (t < best_time) { best_time = t; best = s; }
    }
    return best;
}

double swgb::db_shape_seconds(const sw_ctx *c, int shape, int m, const DbLoad &ld) {
    return db_shape_time(shape_at(shape), m, ld, c->nsm);
}

int swgb::db_resident_blocks_shape(sw_ctx *c, int shape, int codes, int m, int *out) {
    return shape_at(shape).resident(c, codes, m, out);
}

int swgb::db_shape_warps(int shape) { return shape_at(shape).W; }
int swgb::db_shape_rows(int shape) { return shape_at(shape).G * shape_at(shape).R; }

int swgb::db_launch_shape(sw_ctx *c, int shape, const DbJob *jobs, int njobs, int nblocks, const DbView &D, int codes,
                          int m, const DbBufs *bufs) {
    DbBufs B{&c->dbscratch, &c->dbslots, static_cast<const DevScoring *>(c->scorings.p), static_cast<int *>(c->err.p)};
    if (bufs) B = *bufs;
    return shape_at(shape).launch(c, jobs, njobs, nblocks, D, codes, m, B);
}

int swgb::db_scratch_shape(sw_ctx *c, int shape, int codes, int m, int maxlen, size_t *row_bytes, size_t *slot_bytes) {
    int nslots = 0;
    return shape_at(shape).scratch(c, codes, m, maxlen, &nslots, row_bytes, slot_bytes);
}

int swgb::db_view(const sw_db *db, DbView *v, int64_t *nseq, int32_t *max_code, int *device) {
    v->res = static_cast<const uint8_t *>(db->res.p);
    v->off = static_cast<const int64_t *>(db->doff.p);
    v->pairs = static_cast<const int32_t *>(db->pairs.p);
    v->pres = static_cast<const uint16_t *>(db->pres.p);
    v->poff = static_cast<const int64_t *>(db->poff.p);
    v->npairs = db->npairs;
    v->pad = db->max_code + 1;
    v->maxlen = db->maxlen;
    *nseq = db->nseq;
    *max_code = db->max_code;
    *device = db->device;
    return SW_OK;
}

int64_t swgb::db_pair_columns(const sw_db *db) { return db->pcols; }

int64_t swgb::db_total_residues(const sw_db *db) { return db->off.empty() ? 0 : db->off.back(); }

int swgb::db_chunk_maxlen(const sw_db *db, int32_t pair0, int32_t pair1) {
    int64_t mx = 0;
    for (int32_t p = pair0; p < pair1 && p < db->npairs; ++p)
        for (int h = 0; h < 2; ++h) {
            const int32_t s = db->hpairs[(size_t)(2 * p + h)];
            if (s >= 0) mx = std::max(mx, db->off[(size_t)s + 1] - db->off[(size_t)s]);
        }
    return (int)mx;
}

extern "C" int sw_db_create(sw_ctx *c, const uint8_t *residues, const int64_t *offsets, int64_t nseq,
                            sw_db **out) {
    if (!c || !out || !offsets || nseq < 0 || nseq > (int64_t)1 << 30) return SW_EINVAL;
    if (offsets[0] != 0) return SW_EINVAL;
    for (int64_t s = 0; s < nseq; ++s) {
        if (offsets[s + 1] < offsets[s]) return SW_EINVAL;
        if (offsets[s + 1] - offsets[s] > SW_MAX_LEN) return SW_ERANGE;
    }
    const int64_t total = offsets[nseq];
    if (total > 0 && !residues) return SW_EINVAL;
    DeviceGuard g(c->device);
    sw_db *db = new (std::nothrow) sw_db();
    if (!db) return SW_ENOMEM;
    db->device = c->device;
    db->nseq = nseq;
    db->off.assign(offsets, offsets + nseq + 1);
    int rc = db->res.ensure((size_t)total + 16);
    if (!rc) rc = db->doff.ensure((size_t)(nseq + 1) * sizeof(int64_t));
    if (rc) { delete db; return rc; }
    // length-sorted pairs, longest first (ties by index)
    std::vector<int32_t> order((size_t)nseq);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) {
        return offsets[x + 1] - offsets[x] > offsets[y + 1] - offsets[y];
    });
    db->npairs = (int32_t)((nseq + 1) / 2);
    std::vector<int32_t> pairs((size_t)db->npairs * 2, -1);
    for (int64_t k = 0; k < nseq; ++k) pairs[(size_t)k] = order[(size_t)k];
    int64_t maxlen = 0;
    for (int64_t s = 0; s < nseq; ++s) maxlen = std::max(maxlen, offsets[s + 1] - offsets[s]);
    db->maxlen = (int32_t)maxlen;
    db->hpairs = pairs;
    rc = db->pairs.ensure(std::max<size_t>(1, pairs.size()) * sizeof(int32_t));
    if (rc) { delete db; return rc; }
    // interleaved residues of the pairs: max(na, nb) columns plus one padding column each
    std::vector<int64_t> poff((size_t)db->npairs + 1, 0);
    for (int32_t p = 0; p < db->npairs; ++p) {
        const int32_t sa = pairs[2 * (size_t)p], sb = pairs[2 * (size_t)p + 1];
        const int64_t na = offsets[sa + 1] - offsets[sa];
        const int64_t nb = sb >= 0 ? offsets[sb + 1] - offsets[sb] : 0;
        poff[(size_t)p + 1] = poff[(size_t)p] + std::max(na, nb) + 1;
    }
    db->pcols = poff.back() - db->npairs;
    rc = db->pres.ensure(std::max<size_t>(1, (size_t)poff.back()) * sizeof(uint16_t));
    if (!rc) rc = db->poff.ensure(poff.size() * sizeof(int64_t));
    if (rc) { delete db; return rc; }
    const cudaMemcpyKind kind = is_device_ptr(residues) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    bool ok = true;
    if (total > 0) ok &= cudaMemcpyAsync(db->res.p, residues, (size_t)total, kind, c->stream) == cudaSuccess;
    ok &= cudaMemcpyAsync(db->doff.p, offsets, (size_t)(nseq + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, c->stream) == cudaSuccess;
    if (!pairs.empty())
        ok &= cudaMemcpyAsync(db->pairs.p, pairs.data(), pairs.size() * sizeof(int32_t), cudaMemcpyHostToDevice, c->stream) == cudaSuccess;
    ok &= cudaMemcpyAsync(db->poff.p, poff.data(), poff.size() * sizeof(int64_t), cudaMemcpyHostToDevice, c->stream) == cudaSuccess;
    // largest residue code: checked against the alphabet at search time; the next one is the pairs' padding
    ok &= c->misc.ensure(sizeof(int)) == SW_OK;
    ok &= cudaMemsetAsync(c->misc.p, 0, sizeof(int), c->stream) == cudaSuccess;
    if (ok && total > 0) {
        max_code_kernel<<<(unsigned)std::min<long long>((total + 255) / 256, 8LL * c->nsm), 256, 0, c->stream>>>(
            static_cast<const uint8_t *>(db->res.p), total, static_cast<int *>(c->misc.p));
        ok &= cudaGetLastError() == cudaSuccess;
        ++c->launches;
    }
    int mc = 0;
    ok &= cudaMemcpyAsync(&mc, c->misc.p, sizeof(int), cudaMemcpyDeviceToHost, c->stream) == cudaSuccess;
    ok &= cudaStreamSynchronize(c->stream) == cudaSuccess;
    if (ok && db->npairs > 0) {
        pair_residues_kernel<<<(unsigned)std::min<long long>((db->npairs + 7) / 8, 16LL * c->nsm), 256, 0, c->stream>>>(
            static_cast<const uint8_t *>(db->res.p), static_cast<const int64_t *>(db->doff.p),
            static_cast<const int32_t *>(db->pairs.p), static_cast<const int64_t *>(db->poff.p), db->npairs,
            (unsigned)(total > 0 ? mc + 1 : 0), static_cast<uint16_t *>(db->pres.p));
        ok &= cudaGetLastError() == cudaSuccess;
        ++c->launches;
    }
    ok &= cudaStreamSynchronize(c->stream) == cudaSuccess;   // (the offsets' host copies are read until here)
    if (!ok) { cudaGetLastError(); delete db; return SW_ECUDA; }
    db->max_code = total > 0 ? mc : -1;
    *out = db;
    return SW_OK;
}

extern "C" void sw_db_destroy(sw_db *db) {
    if (!db) return;
    DeviceGuard g(db->device);
    delete db;
}

extern "C" int64_t sw_db_size(const sw_db *db) { return db ? db->nseq : -1; }

// Score every subject of the database against query q (device array
// scores, int32 per subject), flagged subjects rescored exactly.
int swgb::db_score_all(sw_ctx *c, const sw_db *db, const uint8_t *dq, int64_t m, const DevScoring &ds,
                       int32_t *dscores) {
    RC(c->dbovf.ensure((size_t)std::max<int64_t>(1, db->nseq) * sizeof(int32_t)));
    RC(c->dbjob.ensure(sizeof(DbJob) + 64));
    int32_t *novf = reinterpret_cast<int32_t *>(static_cast<char *>(c->dbjob.p) + sizeof(DbJob));
    int32_t *next = novf + 1;
    CU(cudaMemsetAsync(novf, 0, 2 * sizeof(int32_t), c->stream));
    DbJob job;
    job.q = dq; job.m = (int32_t)m; job.scoring = 0;
    job.pair0 = 0; job.pair1 = db->npairs; job.pair_stride = 1; job.block0 = 0;
    job.scores = dscores;
    job.ovf = static_cast<int32_t *>(c->dbovf.p);
    job.novf = novf; job.next_pair = next;
    RC(c->stage.ensure(sizeof(DbJob)));
    std::memcpy(c->stage.p, &job, sizeof(job));
    CU(cudaMemcpyAsync(c->dbjob.p, c->stage.p, sizeof(job), cudaMemcpyHostToDevice, c->stream));
    DbView D;
    D.res = static_cast<const uint8_t *>(db->res.p);
    D.off = static_cast<const int64_t *>(db->doff.p);
    D.pairs = static_cast<const int32_t *>(db->pairs.p);
    D.pres = static_cast<const uint16_t *>(db->pres.p);
    D.poff = static_cast<const int64_t *>(db->poff.p);
    D.npairs = db->npairs;
    D.pad = db->max_code + 1;
    D.maxlen = db->maxlen;
    int32_t nflag = 0;
    std::vector<int32_t> flagged;
    const bool packed_ok = fold_open(ds) && ds.go <= 16000 && ds.ge <= 16000;
    int rc = SW_ERANGE;
    if (packed_ok) {
        int nblk = 0;
        const DbLoad ld{(double)db->npairs, (double)db->pcols, db->maxlen};
        const int shape = db_shape(c, D.pad, (int)m, ld);
        rc = db_resident_blocks_shape(c, shape, D.pad, (int)m, &nblk);
        // A long query against few subjects: one int32 task a subject puts all SMs on the query's rows, where the
        // packed search has a warp for each pair.  270 us and 590 GCUPS as measured (9,000 residues, packed / int32: 1 subject 0.79 /
        // 0.29 ms, 30 2.64 / 0.38, 1,000 8.5 / 5.5, 8,000 13.8 / 43.2)
        if (!rc && c->db_forced < 0 &&
            db_shape_seconds(c, shape, (int)m, ld) > 270e-6 + (double)m * (double)db_total_residues(db) / 590e9)
            rc = SW_ERANGE;
        if (!rc) {
            const int W = db_shape_warps(shape);
            nblk = std::max(1, std::min(nblk, (db->npairs + W - 1) / W));
            rc = db_launch_shape(c, shape, static_cast<const DbJob *>(c->dbjob.p), 1, nblk, D, D.pad, (int)m);
        }
    }
    if (rc == SW_ERANGE) {
        // the packed kernel cannot take this query or scoring, or not as fast: score every subject in int32
        flagged.resize((size_t)db->nseq);
        std::iota(flagged.begin(), flagged.end(), 0);
    } else {
        RC(rc);
        CU(cudaMemcpyAsync(c->stage3.p, novf, sizeof(int32_t), cudaMemcpyDeviceToHost, c->stream));
        CU(cudaStreamSynchronize(c->stream));
        std::memcpy(&nflag, c->stage3.p, sizeof(int32_t));
        if (nflag > 0) {
            flagged.resize((size_t)nflag);
            CU(cudaMemcpy(flagged.data(), c->dbovf.p, (size_t)nflag * sizeof(int32_t), cudaMemcpyDeviceToHost));
        }
    }
    if (flagged.empty()) return SW_OK;
    return db_rescore(c, db, dq, m, ds, flagged, dscores);
}

// Exact rescoring: one int32 wavefront task per flagged subject (query down
// the rows); scores[flagged[k]] receives the result.
int swgb::db_rescore(sw_ctx *c, const sw_db *db, const uint8_t *dq, int64_t m, const DevScoring &ds,
                     const std::vector<int32_t> &flagged, int32_t *dscores) {
    const int K = ds.K;
    RC(upload_scorings(c, {ds}));
    // (SWGB_BATCH may name a packed shape, which need not be exact for this scoring)
    const FillConfig cfg = c->bat.P16 ? FillConfig{8, 4} : c->bat;
    const int HC = fill_rows_per_strip(cfg);
    std::vector<FillTask> tasks;
    tasks.reserve(flagged.size());
    long long tickets = 0;
    size_t bnd_need = 0;
    for (int32_t s : flagged) {
        const int64_t n = db->off[(size_t)s + 1] - db->off[(size_t)s];
        const int ns = (int)((m + HC - 1) / HC);
        bnd_need += (size_t)std::min(ns, 2) * (size_t)std::max<int64_t>(n, 1) * sizeof(int2);
    }
    RC(c->tbbnd.ensure(bnd_need));
    size_t boff = 0;
    for (int32_t s : flagged) {
        FillTask u{};
        const int64_t n = db->off[(size_t)s + 1] - db->off[(size_t)s];
        u.a = dq; u.rows = (int32_t)m;
        u.b = static_cast<const uint8_t *>(db->res.p) + db->off[(size_t)s];
        u.ncols = (int32_t)n;
        u.nstrips = (int32_t)((m + HC - 1) / HC);
        u.scoring = 0;
        u.ticket0 = tickets;
        u.nslot = std::min(u.nstrips, 2);
        u.bnd = reinterpret_cast<int2 *>(static_cast<char *>(c->tbbnd.p) + boff);
        boff += (size_t)u.nslot * (size_t)std::max<int64_t>(n, 1) * sizeof(int2);
        tickets += n > 0 ? u.nstrips : 0;
        if (n == 0) { u.nstrips = 0; }
        tasks.push_back(u);
    }
    RC(run_fill(c, cfg, kModeScore, fold_open(ds), tasks, tickets, K));
    const int nt = (int)tasks.size();
    RC(c->result.ensure((size_t)nt * sizeof(int4)));
    reduce_candidates_kernel<<<(nt + 7) / 8, 256, 0, c->stream>>>(static_cast<const FillTask *>(c->tasks.p), nt,
                                                                  static_cast<const int4 *>(c->cand.p),
                                                                  static_cast<const DevScoring *>(c->scorings.p),
                                                                  static_cast<int4 *>(c->result.p));
    CU(cudaGetLastError());
    ++c->launches;
    RC(c->dbovf.ensure((size_t)nt * sizeof(int32_t)));
    CU(cudaMemcpyAsync(c->dbovf.p, flagged.data(), (size_t)nt * sizeof(int32_t), cudaMemcpyHostToDevice, c->stream));
    scatter_scores_kernel<<<(nt + 255) / 256, 256, 0, c->stream>>>(static_cast<const int32_t *>(c->dbovf.p),
                                                                   static_cast<const int4 *>(c->result.p), nt, dscores);
    CU(cudaGetLastError());
    ++c->launches;
    CU(cudaStreamSynchronize(c->stream));      // flagged is host memory used by the copy above
    return SW_OK;
}

// Top-k of a device score array: (subject, score) pairs, score descending,
// subject ascending.
int swgb::db_topk(sw_ctx *c, const int32_t *dscores, int64_t nseq, int k, int2 *dout) {
    const int nb = (int)((nseq + kTopkChunk - 1) / kTopkChunk);
    RC(c->topk.ensure((size_t)std::max(1, nb) * k * sizeof(unsigned long long)));
    topk_phase1_kernel<<<nb, kTopkThreads, 0, c->stream>>>(dscores, (int)nseq, k,
                                                           static_cast<unsigned long long *>(c->topk.p));
    CU(cudaGetLastError());
    ++c->launches;
    const size_t smem = (size_t)nb * k * sizeof(unsigned long long);
    static int attr_set = 0;
    if (!attr_set) {
        CU(cudaFuncSetAttribute(topk_phase2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
        attr_set = 1;
    }
    if (smem > 200 * 1024) return SW_ERANGE;
    topk_phase2_kernel<<<1, kTopkThreads, smem, c->stream>>>(static_cast<const unsigned long long *>(c->topk.p),
                                                             nb * k, k, dout);
    CU(cudaGetLastError());
    ++c->launches;
    return SW_OK;
}

extern "C" int sw_dbsearch(sw_ctx *c, const sw_db *db, const uint8_t *q, int64_t m, const sw_scoring *sc,
                           int32_t k, sw_dbhit *hits, int32_t *nhits, int32_t *all_scores) {
    if (!c || !db || !nhits || k < 0 || k > 64 || (k > 0 && !hits)) return SW_EINVAL;
    if (db->device != c->device) return SW_EINVAL;
    DevScoring ds;
    RC(check_scoring(sc, &ds));
    if (ds.alg != kAlgLocal) return SW_EINVAL;          // database search: the local algorithm
    if (m < 0 || (m > 0 && !q)) return SW_EINVAL;
    if (m > SW_MAX_LEN) return SW_ERANGE;
    if (db->max_code >= ds.K) return SW_EINVAL;
    if ((double)std::min<int64_t>(m, db->maxlen) * (double)max_pos_score(sc) >= (double)kMaxScoreBound) return SW_ERANGE;
    DeviceGuard g(c->device);
    const int64_t nseq = db->nseq;
    RC(c->dbscores.ensure((size_t)std::max<int64_t>(1, nseq) * sizeof(int32_t)));
    int32_t *dscores = static_cast<int32_t *>(c->dbscores.p);
    if (nseq > 0) CU(cudaMemsetAsync(dscores, 0, (size_t)nseq * sizeof(int32_t), c->stream));
    if (m > 0 && nseq > 0) {
        const uint8_t *dq;
        RC(stage_seq(c, q, m, c->seq_a, &dq));
        RC(reset_err(c));
        RC(validate_codes(c, dq, m, ds.K));
        RC(upload_scorings(c, {ds}));
        RC(db_score_all(c, db, dq, m, ds, dscores));
    }
    const int kk = (int)std::min<int64_t>(k, nseq);
    if (kk > 0) {
        RC(c->result.ensure(64 * sizeof(int4)));
        RC(db_topk(c, dscores, nseq, kk, static_cast<int2 *>(c->result.p)));
        CU(cudaMemcpyAsync(c->stage3.p, c->result.p, (size_t)kk * sizeof(int2), cudaMemcpyDeviceToHost, c->stream));
    }
    CU(cudaMemcpyAsync(static_cast<char *>(c->stage3.p) + 1024, c->err.p, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    if (all_scores && nseq > 0) {
        CU(cudaMemcpyAsync(all_scores, dscores, (size_t)nseq * sizeof(int32_t),
                           is_device_ptr(all_scores) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, c->stream));
    }
    CU(cudaStreamSynchronize(c->stream));
    int e;
    std::memcpy(&e, static_cast<char *>(c->stage3.p) + 1024, sizeof(int));
    RC(map_kernel_error(e));
    const int2 *h = static_cast<const int2 *>(c->stage3.p);
    for (int i = 0; i < kk; ++i) hits[i] = sw_dbhit{(int64_t)h[i].x, h[i].y, 0};
    *nhits = kk;
    return SW_OK;
}
