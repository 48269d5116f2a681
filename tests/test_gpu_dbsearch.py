"""GPU parity of the database search (sw_db_create / sw_dbsearch) against the
CPU oracle: every subject's score exactly, the top-k order (score
descending, subject index ascending), the packed-16-bit saturation path and
its exact 32-bit rescoring, long queries, and degenerate databases."""
import numpy as np
import pytest

from paper_2211_10769_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2211_10769_gb300 import binding, build
    build.build()
    c = binding.Context(0)
    yield c
    c.close()


def _db(ctx, subjects):
    from paper_2211_10769_gb300 import binding
    lens = np.array([len(s) for s in subjects], dtype=np.int64)
    off = np.zeros(len(subjects) + 1, dtype=np.int64)
    np.cumsum(lens, out=off[1:])
    res = np.concatenate(subjects) if len(subjects) and off[-1] > 0 else np.zeros(0, np.uint8)
    return binding.Database(ctx, res, off)


def _check_all(ctx, oracle_mod, db, subjects, q, sc, k=20):
    hits, scores = db.search(q, sc.matrix, sc.gap_open, sc.gap_extend, k=k, all_scores=True)
    want = oracle_mod.db_scores(q, subjects, sc.matrix, sc.gap_open, sc.gap_extend)
    bad = np.nonzero(scores != want)[0]
    assert bad.size == 0, (bad[:10], scores[bad[:10]], want[bad[:10]])
    assert hits == oracle_mod.top_k(want, min(k, len(subjects)))
    return want


def test_small_database_all_scores(ctx, oracle_mod):
    sc = W.protein_scoring()
    qs = W.protein_queries((144, 464))
    pdb = W.protein_db(3000, queries=qs, seed_offset=700)
    subjects = [pdb.subject(s) for s in range(pdb.nseq)]
    db = _db(ctx, subjects)
    for qi, q in enumerate(qs):
        want = _check_all(ctx, oracle_mod, db, subjects, q, sc)
        top = oracle_mod.top_k(want, 3)
        assert {s for s, _ in top} & set(pdb.planted[qi])     # the planted homologs are found


def test_every_tile_shape(ctx, oracle_mod):
    """Query lengths that pick the tile shapes of the packed search (two
    16-lane wavefronts a warp at 4 to 32 rows a lane; 16-warp blocks for long
    queries), with one or several passes, the last pass partly padding, and
    warps whose second wavefront finds no pair left."""
    sc = W.protein_scoring()
    lengths = (1, 31, 80, 100, 128, 144, 160, 161, 190, 250, 300, 350, 384, 464, 700, 1000, 1500, 4100)
    qs = W.protein_queries(lengths, seed_offset=760)
    pdb = W.protein_db(400, queries=qs, seed_offset=770)
    subjects = [pdb.subject(s) for s in range(pdb.nseq)]
    db = _db(ctx, subjects)
    for q in qs:
        _check_all(ctx, oracle_mod, db, subjects, q, sc)


@pytest.mark.parametrize("codes", [20, 24])
def test_shape_edges(ctx, oracle_mod, codes):
    """Queries of exactly 16 R rows and one more for every R of the shapes, one to many passes, up to
    the blocks of 16 warps; a database whose residues use every code of the alphabet (the padding code
    is then the alphabet size) and one that stops at 20."""
    sc = W.protein_scoring()
    g = np.random.default_rng(W.BASE_SEED + 765 + codes)
    subjects = [g.integers(0, codes, size=int(n)).astype(np.uint8) for n in (1, 15, 16, 17, 40, 333, 334, 90, 700)]
    subjects[3][0] = codes - 1
    db = _db(ctx, subjects)
    for rows in (4, 7, 9, 11, 13, 16, 18, 20, 22, 24, 26, 29, 32):
        for m in (16 * rows, 16 * rows + 1):
            q = g.integers(0, 24, size=m).astype(np.uint8)
            _check_all(ctx, oracle_mod, db, subjects, q, sc, k=5)
    for m in (4090, 5200, 6100, 7999):
        _check_all(ctx, oracle_mod, db, subjects, g.integers(0, 24, size=m).astype(np.uint8), sc, k=5)


def test_long_query_few_subjects(ctx, oracle_mod):
    """Queries on both sides of the line above which a few subjects are scored in int32 tasks, up to one that the
    packed profile has no room for with this database's codes."""
    sc = W.protein_scoring()
    g = np.random.default_rng(W.BASE_SEED + 795)
    subjects = [g.integers(0, 20, size=int(n)).astype(np.uint8) for n in (700, 3, 1, 333, 90, 1500)]
    db = _db(ctx, subjects)
    for m in (500, 1500, 2500, 4000, 9000, 10000):
        q = np.concatenate([W.mutate(subjects[5], 20, W.BASE_SEED + 796), W.random_protein(m, W.BASE_SEED + m)])[:m]
        _check_all(ctx, oracle_mod, db, subjects, q, sc, k=4)
    db.close()


SHAPES = [(r, 16) for r in (4, 7, 9, 11, 13, 16, 18, 20, 22, 24, 26, 29, 32)] + \
    [(32, 32), (29, 32), (24, 32), (16, 32), (6, 16), (4, 32), (8, 32), (12, 32), (16, 32), (24, 32), (32, 32), (12, 16)]


@pytest.mark.parametrize("shape", range(len(SHAPES)))
def test_forced_shapes(oracle_mod, monkeypatch, shape):
    """Every tile shape (by its index) at one pass less a row, exactly one, one row more and two and a half passes,
    over subjects shorter than, equal to and longer than a wavefront, an odd number of them."""
    from paper_2211_10769_gb300 import binding
    monkeypatch.setenv("SWGB_DB_SHAPE", str(shape))
    c = binding.Context(0)
    try:
        sc = W.protein_scoring()
        g = np.random.default_rng(W.BASE_SEED + 790 + shape)
        subjects = [g.integers(0, 20, size=int(n)).astype(np.uint8) for n in (1, 15, 16, 17, 31, 32, 33, 90, 333, 334, 800)]
        db = _db(c, subjects)
        rows = SHAPES[shape][0] * SHAPES[shape][1]
        for m in (rows - 1, rows, rows + 1, 2 * rows + rows // 2):
            _check_all(c, oracle_mod, db, subjects, g.integers(0, 24, size=m).astype(np.uint8), sc, k=5)
        db.close()
    finally:
        c.close()


@pytest.mark.parametrize("nseq", [1, 2, 3, 5, 7])
def test_tiny_databases_short_queries(ctx, oracle_mod, nseq):
    """One to four subject pairs against queries that take the two-wavefront
    shapes: most warps find one pair or none, and a warp's second wavefront
    often has no pair (its lanes still take part in the shuffles)."""
    sc = W.protein_scoring()
    g = np.random.default_rng(W.BASE_SEED + 780 + nseq)
    subjects = [W.random_protein(int(g.integers(1, 400)), W.BASE_SEED + 790 + 10 * nseq + i) for i in range(nseq)]
    db = _db(ctx, subjects)
    for m in (5, 60, 90, 140, 190):
        q = W.random_protein(m, W.BASE_SEED + 800 + m)
        if nseq > 2:
            subjects_q = list(subjects)
            subjects_q[1] = W.mutate(q, 20, W.BASE_SEED + 801 + m, p_sub=0.2)   # a homolog among them
            dbq = _db(ctx, subjects_q)
            _check_all(ctx, oracle_mod, dbq, subjects_q, q, sc, k=min(4, nseq))
        _check_all(ctx, oracle_mod, db, subjects, q, sc, k=min(4, nseq))


def test_long_query_and_dna(ctx, oracle_mod):
    sc = W.protein_scoring()
    q = W.protein_queries((5478,))[0]
    pdb = W.protein_db(160, queries=[q], seed_offset=710)
    subjects = [pdb.subject(s) for s in range(pdb.nseq)]
    _check_all(ctx, oracle_mod, _db(ctx, subjects), subjects, q, sc)
    dna = W.dna_scoring()
    dsubj = [W.uniform_dna(int(L), W.BASE_SEED + 720 + i) for i, L in enumerate(np.linspace(1, 900, 97))]
    dq = W.uniform_dna(700, W.BASE_SEED + 719)
    dsubj[5] = W.mutate(dq, 4, W.BASE_SEED + 730)
    _check_all(ctx, oracle_mod, _db(ctx, dsubj), dsubj, dq, dna, k=10)


def test_saturating_subjects_are_rescored(ctx, oracle_mod):
    """Scores above 32767 - max(S) cannot stay in 16-bit lanes: a W-rich query
    against W-rich subjects pushes them over; those must come back exact."""
    sc = W.protein_scoring()
    Wc = W.PROTEIN_ALPHABET.index("W")
    g = np.random.default_rng(W.BASE_SEED + 740)
    q = np.full(3300, Wc, np.uint8)
    q[g.integers(0, 3300, 40)] = 0
    subjects = []
    for i in range(40):
        if i % 4 == 0:
            s = q.copy()
            s[g.integers(0, len(s), 30)] = 3
        else:
            s = W.random_protein(int(g.integers(50, 900)), W.BASE_SEED + 750 + i)
        subjects.append(s)
    want = _check_all(ctx, oracle_mod, _db(ctx, subjects), subjects, q, sc)
    assert (want > 32767 - 11).sum() >= 10


@pytest.mark.parametrize("go,ge", [(0, 0), (1, 1), (10, 1), (11, 11), (60, 2), (110, 110)])
def test_half_beside_a_saturated_one(ctx, oracle_mod, go, ge):
    """A saturating subject in either half of a packed pair leaves its
    neighbour's score exact (the halves share plain 32-bit subtractions), and
    so do scores just below and above the flagging threshold."""
    S = W.blosum62()
    Wc = W.PROTEIN_ALPHABET.index("W")
    q = np.full(3100, Wc, np.uint8)
    q[np.arange(0, 3100, 150)] = 0
    subjects = [q.copy(), W.random_protein(3100, W.BASE_SEED + 781),           # low half saturates
                W.random_protein(3090, W.BASE_SEED + 782), q[:3090].copy()]    # high half saturates
    # runs of W around (32767 - 11 - go) / 11 residues: on both sides of the threshold
    edge = (32767 - 11 - go) // 11
    q2 = np.full(edge + 6, Wc, np.uint8)
    runs = [np.full(edge + d, Wc, np.uint8) for d in (-2, -1, 0, 1, 2, 3)]
    for query, subj in ((q, subjects), (q2, runs)):
        want = oracle_mod.db_scores(query, subj, S, go, ge)
        hits, scores = _db(ctx, subj).search(query, S, go, ge, k=4, all_scores=True)
        assert scores.tolist() == want.tolist()


@pytest.mark.parametrize("shape", ["12,4,1", "8,2,2"])
def test_rescoring_under_a_packed_batch_override(oracle_mod, monkeypatch, shape):
    """The rescoring of saturated subjects is an int32 fill whatever shape batches are told to take: here
    the packed one, with scores it is not exact for."""
    from paper_2211_10769_gb300 import binding
    monkeypatch.setenv("SWGB_BATCH", shape)
    c = binding.Context(0)
    try:
        S = np.full((24, 24), -60, np.int8)
        np.fill_diagonal(S, 90)
        a = W.random_protein(900, W.BASE_SEED + 798)
        subjects = [a, W.mutate(a, 20, W.BASE_SEED + 799, p_sub=0.05), W.random_protein(300, W.BASE_SEED + 800)]
        want = oracle_mod.db_scores(a, subjects, S, 30, 2)
        assert max(want) > 32767
        hits, scores = _db(c, subjects).search(a, S, 30, 2, k=2, all_scores=True)
        assert scores.tolist() == want.tolist()
    finally:
        c.close()


def test_degenerate_databases(ctx, oracle_mod):
    sc = W.protein_scoring()
    q = W.random_protein(200, W.BASE_SEED + 760)
    subjects = [np.zeros(0, np.uint8), W.random_protein(1, 1), np.zeros(0, np.uint8), W.random_protein(31, 2),
                W.random_protein(33, 3)]
    _check_all(ctx, oracle_mod, _db(ctx, subjects), subjects, q, sc, k=64)      # k > nseq
    one = [W.random_protein(250, 4)]
    _check_all(ctx, oracle_mod, _db(ctx, one), one, q, sc, k=5)
    hits, scores = _db(ctx, one).search(np.zeros(0, np.uint8), sc.matrix, 10, 1, k=3, all_scores=True)
    assert hits == [(0, 0)] and scores.tolist() == [0]


def test_full_size_database_sampled(ctx, oracle_mod):
    """The 500,000-subject database: every query's top hits and a seeded
    sample of subjects checked against the oracle one by one."""
    sc = W.protein_scoring()
    qs = W.protein_queries()
    pdb = W.protein_db(500_000, queries=qs)
    from paper_2211_10769_gb300 import binding
    db = binding.Database(ctx, pdb.residues, pdb.offsets)
    g = np.random.default_rng(W.BASE_SEED + 770)
    for qi, q in enumerate(qs):
        hits, scores = db.search(q, sc.matrix, sc.gap_open, sc.gap_extend, k=20, all_scores=True)
        nsample = 400 if len(q) < 1500 else 120
        sample = sorted(set(g.integers(0, pdb.nseq, nsample).tolist()) | set(pdb.planted[qi]) |
                        {s for s, _ in hits[:5]})
        for s in sample:
            assert scores[s] == oracle_mod.sw_score(q, pdb.subject(s), sc.matrix, sc.gap_open, sc.gap_extend)[0]
        # top-k is consistent with the score array (score desc, index asc)
        order = np.lexsort((np.arange(pdb.nseq), -scores.astype(np.int64)))[:20]
        assert hits == [(int(s), int(scores[s])) for s in order]
        assert set(pdb.planted[qi]) <= {s for s, _ in hits}
