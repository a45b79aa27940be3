"""The bit-parallel alignment kernel against the oracle, bit for bit: every step class it is built for, every number of
words per lane (word lengths 0 to 40), chunk edges, and the largest alphabet."""
import numpy as np
import pytest

from paper_2509_01654_gb300 import nw, synth

pytestmark = pytest.mark.gpu

# one scoring of each class of reduced steps (match - 2 gap, mismatch - 2 gap) / gcd, the last two beyond the kernel
SCORINGS = [(1, -2, -1), (0, -1, -1), (1, -1, -1), (1, -2, -4), (2, -1, -1), (0, -1, -2), (3, -1, -1), (1, -2, -2),
            (1, -1, -2), (1, 0, -2), (2, -2, -2), (1, -1, -3), (1, 1, -1)]


@pytest.fixture(scope="module")
def ctx():
    from paper_2509_01654_gb300 import build
    build.build()
    with nw.Context(0) as c:
        yield c


def _words(lengths, alphabet, seed):
    r = np.random.default_rng(seed)
    offs = np.zeros(len(lengths) + 1, np.uint32)
    offs[1:] = np.cumsum(lengths)
    return synth.WordList(r.integers(0, alphabet, int(offs[-1])).astype(np.uint8), offs, alphabet)


def _check(ctx, oracle, w, sc, k):
    d = ctx.load_dictionary(w.codes, w.offsets, w.alphabet, sc)
    idx, score, hist, lo = d.all_pairs_topk(k)
    wi, ws = oracle.topk_rows(w, np.arange(w.n), k, sc)
    ws = np.where(ws == oracle.MISSING_SCORE, nw.MISSING_SCORE, ws)
    assert np.array_equal(idx, wi) and np.array_equal(score.astype(np.int32), ws)
    assert np.array_equal(hist, oracle.histogram(w, sc, lo, hist.size))
    return d


@pytest.mark.parametrize("sc", SCORINGS)
def test_every_step_class_and_length(ctx, oracle_mod, sc):
    lengths = np.concatenate([np.arange(41), np.random.default_rng(1).integers(0, 41, 400)])
    w = _words(lengths, 4, 2)
    d = _check(ctx, oracle_mod, w, sc, 7)
    q = _words(np.random.default_rng(3).integers(0, 41, 90), 4, 4)
    qi, qs = d.query(q.codes, q.offsets, 7)
    oi, os_ = oracle_mod.query_topk(q, w, 7, sc)
    assert np.array_equal(qi, oi) and np.array_equal(qs.astype(np.int32), os_)
    d.free()


# the last word of a lane's field, of a chunk (32 words a lane slot) and of a strip
@pytest.mark.parametrize("length,n", [(8, 255), (8, 257), (9, 225), (12, 161), (21, 97), (32, 65), (33, 33), (40, 300)])
def test_single_length_chunk_edges(ctx, oracle_mod, length, n):
    _check(ctx, oracle_mod, _words([length] * n, 3, n), (1, -1, -1), 5).free()


def test_largest_alphabet_and_matrix(ctx, oracle_mod):
    w = _words(np.random.default_rng(5).integers(0, 26, 500), 256, 6)
    d = _check(ctx, oracle_mod, w, (1, -1, -1), 128)
    assert np.array_equal(d.all_pairs_matrix().astype(np.int32), oracle_mod.all_pairs(w, (1, -1, -1)))
    assert np.array_equal(d.all_pairs_matrix_chunked(10007).astype(np.int32), oracle_mod.all_pairs(w, (1, -1, -1)))
    d.free()


# words of up to 15 symbols (whole in a record), 32 (one 32-bit column word) and 40; few pairs read no records
@pytest.mark.parametrize("sc", SCORINGS[:10])
@pytest.mark.parametrize("top", [15, 32, 40])
@pytest.mark.parametrize("m", [30, 3001])
def test_explicit_pairs(ctx, oracle_mod, sc, top, m):
    lengths = np.concatenate([np.arange(top + 1), np.random.default_rng(7).integers(0, top + 1, 300)])
    w = _words(lengths, 5, 8 + top)
    d = ctx.load_dictionary(w.codes, w.offsets, w.alphabet, sc)
    r = np.random.default_rng(m)
    i, j = r.integers(0, w.n, m).astype(np.uint32), r.integers(0, w.n, m).astype(np.uint32)
    assert np.array_equal(d.score_pairs(i, j).astype(np.int32), oracle_mod.score_pairs(w, i, j, sc))
    d.free()


@pytest.mark.parametrize("sc", SCORINGS[:10])
@pytest.mark.parametrize("C,k", [(1, 1), (31, 40), (257, 10), (512, 128)])
def test_rescoring_every_class(ctx, oracle_mod, sc, C, k):
    w = _words(np.random.default_rng(9).integers(0, 41, 530), 4, 10)
    d = ctx.load_dictionary(w.codes, w.offsets, w.alphabet, sc)
    r = np.random.default_rng(C)
    cand = np.array([r.permutation(np.delete(np.arange(w.n), row))[:C] for row in range(w.n)]).astype(np.uint32)
    cand[r.random(cand.shape) < 0.1] = nw.MISSING_IDX
    idx, score = nw.rescore_topk(d, cand, k)
    full = np.zeros((w.n, w.n), np.int64)
    full[np.triu_indices(w.n, 1)] = oracle_mod.all_pairs(w, sc)
    full += full.T
    for row in range(0, w.n, 13):
        c = cand[row][cand[row] != nw.MISSING_IDX].astype(np.int64)
        c = c[np.lexsort((c, -full[row, c]))][:k]
        assert np.array_equal(idx[row, :c.size], c) and np.array_equal(score[row, :c.size], full[row, c])
        assert (idx[row, c.size:] == nw.MISSING_IDX).all() and (score[row, c.size:] == nw.MISSING_SCORE).all()
    d.free()


# words read 16 symbols at a time, blocks of 128, 64 and 32 threads by the size of the masks, and one length above 32
@pytest.mark.parametrize("alphabet", [7, 60, 97, 128])
@pytest.mark.parametrize("lengths", [[0, 1, 15, 16, 17, 31, 32], [0, 1, 15, 16, 17, 31, 32, 33, 40], [33]])
@pytest.mark.parametrize("sc", [(1, -1, -1), (0, -1, -1), (3, 0, -1)])
@pytest.mark.parametrize("m", [20, 2000])
def test_explicit_pairs_at_chunk_edges(ctx, oracle_mod, alphabet, lengths, sc, m):
    w = _words(np.random.default_rng(11).choice(lengths, 300), alphabet, alphabet)
    d = ctx.load_dictionary(w.codes, w.offsets, alphabet, sc)
    r = np.random.default_rng(m)
    i, j = r.integers(0, w.n, m).astype(np.uint32), r.integers(0, w.n, m).astype(np.uint32)
    by_length = np.argsort(np.maximum(w.lengths[i], w.lengths[j]), kind="stable")
    for p in (np.arange(m), by_length):
        assert np.array_equal(d.score_pairs(i[p], j[p]).astype(np.int32), oracle_mod.score_pairs(w, i[p], j[p], sc))
    d.free()


# classes whose pairs of words above 32 symbols go to the DPX kernel when there are many: 4.9M such pairs do, the
# parts of a sharded run (at most 1.7M each) and small query sets do not
@pytest.mark.parametrize("sc", [(2, -1, -1), (3, -1, -1), (3, 0, -1), (3, 1, -1)])
def test_long_words_of_the_dearest_classes(ctx, oracle_mod, sc):
    r = np.random.default_rng(13)
    w = _words(np.concatenate([r.integers(33, 41, 3150), r.integers(0, 33, 400)])[r.permutation(3550)], 6, 14)
    d = ctx.load_dictionary(w.codes, w.offsets, w.alphabet, sc)
    idx, score, hist, lo = d.all_pairs_topk(6)
    rows = r.integers(0, w.n, 12)
    wi, ws = oracle_mod.topk_rows(w, rows, 6, sc)
    assert np.array_equal(idx[rows], wi) and np.array_equal(score[rows].astype(np.int32), ws)
    parts = [d.all_pairs_topk(6, shard=(g, 3)) for g in range(3)]
    mi, ms = nw.topk_merge([p[:2] for p in parts], 6)
    assert np.array_equal(idx, mi) and np.array_equal(score, ms)
    assert np.array_equal(hist, sum(p[2] for p in parts)) and hist.sum() == w.n * (w.n - 1) // 2
    q = _words(r.integers(30, 41, 1900), 6, 15)
    qi, qs = d.query(q.codes, q.offsets, 6)
    for a in range(0, q.n, 500):
        part = q.subset(np.arange(a, min(q.n, a + 500)))
        pi, ps = d.query(part.codes, part.offsets, 6)
        assert np.array_equal(qi[a:a + 500], pi) and np.array_equal(qs[a:a + 500], ps)
    with nw.Context(0) as c:
        batch = nw.Batch(c, [(w.codes, w.offsets, 6, sc, (q.codes, q.offsets)), (q.codes, q.offsets, 6, (1, -1, -1))], k=6)
        (bi, bs), _ = batch.run_queries()[0]
        assert np.array_equal(bi, idx) and np.array_equal(bs, score)
        assert np.array_equal(batch.run_queries()[1][0][0], qi)
    d.free()


# query lists of one slot, of a warp's width and past it, which start empty under many warps at once; the similarity
# matrix of the second scoring has to give its lists
@pytest.mark.parametrize("k", [1, 7, 32, 33, 128])
@pytest.mark.parametrize("length,n,nq", [(6, 4000, 40), (12, 900, 300), (35, 300, 5)])
def test_query_lists_of_every_width(ctx, oracle_mod, k, length, n, nq):
    w, q = _words([length] * n, 5, n), _words([length] * nq, 5, nq)
    for sc in ((1, -1, -1), (4, -1, -1)):
        d = ctx.load_dictionary(w.codes, w.offsets, 5, sc)
        got = d.query(q.codes, q.offsets, k)
        wi, ws = oracle_mod.query_topk(q, w, k, sc)
        assert np.array_equal(got[0], wi) and np.array_equal(got[1].astype(np.int32), ws)
        d.free()
    d = ctx.load_dictionary_sim(w.codes, w.offsets, 5, np.where(np.eye(5, dtype=bool), 4, -1).astype(np.int32), -1)
    assert all(np.array_equal(x, y) for x, y in zip(d.query(q.codes, q.offsets, k), got))
    d.free()
