"""The bit-parallel alignment kernel's plans, on the CPU: every pair is in exactly one task, and a shard holds
the same pairs whichever kernel scores it."""
import numpy as np
import pytest

from paper_2509_01654_gb300 import nw


@pytest.fixture(scope="module")
def lib():
    from paper_2509_01654_gb300 import build
    build.build()
    return nw.load_library()


def _lengths(n, lo, hi, seed):
    return np.random.default_rng(seed).integers(lo, hi + 1, n).astype(np.uint32)


def _codes(a, b, n):
    lo, hi = np.minimum(a, b).astype(np.uint64), np.maximum(a, b).astype(np.uint64)
    return lo * np.uint64(n) + hi


# one bucket at a chunk's edges (256 words of up to eight symbols, 32 of more than 32), mixed lengths, empty words
@pytest.mark.parametrize("lengths", [
    np.full(2, 5), np.full(255, 8), np.full(257, 8), np.full(33, 40), np.full(65, 33),
    _lengths(700, 0, 40, 1), _lengths(900, 5, 12, 2), np.concatenate([np.zeros(40, int), _lengths(300, 1, 3, 3)])])
@pytest.mark.parametrize("ta", [0, 16, 256])
def test_all_pairs_once(lib, lengths, ta):
    n = len(lengths)
    a, b = nw.debug_enumerate_bit_pairs(lengths, ta=ta)
    assert a.size == n * (n - 1) // 2 and (a != b).all()
    assert np.unique(_codes(a, b, n)).size == a.size


@pytest.mark.parametrize("nq,n", [(1, 600), (700, 1), (300, 500), (40, 0)])
@pytest.mark.parametrize("ta", [0, 16, 256])
def test_query_pairs_once(lib, nq, n, ta):
    q, d = nw.debug_enumerate_bit_pairs(_lengths(n, 0, 25, 4), q_lengths=_lengths(nq, 0, 40, 5), ta=ta)
    assert q.size == nq * n and (n == 0 or (q.max() < nq and d.max() < n))
    assert np.unique(q.astype(np.uint64) * np.uint64(max(n, 1)) + d).size == nq * n


@pytest.mark.parametrize("nshards", [2, 3, 7, 64])
def test_shards_hold_the_same_pairs_as_the_dpx_plan(lib, nshards):
    lengths = np.concatenate([_lengths(900, 0, 12, 6), np.full(700, 7)])
    n = len(lengths)
    for s in range(nshards):
        a, b = nw.debug_enumerate_bit_pairs(lengths, shard=s, nshards=nshards)
        x, y = nw.debug_enumerate_pairs(lengths, s, nshards)
        assert np.array_equal(np.sort(_codes(a, b, n)), np.sort(_codes(x, y, n)))


@pytest.mark.parametrize("length", [2, 8, 16, 24, 32])
@pytest.mark.parametrize("queries", [64, 256, 1000])
def test_queries_of_one_length_are_the_a_words(lib, length, queries):
    """Cold query lists: the pairs of a task run over the dictionary's words first, whatever a few percent of rows say."""
    q, w = nw.debug_enumerate_bit_pairs([length] * 4100, [length] * queries)
    assert q.size == 4100 * queries
    assert (q[:32] == q[0]).all() and np.unique(w[:32]).size == 32
