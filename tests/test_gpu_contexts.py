"""Calls of two contexts on two host threads at once, and calls of one context between a batch's creation and its
replay: what a kernel asks for in one call (its shared memory grows with the alphabet, the longest word and the rows)
is no business of another call of the same kernel."""
import threading

import numpy as np
import pytest

from paper_2509_01654_gb300 import nw, synth

pytestmark = pytest.mark.gpu

SC = (1, -1, -1)


def _words(n, alphabet, lo, hi, seed):
    return synth.make_uniform_length_words(n, alphabet, 1.0, lo, hi, seed=seed)


class Program:
    """One context with a dictionary of `alphabet` codes, and the calls of a program on it."""

    def __init__(self, alphabet, length, n, C, seed):
        self.ctx = nw.Context(0)
        w = _words(n, alphabet, max(0, length - 3), length, seed)
        self.d = self.ctx.load_dictionary(w.codes, w.offsets, alphabet, SC)
        self.q = _words(3, alphabet, 0, length, seed + 1)
        r = np.random.default_rng(seed)
        self.i, self.j = r.integers(0, n, (2, 500)).astype(np.uint32)
        self.cand = ((np.arange(n)[:, None] + 1 + np.arange(min(C, n - 1))) % n).astype(np.uint32)
        self.rows = np.zeros((40 * C, 64), np.int8)
        self.rows[:, :63] = r.integers(-30, 31, (40 * C, 63))
        self.C = C

    def calls(self, kind):
        if kind == "query":
            return self.d.query(self.q.codes, self.q.offsets, 5)
        if kind == "pairs":
            return [self.d.score_pairs(self.i, self.j)]
        if kind == "rescore":
            return nw.rescore_topk(self.d, self.cand, 3)
        if kind == "topk":
            return self.d.all_pairs_topk(4)[:3]
        return nw.dot_topk(self.ctx, self.rows, self.C)


@pytest.mark.parametrize("kind,alphabet,C,rounds", [("query", 256, 96, 1500), ("topk", 256, 96, 800),
                                                    ("pairs", 128, 96, 3000), ("rescore", 128, 96, 1500),
                                                    ("dot", 128, 512, 150)])
def test_two_contexts_on_two_threads(kind, alphabet, C, rounds):
    programs = [Program(alphabet, 40, 700, C, 1), Program(4, 6, 300, 16, 2)]
    want = [p.calls(kind) for p in programs]
    stop, failures = threading.Event(), []

    def run(p, w, rounds):
        try:
            for _ in range(rounds):
                if stop.is_set():
                    return
                if not all(np.array_equal(x, y) for x, y in zip(p.calls(kind), w)):
                    raise AssertionError("results differ from the same call alone")
        except Exception as e:  # noqa: BLE001 -- reported below
            failures.append(repr(e))
        stop.set()

    threads = [threading.Thread(target=run, args=(p, w, r)) for p, w, r in zip(programs, want, (rounds, 1 << 30))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for p in programs:
        p.ctx.close()
    assert not failures


def test_queries_between_a_batch_and_its_replay():
    with nw.Context(0) as big, nw.Context(0) as small:
        w, q = _words(700, 250, 20, 40, 3), _words(40, 250, 20, 40, 4)
        batch = nw.Batch(big, [(w.codes, w.offsets, 250, SC, (q.codes, q.offsets))], k=6)
        want = batch.run_queries()
        v = _words(200, 3, 0, 5, 5)
        d = small.load_dictionary(v.codes, v.offsets, 3, SC)
        d.query(v.codes[:int(v.offsets[7])], v.offsets[:8], 6)
        got = batch.run_queries()
        for side_got, side_want in zip(got, want):
            for a, b in zip(side_got, side_want):
                assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
        again = nw.Batch(big, [(w.codes, w.offsets, 250, SC, (q.codes, q.offsets))], k=6).run_queries()
        assert np.array_equal(again[1][0][0], want[1][0][0])
