"""The word records that a dictionary keeps for long pair lists: when they are made, that scores are the same with and
without them, and that they never stand in the way of a call that fits without them."""
import numpy as np
import pytest

from paper_2509_01654_gb300 import nw, synth

pytestmark = pytest.mark.gpu

MANY = 3 << 20  # pairs after which a dictionary makes its records


def _dictionary(ctx, alphabet, hi, n=600, sc=(1, -1, -1)):
    w = synth.make_uniform_length_words(n, alphabet, 1.0, 0, hi, seed=alphabet + hi)
    return w, ctx.load_dictionary(w.codes, w.offsets, alphabet, sc)


@pytest.mark.parametrize("alphabet,hi,makes", [(5, 15, True), (40, 40, True), (128, 25, True), (129, 25, False)])
def test_records_after_many_pairs_and_equal_scores(oracle_mod, alphabet, hi, makes):
    import torch
    with nw.Context(0) as ctx:
        w, d = _dictionary(ctx, alphabet, hi)
        r = np.random.default_rng(1)
        i, j = r.integers(0, w.n, (2, 3000)).astype(np.uint32)
        bare = d.info()["device_bytes"]
        want = oracle_mod.score_pairs(w, i, j, (1, -1, -1))
        assert np.array_equal(d.score_pairs(i, j).astype(np.int32), want)
        assert d.info()["device_bytes"] == bare  # a short list does not repay them
        p = torch.randint(0, w.n, (MANY,), device="cuda", dtype=torch.int32)
        d.score_pairs(p, p.flip(0))
        more = d.info()["device_bytes"] - bare
        assert more >= 16 * w.n if makes else more == 0
        assert np.array_equal(d.score_pairs(i, j).astype(np.int32), want)


@pytest.mark.parametrize("warm", [10, MANY])
def test_pairs_in_a_captured_graph(warm):
    """A call on a stream that is being captured neither allocates nor waits, and replays after the records have gone
    or come."""
    import torch
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream), nw.Context(0, stream=stream.cuda_stream) as ctx:
        w, d = _dictionary(ctx, 20, 30)
        i = torch.randint(0, w.n, (5000,), device="cuda", dtype=torch.int32)
        j = torch.randint(0, w.n, (5000,), device="cuda", dtype=torch.int32)
        p = torch.randint(0, w.n, (warm,), device="cuda", dtype=torch.int32)
        d.score_pairs(p, p)
        out = torch.zeros(5000, device="cuda", dtype=torch.int16)
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            d.score_pairs(i, j, out=out, async_=True)
        p = torch.randint(0, w.n, (MANY,), device="cuda", dtype=torch.int32)
        d.score_pairs(p, p)
        graph.replay()
        stream.synchronize()
        assert torch.equal(out, d.score_pairs(i, j))


def _least(run):
    """The least budget, to 1 KiB, that run(budget) fits."""
    lo, hi = 0, 4 << 30
    while hi - lo > 1024:
        mid = (lo + hi) // 2
        try:
            run(mid)
            hi = mid
        except nw.NwError:
            lo = mid
    return hi


def test_records_give_way_under_a_memory_budget():
    """A call that fits the budget before a long pair list fits it after."""
    import torch
    n, k = 20_000, 10
    w = synth.make_uniform_length_words(n, 30, 1.0, 1, 15, seed=9)
    idx = torch.empty((n, k), dtype=torch.int32, device="cuda")
    score = torch.empty((n, k), dtype=torch.int16, device="cuda")
    p = torch.randint(0, n, (MANY,), device="cuda", dtype=torch.int32)

    def run(budget, pairs):
        with nw.Context(0, mem_budget_bytes=budget) as ctx:
            d = ctx.load_dictionary(w.codes, w.offsets, 30, (1, -1, -1))
            if pairs:
                bare = d.info()["device_bytes"]
                d.score_pairs(p, p.flip(0))
                assert d.info()["device_bytes"] >= bare + 16 * n  # (there was room)
            d.all_pairs_topk(k, idx, score, hist=False)

    run(_least(lambda budget: run(budget, False)), True)


def test_rescoring_takes_no_more_memory_than_without_records():
    """Queries and lists through the proposal fit the budget that they fit with a scoring that uses no records."""
    n, C, k = 20_000, 16, 5
    w = synth.make_uniform_length_words(n, 30, 1.0, 1, 15, seed=9)
    q = synth.make_uniform_length_words(2, 30, 1.0, 1, 15, seed=10)

    def run(budget, sc, lists):
        with nw.Context(0, mem_budget_bytes=budget) as ctx:
            d = ctx.load_dictionary(w.codes, w.offsets, 30, sc)
            model = nw.Model(ctx, 30, seed=1)
            return model.proposal_topk(d, C, k)[:2] if lists else model.query(d, q.codes, q.offsets, C, k)

    for lists in (False, True):
        budget = _least(lambda b: run(b, (4, -1, -1), lists)) + (64 << 10)
        got, want = run(budget, (1, -1, -1), lists), run(0, (1, -1, -1), lists)
        assert all(np.array_equal(x, y) for x, y in zip(got, want))
