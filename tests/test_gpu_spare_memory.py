"""Buffers that a finished call leaves with its context: later calls of other
sizes return what a fresh context returns, and the spare memory never makes a
call exceed the budget that the call alone fits."""
import numpy as np
import pytest

from paper_2509_01654_gb300 import nw, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("budget", [0, 300 << 20])
def test_calls_of_changing_size_equal_a_fresh_context(budget):
    rng = np.random.default_rng(5)
    shared = nw.Context(0, mem_budget_bytes=budget)
    w = synth.make_uniform_length_words(900, 30, 1.0, 0, 20, seed=3)
    d = shared.load_dictionary(w.codes, w.offsets, 30, (1, -1, -1))
    # 2,000 rows take 262 MB of candidate buffers, 1,000 rows 66 MB
    for n in (2000, 1000, 2000, 37, 1990, 1000):
        q = rng.integers(-128, 128, (n, 64), dtype=np.int8)
        b = rng.integers(-5000, 5000, n, dtype=np.int32)
        got = nw.dot_topk(shared, q, 32, bias=b)
        fresh = nw.Context(0)
        want = nw.dot_topk(fresh, q, 32, bias=b)
        assert all(np.array_equal(x, y) for x, y in zip(got, want)), n
        qs = synth.make_uniform_length_words(1 + n % 41, 30, 1.0, 0, 30, seed=n)
        got = d.query(qs.codes, qs.offsets, 7)
        want = fresh.load_dictionary(w.codes, w.offsets, 30, (1, -1, -1)).query(qs.codes, qs.offsets, 7)
        assert all(np.array_equal(x, y) for x, y in zip(got, want)), n
        fresh.close()
    if budget:  # a call that does not fit by itself is still refused, and leaves the context usable
        q = rng.integers(-128, 128, (4000, 64), dtype=np.int8)
        with pytest.raises(nw.NwError):
            nw.dot_topk(shared, q, 32)
        assert nw.dot_topk(shared, q[:50], 8)[0].shape == (50, 8)
    shared.close()


def test_another_context_can_have_the_memory():
    """What one context keeps for its next call does not refuse another's, and a program can have it back."""
    import torch
    q = np.random.default_rng(1).integers(-128, 128, (20_000, 64), dtype=np.int8)
    with nw.Context(0) as a, nw.Context(0) as b:
        want = nw.dot_topk(a, q, 32)  # leaves more than a gigabyte of buffers
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        hog = torch.empty(free - (1 << 30), dtype=torch.uint8, device="cuda")
        got = nw.dot_topk(b, q, 32)
        assert all(np.array_equal(x, y) for x, y in zip(got, want))
        held = torch.cuda.mem_get_info()[0]
        b.trim()
        assert torch.cuda.mem_get_info()[0] - held > 1 << 30
        del hog
        torch.cuda.empty_cache()
        got = nw.dot_topk(a, q, 32)
        assert all(np.array_equal(x, y) for x, y in zip(got, want))


def test_two_contexts_in_turn_keep_their_speed():
    """Calls of two contexts, one after the other, do not allocate each time."""
    import time

    import torch
    q = torch.randint(-128, 128, (60_000, 64), dtype=torch.int8, device="cuda")  # about 2 GB of buffers a call
    with nw.Context(0) as a, nw.Context(0) as b:
        took = {}
        for name, contexts in (("one", [a, a]), ("two", [a, b])):
            times = []
            for _ in range(8):
                for c in contexts:
                    torch.cuda.synchronize()
                    t0 = time.perf_counter()
                    nw.dot_topk(c, q, 64)
                    times.append(time.perf_counter() - t0)
            took[name] = np.median(times[4:])
    assert took["two"] < 1.3 * took["one"], took


LAST = """
import torch
from paper_2509_01654_gb300 import nw
q = torch.randint(-128, 128, (20_000, 64), dtype=torch.int8, device="cuda")
for _ in range(2):
    a, b = nw.Context(0), nw.Context(0)
    want = nw.dot_topk(a, q, 32)
    a.close()
    got = nw.dot_topk(b, q, 32)  # with the blocks that a left
    assert all(torch.equal(x, y) for x, y in zip(got, want))
    before = torch.cuda.mem_get_info()[0]
    b.close()
    assert torch.cuda.mem_get_info()[0] - before > 1 << 30
"""


def test_the_last_context_gives_the_memory_back():
    """In a process of its own: no other context may be alive."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", LAST], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
