"""The two-sweep path of nw_dot_topk against plain integer arithmetic, on sampled rows: at the smallest size it takes, at
ragged sizes of each group width, past the size where its first sweep takes half the columns, and with masses of ties
(which its id limit, or the candidate kernel behind it, has to settle by the lower index)."""
import numpy as np
import pytest

from paper_2509_01654_gb300 import nw

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2509_01654_gb300 import build
    build.build()
    with nw.Context(0) as c:
        yield c


def _rows(kind, n, seed):
    r = np.random.default_rng(seed)
    q = np.zeros((n, 64), np.int8)
    if kind == "spread":
        q[:, :63] = r.integers(-127, 128, (n, 63))
        bias = r.integers(-2 ** 23, 2 ** 23 + 1, n)
    elif kind == "duplicates":  # every row about 60 times, in no order
        q[:, :63] = r.integers(-30, 31, (max(2, n // 60), 63))[r.integers(0, max(2, n // 60), n)]
        bias = np.zeros(n)
    elif kind == "skewed":      # one row a third of the time
        q[:, :63] = np.where(r.random((n, 1)) < 0.33, 9, r.integers(-20, 21, (n, 63)))
        bias = np.zeros(n)
    else:                       # constant
        q[:, :63] = 1
        bias = np.zeros(n)
    return q, bias.astype(np.int32)


@pytest.mark.parametrize("kind", ["spread", "duplicates", "skewed", "constant"])
@pytest.mark.parametrize("n,C", [(2 * 33 * 32, 32), (2 * 33 * 32 + 1, 32), (8191, 32), (20_001, 100), (45_000, 256)])
@pytest.mark.parametrize("locality", [True, False])
def test_lists_equal_integer_arithmetic(ctx, kind, n, C, locality):
    _check(ctx, kind, n, C, locality)


def test_first_sweep_over_half_of_the_columns(ctx):
    _check(ctx, "duplicates", (1 << 18) + 77, 40, True)


def _check(ctx, kind, n, C, locality):
    q, bias = _rows(kind, n, n + C)
    idx, val = nw.dot_topk(ctx, q, C, bias=bias, locality=locality)
    cols = q.astype(np.float64)
    for i in np.unique(np.r_[0, 1, n - 1, np.random.default_rng(1).integers(0, n, 24)]):
        v = (cols @ cols[i]).astype(np.int64) + bias
        v[i] = -(1 << 40)  # the row itself
        want = np.lexsort((np.arange(n), -v))[:C]
        assert np.array_equal(idx[i], want), (kind, n, C, i)
        assert np.array_equal(val[i], v[want])


def _ordered(kind, n, seed):
    """Rows in clusters of about 50, in no order, or clusters adjacent, or duplicates of one row in every third."""
    r = np.random.default_rng(seed)
    pick = r.integers(0, max(2, n // 50), n)
    if kind != "random":
        pick = np.sort(pick)
    centres = r.normal(0, 18, (max(2, n // 50), 63)) * np.linspace(2.2, 0.4, 63)
    q = np.zeros((n, 64), np.int8)
    q[:, :63] = np.clip(np.rint(centres[pick] + r.normal(0, 7, (n, 63))), -127, 127)
    if kind == "copies":
        q[::3] = q[n // 2]
    return q, (-0.4 * (q.astype(np.float32) ** 2).sum(1)).astype(np.int32)


@pytest.mark.parametrize("kind", ["clustered", "copies"])
@pytest.mark.parametrize("n,C", [(9000, 64), (30_011, 256), (60_000, 512)])
@pytest.mark.parametrize("locality", [True, False])
def test_ordered_rows(ctx, kind, n, C, locality):
    q, bias = _ordered(kind, n, n)
    idx, val = nw.dot_topk(ctx, q, C, bias=bias, locality=locality)
    cols = q.astype(np.float64)
    for i in np.r_[0, 3, n // 2, n - 1, np.random.default_rng(2).integers(0, n, 12)]:
        v = (cols @ cols[i]).astype(np.int64) + bias
        v[i] = -(1 << 40)
        want = np.lexsort((np.arange(n), -v))[:C]
        assert np.array_equal(idx[i], want) and np.array_equal(val[i], v[want])


@pytest.mark.parametrize("n,C", [(40_000, 100), (100_000, 256)])
def test_time_does_not_depend_on_the_row_order(ctx, n, C):
    """Clustered rows cost what rows in no order cost (they cost 2.5 to 3 times as much when the candidate kernel had
    to redo them)."""
    import time

    import torch
    took = {}
    for kind in ("random", "clustered"):
        q, bias = (torch.from_numpy(x).cuda() for x in _ordered(kind, n, 3))
        times = []
        for _ in range(7):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            nw.dot_topk(ctx, q, C, bias=bias)
            times.append(time.perf_counter() - t0)
        took[kind] = np.median(times[2:])
    assert took["clustered"] < 1.6 * took["random"], took
