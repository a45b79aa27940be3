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
