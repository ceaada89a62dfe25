"""The start vertex where it turns on the last bit of a column's mean, for columns
that make the library's mean kernel take each of its ways to add a block of 2,048
rows (one binade, exact, 256 and 64 rows at a time, row by row) and for row counts
that are no whole number of blocks.

One column decides, as in ``medoid_cases``: rows 0 and 1 hold adjacent float32
values a < b, the rows after them the kind's values, and the last few steer the
index-order binary64 sum to n mid + k ulp, mid = (a + b) / 2.  The mean is then mid
for k = 0 (a tie, row 0), and above or below it for k = 1 or -1: n mid is exact and
an ulp of it is more than half an ulp of mid times n."""
import numpy as np
import pytest

import oracle
from medoid_cases import sequential_sum

rp = pytest.importorskip("paper_2602_08097_gb300")
KINDS = ["one binade", "signs", "whole", "ties", "wide", "subnormal"]
SIZES = [500, 2047, 2049, 4096, 6147]


def _values(kind, m, mid, rng):
    if kind == "one binade":  # the sum grows slowly; few changes of binade
        return mid * (1.0 + 0.2 * rng.random(m))
    if kind == "signs":  # the sum stays near zero and changes sign and binade all the time
        return rng.normal(size=m)
    if kind == "whole":  # every partial sum is exact
        return rng.integers(-1000, 1000, m)
    if kind == "ties":  # halves of the sum's last place among larger values
        return np.where(rng.random(m) < 0.2, 2.0 ** -rng.integers(40, 50, m), rng.integers(1, 64, m))
    if kind == "wide":
        return rng.normal(size=m) * 2.0 ** rng.integers(-100, 40, m)
    return np.where(rng.random(m) < 0.5, rng.normal(size=m) * 1e-41, 0.0)


def _case(kind, n, k):
    rng = np.random.default_rng(n + KINDS.index(kind))
    a = np.float32(0.0390625 + float(rng.random()) * 1e-3)
    b = np.nextafter(a, np.float32(1.0))
    mid = (float(a) + float(b)) / 2.0
    target = n * mid + k * float(np.spacing(n * mid))
    column = np.zeros(n, dtype=np.float32)
    m = n - 12
    column[:2] = a, b
    column[2:m] = _values(kind, m - 2, mid, rng)
    s = sequential_sum(column[:m])
    while s != target:
        column[m] = np.float32(target - s)
        s += float(column[m])
        m += 1  # at most twelve: each takes the 24 leading bits of what is left
    assert sequential_sum(column) == target
    X = np.full((n, 5), 0.5, dtype=np.float32)
    X[:, 3] = column
    return X, 1 if k > 0 else 0


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("kind", KINDS)
def test_the_oracle_agrees(kind, n):
    for k in (-1, 0, 1):
        X, expect = _case(kind, n, k)
        assert oracle.medoid(X) == expect


@pytest.mark.gpu
@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("kind", KINDS)
def test_the_start_vertex_is_the_nearest_to_the_exact_mean(kind, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_08097_gb300 import build as b
    b.build()
    ctx = rp.rp_create(0)
    try:
        for k in (-1, 0, 1):
            X, expect = _case(kind, n, k)
            g = rp.rp_load_graph(ctx, X)
            assert rp.rp_graph_info(ctx, g)["start"] == expect, k
            rp.rp_graph_free(ctx, g)
    finally:
        rp.rp_destroy(ctx)
