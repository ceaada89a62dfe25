"""The tensor-core kNN on float rows of unequal norms: the filter's error bound
grows with the square of a point's norm, and one row of large norm must not widen
the window of every other point.  Against the CUDA-core scan, distances included,
and the oracle's lists."""
import numpy as np
import pytest

import oracle

rp = pytest.importorskip("paper_2602_08097_gb300")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_08097_gb300 import build as b
    b.build()
    c = rp.rp_create(0)
    yield c
    rp.rp_destroy(c)


def _both(ctx, g, Q, k, nq=None):
    out = []
    for m in (rp.RP_KNN_TENSOR, rp.RP_KNN_CUDA_CORE):
        rp.rp_set_knn_method(ctx, m)
        out.append(rp.rp_knn(ctx, g, Q, k, nq=nq))
    rp.rp_set_knn_method(ctx, rp.RP_KNN_AUTO)
    return out


def _check(ctx, X, Q, k, base):
    """Queries Q and the first `base` points, both ways and against the oracle."""
    g = rp.rp_load_graph(ctx, X)
    for q, nq in ((Q, None), (None, base)):
        if q is None and base == 0:
            continue
        (ti, td), (ci, cd) = _both(ctx, g, q, k, nq=nq)
        assert np.array_equal(ti, ci) and np.array_equal(td, cd)
        sel = np.arange(0, len(ti), max(1, len(ti) // 40))
        ref = oracle.knn(X, k, Q=np.ascontiguousarray(q[sel])) if q is not None else oracle.knn(X, k, qid=sel)
        assert np.array_equal(ti[sel], ref[0])
    rp.rp_graph_free(ctx, g)


@pytest.mark.parametrize("k", [10, 100])
@pytest.mark.parametrize("times", [100, 300, 1000])
@pytest.mark.parametrize("at", ["start", "middle", "end"])
def test_one_row_of_large_norm(ctx, at, times, k):
    n = 20000
    X = np.random.default_rng(k).normal(size=(n, 96)).astype(np.float32)
    Q = np.random.default_rng(5).normal(size=(300, 96)).astype(np.float32)
    row = {"start": 0, "middle": n // 2, "end": n - 1}[at]
    X[row] *= np.float32(times)
    _check(ctx, X, Q, k, min(row, 3000))


@pytest.mark.parametrize("size", [0.0, 1e-12, 1e-9, 1e-6, 1e-3, 1e3])
def test_queries_far_smaller_or_larger_than_the_points(ctx, size):
    rng = np.random.default_rng(3)
    X = rng.normal(size=(20000, 48)).astype(np.float32)
    Q = (rng.normal(size=(200, 48)) * size).astype(np.float32)
    if size > 1:  # all points lie alike from afar: few enough of them to be told apart
        X = X[:300].copy()
    _check(ctx, X, Q, 10, 0)


@pytest.mark.parametrize("d,k", [(16, 10), (32, 100), (96, 128)])
def test_norms_over_many_sizes(ctx, d, k):
    rng = np.random.default_rng(d)
    X, Q = (rng.normal(size=(m, d)) * np.exp(rng.normal(size=(m, 1))) for m in (60000, 500))
    _check(ctx, X.astype(np.float32), Q.astype(np.float32), k, 0)
