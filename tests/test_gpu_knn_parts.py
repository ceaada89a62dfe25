"""The tensor-core kNN scan where its cuts fall: point sets and query sets at the
edges of 128-row tiles, fewer points than k, few queries (a query tile scanned in
many parts), more query tiles than one launch takes, and repeated rows (equal
distances across parts).  Against the CUDA-core scan, distances included, and the
oracle's lists."""
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


def _rows(dtype, n, d, rng, few=0):
    if dtype == "u8":
        X = rng.integers(0, 256, (n, d)).astype(np.uint8)
    else:
        X = rng.normal(size=(n, d)).astype(np.float32)
    return X[rng.integers(0, few, n)] if few else X


def _both(ctx, g, Q, k, nq=None):
    out = []
    for m in (rp.RP_KNN_TENSOR, rp.RP_KNN_CUDA_CORE):
        rp.rp_set_knn_method(ctx, m)
        out.append(rp.rp_knn(ctx, g, Q, k, nq=nq))
    rp.rp_set_knn_method(ctx, rp.RP_KNN_AUTO)
    return out


@pytest.mark.parametrize("dtype,d", [("u8", 5), ("u8", 128), ("f32", 16), ("f32", 96), ("f32", 113), ("f32", 128)])
@pytest.mark.parametrize("n,nq,k", [(1, 3, 4), (2, 2, 128), (127, 128, 10), (128, 1, 128), (129, 129, 1),
                                    (1153, 300, 100), (30001, 2, 128)])
def test_edges(ctx, dtype, d, n, nq, k):
    rng = np.random.default_rng(n * 131 + d)
    X, Q = _rows(dtype, n, d, rng), _rows(dtype, nq, d, rng)
    g = rp.rp_load_graph(ctx, X)
    (ti, td), (ci, cd) = _both(ctx, g, Q, k)
    assert np.array_equal(ti, ci) and np.array_equal(td, cd)
    kk = min(k, n)
    assert np.array_equal(ti[:, :kk], oracle.knn(X, kk, Q=Q)[0])
    (ti, td), (ci, cd) = _both(ctx, g, None, k, nq=min(n, nq))  # base points leave themselves out
    assert np.array_equal(ti, ci) and np.array_equal(td, cd)
    rp.rp_graph_free(ctx, g)


@pytest.mark.parametrize("dtype,d,few", [("u8", 32, 0), ("f32", 96, 0), ("u8", 64, 400)])
def test_more_query_tiles_than_a_launch_takes(ctx, dtype, d, few):
    rng = np.random.default_rng(7)
    X, Q = _rows(dtype, 3000, d, rng, few), _rows(dtype, 45_000, d, rng, few)
    g = rp.rp_load_graph(ctx, X)
    (ti, td), (ci, cd) = _both(ctx, g, Q, 20)
    assert np.array_equal(ti, ci) and np.array_equal(td, cd)
    rp.rp_graph_free(ctx, g)


@pytest.mark.parametrize("dtype,nq", [("u8", 25600), ("f32", 12800)])
def test_a_part_that_starts_among_repeated_rows(ctx, dtype, nq):
    # The near points lie in the first tile, the rest is one row over and over.  With
    # two thirds as many query tiles as CTAs, most queries' second part is scanned
    # before their first: it meets nothing but equal distances.
    rng = np.random.default_rng(11)
    n, d, k = 2048, 32, 10
    if dtype == "u8":
        X, Q = rng.integers(0, 20, (n, d)).astype(np.uint8), rng.integers(0, 20, (nq, d)).astype(np.uint8)
        X[128:] = 200
    else:
        X, Q = rng.normal(size=(n, d)).astype(np.float32), rng.normal(size=(nq, d)).astype(np.float32)
        X[128:] = 10.0
    g = rp.rp_load_graph(ctx, X)
    (ti, td), (ci, cd) = _both(ctx, g, Q, k)
    assert np.array_equal(ti, ci) and np.array_equal(td, cd)
    sel = np.arange(0, nq, 97)
    assert np.array_equal(ti[sel], oracle.knn(X, k, Q=np.ascontiguousarray(Q[sel]))[0])
    rp.rp_graph_free(ctx, g)


def test_more_equal_distances_than_the_scan_holds_are_refused(ctx):
    X = np.full((3000, 16), 7, np.uint8)
    X[:5] = 1
    g = rp.rp_load_graph(ctx, X)
    Q = np.full((3, 16), 8, np.uint8)
    rp.rp_set_knn_method(ctx, rp.RP_KNN_TENSOR)
    with pytest.raises(rp.RPError):
        rp.rp_knn(ctx, g, Q, 10)
    rp.rp_set_knn_method(ctx, rp.RP_KNN_AUTO)
    Q[:] = 0  # the context goes on: the five others are nearest
    assert np.array_equal(np.sort(rp.rp_knn(ctx, g, Q, 5)[0], axis=1), np.tile(np.arange(5), (3, 1)))
    rp.rp_graph_free(ctx, g)
