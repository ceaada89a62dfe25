"""Every form of the search kernel against the oracle's lists: the list in
registers (L up to 256, 4 or 8 slots) and in shared memory, one warp or a team
per query (by the number of queries), every way lanes share a row (by its
length), lists of more than one 64-neighbour chunk, and data full of equal
distances."""
import numpy as np
import pytest

import datagen
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


def _data(dtype, d, n, nq, seed, ties):
    rng = np.random.default_rng(seed)
    if dtype == "u8":
        hi = 2 if ties else 256
        return rng.integers(0, hi, (n, d)).astype(np.uint8), rng.integers(0, hi, (nq, d)).astype(np.uint8)
    X = rng.normal(size=(n, d)).astype(np.float32)
    if ties:
        X[n // 2:] = X[:n - n // 2]  # every point twice: equal distances, ordered by id
    return X, rng.normal(size=(nq, d)).astype(np.float32)


@pytest.mark.parametrize("ties", [False, True])
@pytest.mark.parametrize("dtype,d", [("u8", 16), ("u8", 128), ("u8", 200), ("u8", 384), ("u8", 500),
                                     ("f32", 4), ("f32", 64), ("f32", 96), ("f32", 100), ("f32", 256), ("f32", 300)])
def test_search_forms_match_oracle(ctx, dtype, d, ties):
    n, most = 1200, 1300
    X, Q = _data(dtype, d, n, most, d, ties)
    row_ptr, col = datagen.random_graph(n, 0, 150, seed=d)
    g = rp.rp_load_graph(ctx, X, row_ptr, col, start=7)
    row_ptr, col = rp.rp_graph_export(ctx, g)  # cleaned
    chunks = (X.shape[1] * X.itemsize + 127) // 128 * 8
    lanes = 4 if chunks <= 24 else 8 if chunks <= 64 else 32
    rtol = ((chunks + lanes - 1) // lanes + 9) * 2.0 ** -24  # the roundings of a distance's sum
    for L, k, nq in [(1, 1, 5), (32, 32, 600), (33, 10, 3), (100, 100, 1300), (128, 128, 600), (129, 1, 1300),
                     (256, 256, 7), (257, 257, 40)]:
        ids, dists = rp.rp_search(ctx, g, Q[:nq], L, k)
        ref, refd, _ = oracle.greedy_search(X, row_ptr, col, 7, Q[:nq], L, k)
        assert np.array_equal(ids, ref), (L, k, nq)
        if dtype == "u8":
            assert np.array_equal(dists.astype(np.float64), refd)
        else:
            np.testing.assert_allclose(dists, refd, rtol=rtol)
    # a query's result does not depend on the launch it is part of
    q_L = np.resize(np.array([40, 100, 256, 300], np.int32), 64)
    ids, dists = rp.rp_search_multi(ctx, [g], np.zeros(64, np.int32), q_L, Q[:64], 40)
    for L in (40, 100, 256, 300):
        one, oned = rp.rp_search(ctx, g, np.ascontiguousarray(Q[:64][q_L == L]), L, 40)
        assert np.array_equal(ids[q_L == L], one) and np.array_equal(dists[q_L == L], oned)
    rp.rp_graph_free(ctx, g)


@pytest.mark.parametrize("nq", [3, 600, 1300])
def test_queries_that_hold_no_numbers_return(ctx, nq):
    X, Q = _data("f32", 96, 800, nq, 1, False)
    Q[::3] = np.nan
    Q[1::3, 5] = np.inf
    row_ptr, col = datagen.random_graph(800, 5, 40, seed=3)
    g = rp.rp_load_graph(ctx, X, row_ptr, col, start=0)
    ids, _ = rp.rp_search(ctx, g, Q, 64, 10)
    assert ((ids >= -1) & (ids < 800)).all()
    row_ptr, col = rp.rp_graph_export(ctx, g)
    ref, _, _ = oracle.greedy_search(X, row_ptr, col, 0, Q[2::3], 64, 10)
    assert np.array_equal(ids[2::3], ref)
    rp.rp_graph_free(ctx, g)


@pytest.mark.parametrize("nq", [16, 20000])
@pytest.mark.parametrize("dtype,d", [("u8", 128), ("f32", 32), ("f32", 24)])
def test_results_may_lie_over_the_queries(ctx, dtype, d, nq):
    # ids over the second half of the queries, distances over the first: the ids of
    # the first queries lie over rows that are searched much later
    torch = pytest.importorskip("torch")
    X, Q = _data(dtype, d, 500, nq, 2, False)
    row_ptr, col = datagen.random_graph(500, 5, 40, seed=3)
    g = rp.rp_load_graph(ctx, X, row_ptr, col, start=0)
    k = Q.nbytes // nq // 8
    q = torch.from_numpy(Q).cuda()
    ref, refd = rp.rp_search(ctx, g, q.clone(), 32, k)
    rp.rp_sync(ctx)
    words = q.view(torch.int32).flatten()
    ids, dists = words[nq * k:].view(nq, k), words[:nq * k].view(torch.float32).view(nq, k)
    torch.cuda.synchronize()
    rp.rp_search(ctx, g, q, 32, k, ids=ids, dists=dists)
    rp.rp_sync(ctx)
    assert torch.equal(ids, ref) and torch.equal(dists, refd)
    rp.rp_graph_free(ctx, g)
