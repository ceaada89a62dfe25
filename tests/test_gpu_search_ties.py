"""Float searches where distances tie all the time (rows of zeros and ones, rows
many times over) or are no numbers: lists of up to 256 entries give such queries to
the kernel of longer lists, which settles close decisions 32 at a time.  The lists
are the oracle's, and a list of 100 does not take longer than one of 300."""
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


def _data(kind, n, nq, d):
    rng = np.random.default_rng(d)
    if kind == "bits":
        return (rng.integers(0, 2, (m, d)).astype(np.float32) for m in (n, nq))
    few = rng.normal(size=(40, d)).astype(np.float32)
    X, Q = few[rng.integers(0, 40, n)], rng.normal(size=(nq, d)).astype(np.float32)
    if kind == "some":  # most queries of a launch meet no ties, some meet many
        X[: n // 2] = rng.normal(size=(n // 2, d))
        Q[::7] = few[rng.integers(0, 40, len(Q[::7]))]
    return X, Q


@pytest.mark.parametrize("kind,d", [("bits", 96), ("bits", 300), ("rows", 96), ("some", 32)])
@pytest.mark.parametrize("nq", [1, 300, 1300, 6000])  # teams of five and of three, one warp a query, several a warp
def test_lists_are_the_oracles(ctx, kind, d, nq):
    X, Q = _data(kind, 1500, nq, d)
    row_ptr, col = datagen.random_graph(1500, 0, 90, seed=d)
    g = rp.rp_load_graph(ctx, X, row_ptr, col, start=3)
    row_ptr, col = rp.rp_graph_export(ctx, g)
    sel = np.arange(0, nq, max(1, nq // 60))
    for L, k in [(20, 20), (100, 10), (256, 256)]:
        if nq > 2000 and L > 100:
            continue
        ids, dists = rp.rp_search(ctx, g, Q, L, k)
        ref, refd, _ = oracle.greedy_search(X, row_ptr, col, 3, np.ascontiguousarray(Q[sel]), L, k)
        assert np.array_equal(ids[sel], ref), (L, k)
        np.testing.assert_allclose(dists[sel], refd, rtol=2e-5)
    q_L = np.resize(np.array([30, 256, 100], np.int32), min(nq, 64))
    ids, _ = rp.rp_search_multi(ctx, [g], np.zeros(len(q_L), np.int32), q_L, Q[: len(q_L)], 30)
    for L in np.unique(q_L):
        ref, _, _ = oracle.greedy_search(X, row_ptr, col, 3, np.ascontiguousarray(Q[: len(q_L)][q_L == L]), int(L), 30)
        assert np.array_equal(ids[q_L == L], ref)
    rp.rp_graph_free(ctx, g)


@pytest.mark.parametrize("kind", ["bits", "rows", "nan"])
def test_a_list_of_100_takes_no_longer_than_one_of_300(ctx, kind):
    X, Q = _data("bits" if kind == "nan" else kind, 4000, 300, 96)
    if kind == "nan":
        Q[:] = np.nan
    row_ptr, col = datagen.random_graph(4000, 20, 40, seed=2)
    g = rp.rp_load_graph(ctx, X, row_ptr, col, start=3)
    ms = {}
    for L in (100, 300):
        for _ in range(3):
            rp.rp_search(ctx, g, Q, L, 10)
            ms[L] = min(ms.get(L, np.inf), rp.rp_stats(ctx)["last_search_ms"])
    assert ms[100] < 1.5 * ms[300], ms
    rp.rp_graph_free(ctx, g)


@pytest.mark.parametrize("all_rows", [False, True])
@pytest.mark.parametrize("n,d,nq", [(1500, 96, 1), (1500, 96, 300), (1500, 96, 6000), (1500, 960, 300), (200, 20000, 1)])
def test_sums_that_differ_in_their_order_alone(ctx, n, d, nq, all_rows):
    """Queries of equal numbers and rows that permute each other: the distances are
    equal but for the rounding of binary64 sums in index order.  A pair of such rows
    takes no second launch."""
    rng = np.random.default_rng(d)
    X = rng.normal(size=(n, d)).astype(np.float32)
    row_ptr, col = datagen.random_graph(n, 20, 60, seed=d)
    u, v = col[row_ptr[3] : row_ptr[3] + 2]  # both met by every search
    X[u] = 0.5 + 0.1 * X[u]
    for i in range(n) if all_rows else [v]:
        X[i] = rng.permutation(X[u])
    Q = np.repeat(rng.uniform(0.4, 0.6, (nq, 1)), d, axis=1).astype(np.float32)
    g = rp.rp_load_graph(ctx, X, row_ptr, col, start=3)
    row_ptr, col = rp.rp_graph_export(ctx, g)
    other = rng.normal(size=Q.shape).astype(np.float32)
    count = [rp.rp_stats(ctx)]
    for q in (other, Q):
        ids, dists = rp.rp_search(ctx, g, q, 50, 10)
        count.append(rp.rp_stats(ctx))
    launches = [b["kernel_launches"] - a["kernel_launches"] for a, b in zip(count, count[1:])]
    assert count[2]["fp64_search_dists"] - count[1]["fp64_search_dists"] >= 2 * nq
    if not all_rows:
        assert launches[1] == launches[0]
    sel = np.arange(0, nq, max(1, nq // 60))
    ref, refd, _ = oracle.greedy_search(X, row_ptr, col, 3, np.ascontiguousarray(Q[sel]), 50, 10)
    assert np.array_equal(ids[sel], ref)
    np.testing.assert_allclose(dists[sel], refd, rtol=2e-5)
    rp.rp_graph_free(ctx, g)


def test_a_vamana_build_over_ties_matches_the_oracle(ctx):
    X, _ = _data("bits", 600, 1, 24)
    g = rp.rp_load_graph(ctx, X)
    start = rp.rp_graph_info(ctx, g)["start"]
    v, cut = rp.rp_build_vamana(ctx, g, [1.0, 1.2], 24, 40)
    got = rp.rp_graph_export(ctx, v)
    ref_rp, ref_col, ref_cut = oracle.vamana(X, np.arange(600), [1.0, 1.2], 24, 40, 160, 12, start)
    assert cut == ref_cut and np.array_equal(got[0], ref_rp) and np.array_equal(got[1], ref_col)
    rp.rp_graph_free(ctx, v)
    rp.rp_graph_free(ctx, g)
