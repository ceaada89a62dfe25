"""The float prune where the canonical decisions tie all the time: rows of zeros
and ones, rows many times over.  Row by row against the oracle in every degree
bucket, and the time of a launch stays within a multiple of the same launch over
rows without ties."""
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


def _rows(kind, n, d):
    rng = np.random.default_rng(d)
    if kind == "bits":
        return rng.integers(0, 2, (n, d)).astype(np.float32)
    if kind == "scaled bits":  # ties that single-precision sums of squares cannot hold exactly
        return (rng.integers(0, 2, (n, d)) * 0.1).astype(np.float32)
    X = rng.normal(size=(n, d)).astype(np.float32)
    return X[rng.integers(0, n // 50, n)] if kind == "rows" else X


TARGETS = ([1.0, 1.0, 1.05, 1.2], [16, 64, 32, 48])


@pytest.mark.parametrize("kind", ["bits", "scaled bits", "rows"])
@pytest.mark.parametrize("d", [17, 96, 300])
@pytest.mark.parametrize("lo,hi", [(0, 64), (65, 128), (129, 300)])
def test_rows_are_the_oracles(ctx, kind, d, lo, hi):
    n = 400
    X = _rows(kind, n, d)
    row_ptr, col = datagen.random_graph(n, lo, hi, seed=d + hi)
    g = rp.rp_load_graph(ctx, X, row_ptr, col, start=0)
    row_ptr, col = rp.rp_graph_export(ctx, g)
    for t, alpha, R in zip(rp.rp_tune_batch(ctx, g, *TARGETS), *TARGETS):
        got = rp.rp_graph_export(ctx, t)
        ref = oracle.rp_tune(X, row_ptr, col, alpha, R)
        assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1]), (alpha, R)
        rp.rp_graph_free(ctx, t)
    rp.rp_graph_free(ctx, g)


@pytest.mark.parametrize("kind,lo,hi,times", [("bits", 40, 64, 40), ("rows", 40, 64, 40), ("bits", 70, 128, 60),
                                              ("rows", 70, 128, 60), ("bits", 150, 300, 9)])
def test_time_stays_within_a_multiple(ctx, kind, lo, hi, times):
    ms = {}
    for k in (kind, "none"):
        X = _rows(k, 10000, 96)
        row_ptr, col = datagen.random_graph(10000, lo, hi, seed=1)
        g = rp.rp_load_graph(ctx, X, row_ptr, col, start=0)
        for _ in range(3):
            rp.rp_graph_free(ctx, rp.rp_tune(ctx, g, 1.0, 32))
            ms[k] = min(ms.get(k, np.inf), rp.rp_stats(ctx)["last_prune_ms"])
        rp.rp_graph_free(ctx, g)
    assert ms[kind] < times * ms["none"], ms
