"""Row pointers of a loaded graph on either side of the one-CTA scan's steps (4,096
counts) and of its limit (16,384), exact against the degrees that went in."""
import numpy as np
import pytest

rp = pytest.importorskip("paper_2602_08097_gb300")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 4095, 4096, 4097, 16383, 16384, 16385, 20001])
def test_row_pointers(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_08097_gb300 import build as b
    b.build()
    rng = np.random.default_rng(n)
    deg = np.minimum(rng.integers(0, 9, n), n - 1)
    deg[-1] = min(37, n - 1)  # the largest, in the last place
    ptr = np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)
    row = np.repeat(np.arange(n), deg)
    col = ((row + 1 + np.arange(len(row)) - ptr[row]) % n).astype(np.int32)  # the next points: distinct, never itself
    X = rng.integers(0, 256, (n, 8)).astype(np.uint8)
    ctx = rp.rp_create(0)
    g = rp.rp_load_graph(ctx, X, ptr, col, start=0)
    got = rp.rp_graph_export(ctx, g)
    assert np.array_equal(got[0], ptr) and np.array_equal(got[1], col)
    assert rp.rp_graph_info(ctx, g)["max_degree"] == deg.max()
    rp.rp_graph_free(ctx, g)
    rp.rp_destroy(ctx)
