"""Rows that need padding go up packed, in chunks, and are padded on the device:
every byte of every chunk must arrive (host rows of odd and even lengths, more
than one 16 MB chunk), and rows of a whole number of 128 bytes in one copy."""
import numpy as np
import pytest

rp = pytest.importorskip("paper_2602_08097_gb300")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d,n", [(np.uint8, 1, 300), (np.uint8, 99, 400_000), (np.uint8, 100, 1000),
                                       (np.uint8, 128, 5000), (np.float32, 1, 70), (np.float32, 33, 300_000),
                                       (np.float32, 96, 3000)])
def test_uploaded_rows_are_the_callers(dtype, d, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_08097_gb300 import build as b
    b.build()
    rng = np.random.default_rng(d)
    X = rng.integers(0, 256, (n, d)).astype(dtype)
    ctx = rp.rp_create(0)
    try:
        # the same rows from the device (a pitched device copy) and from the host
        # give the same start vertex and the same neighbours of rows in every chunk
        host = rp.rp_load_graph(ctx, X)
        dev = rp.rp_load_graph(ctx, torch.from_numpy(X).cuda())
        assert rp.rp_graph_info(ctx, host)["start"] == rp.rp_graph_info(ctx, dev)["start"]
        Q = np.ascontiguousarray(X[np.linspace(0, n - 1, 24).astype(np.int64)])
        k = min(5, n)
        hi, hd = rp.rp_knn(ctx, host, Q, k)
        di, dd = rp.rp_knn(ctx, dev, torch.from_numpy(Q).cuda(), k)
        rp.rp_sync(ctx)
        assert np.array_equal(hi, di.cpu().numpy()) and np.array_equal(hd, dd.cpu().numpy())
        assert np.all(hd[:, 0] == 0)  # each query finds its own row
        want = ((X[hi].astype(np.int64) - Q[:, None, :].astype(np.int64)) ** 2).sum(2)
        assert np.array_equal(hd.astype(np.int64), want)
    finally:
        rp.rp_destroy(ctx)
