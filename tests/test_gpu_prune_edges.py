"""The prune kernels where their cuts fall, against the oracle edge for edge: list
lengths at the edges of the 64- and 128-row kernels and past them (batches of 32
on the general path, rows staged in shared memory or not), rows of one and of
several 128-dimension slices, many targets, R at the edges of a batch, both
variants, and data with equal and nearly equal distances."""
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


def _rows(dtype, n, d, seed, ties):
    rng = np.random.default_rng(seed)
    if dtype == "u8":
        return rng.integers(0, 3 if ties else 256, (n, d)).astype(np.uint8)
    X = rng.normal(size=(n, d)).astype(np.float32)
    if ties:  # repeated points, and points an ulp or so apart
        X[n // 3:2 * (n // 3)] = X[:n // 3]
        X[2 * (n // 3):3 * (n // 3)] = X[:n // 3] * np.float32(1 + 2.0 ** -22)
    return X


def _lists(n, degrees, seed):
    """Node i has degrees[i] distinct neighbours (0 past the end)."""
    rng = np.random.default_rng(seed)
    rows = [rng.permutation(n - 1)[:k] for k in degrees]
    rows = [np.where(r >= i, r + 1, r) for i, r in enumerate(rows)]
    ptr = np.zeros(n + 1, np.int64)
    ptr[1:len(rows) + 1] = np.cumsum([len(r) for r in rows])
    ptr[len(rows) + 1:] = ptr[len(rows)]
    return ptr, np.concatenate(rows).astype(np.int32)


def _check(ctx, X, ptr, col, targets, variant):
    g = rp.rp_load_graph(ctx, X, ptr, col, start=0)
    code = rp.RP_UNSORTED if variant == "unsorted" else rp.RP_SORTED
    outs = rp.rp_tune_batch(ctx, g, [a for a, _ in targets], [r for _, r in targets], code)
    for t, (alpha, R) in zip(outs, targets):
        got = rp.rp_graph_export(ctx, t)
        ref = oracle.rp_tune(X, ptr, col, alpha, R, variant=variant)
        assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1]), (alpha, R)
        rp.rp_graph_free(ctx, t)
    rp.rp_graph_free(ctx, g)


SWEEP = [(1.0, 64), (1.05, 3), (1.1, 64), (1.2, rp.RP_R_INF), (1.0, 1)]


@pytest.mark.parametrize("variant,ties", [("sorted", False), ("sorted", True), ("unsorted", True)])
@pytest.mark.parametrize("dtype,d", [("u8", 17), ("u8", 128), ("u8", 200), ("f32", 3), ("f32", 32), ("f32", 96),
                                     ("f32", 128), ("f32", 129), ("f32", 300)])
def test_short_lists(ctx, dtype, d, variant, ties):
    n = 300
    degrees = [0, 1, 2, 3, 4, 5, 15, 16, 17, 31, 32, 33, 47, 48, 49, 62, 63, 64, 65, 66, 80, 96, 97, 112, 126, 127, 128] * 3
    ptr, col = _lists(n, degrees, d)
    _check(ctx, _rows(dtype, n, d, d, ties), ptr, col, SWEEP, variant)


@pytest.mark.parametrize("d", [96, 260])
def test_sixteen_alphas(ctx, d):
    ptr, col = _lists(300, [64, 63, 10, 128, 100] * 12, d)
    targets = [(1.0 + 0.012 * i, 64 if i % 2 else 128) for i in range(16)]
    _check(ctx, _rows("f32", 300, d, 5, True), ptr, col, [(round(a, 3), r) for a, r in targets], "sorted")


@pytest.mark.parametrize("variant,ties", [("sorted", False), ("sorted", True), ("unsorted", False)])
@pytest.mark.parametrize("dtype,d", [("u8", 128), ("u8", 300), ("f32", 20), ("f32", 96), ("f32", 500), ("f32", 1500),
                                     ("f32", 3000)])
def test_long_lists(ctx, dtype, d, variant, ties):
    # 20 floats: every kept row fits in shared memory; 500: one CTA per SM; 1500: one
    # batch of rows; 3000: none
    n = 620
    degrees = [129, 160, 161, 255, 256, 257, 300, 512, 513, 600, 64, 0, 191, 192, 193]
    ptr, col = _lists(n, degrees, d)
    targets = [(1.0, rp.RP_R_INF), (1.1, 64), (1.2, 31), (1.2, 32), (1.2, 33), (1.5, 1)]
    _check(ctx, _rows(dtype, n, d, d + 1, ties), ptr, col, targets, variant)
