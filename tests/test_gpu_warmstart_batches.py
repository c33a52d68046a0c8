"""Warm-start network: small batches, and derivatives near the ends of FP32."""
import numpy as np
import pytest

from oracle import mlp as omlp

from test_gpu_warmstart import random_net

pytestmark = pytest.mark.gpu


# Inference of few rows takes tiles of 16 rows, of many rows tiles of 64; a row's sums run
# over k in order in both, so the results are the same bits.
@pytest.mark.parametrize("I,H,O,B", [(1, 1, 1, 1), (7, 33, 50, 15), (7, 256, 50, 16), (7, 256, 50, 17), (12, 300, 70, 100)])
def test_small_batches_match_rows_of_a_large_one(dv, ctx, I, H, O, B):
    p, X, _, _ = random_net(I, H, O, 16384, B)
    ws = dv.dvqls_ws_create(ctx, I, H, O, p)
    try:
        full, y = np.zeros((16384, O), np.float32), np.zeros((B, O), np.float32)
        dv.dvqls_ws_infer(ws, 16384, X, full)
        ref, _ = omlp.forward(p.astype(np.float64), X[:B], I, H, O)
        for first in (0, 64, 16384 - B):
            dv.dvqls_ws_infer(ws, B, np.ascontiguousarray(X[first:first + B]), y)
            assert np.array_equal(y, full[first:first + B])
        dv.dvqls_ws_infer(ws, B, X[:B].copy(), y)
        assert np.abs(y - ref).max() <= 1e-4 * max(1.0, np.abs(ref).max())
    finally:
        dv.dvqls_ws_destroy(ws)


@pytest.mark.parametrize("scale", [1e37, 1e-30])
@pytest.mark.parametrize("O,B", [(50, 2000), (3, 130)])
def test_derivatives_of_large_and_small_errors(dv, ctx, O, B, scale):
    """The gradient is a mean over the batch: it fits where a sum over the batch would not.
    Bound as in the other gradient tests (FP32 sums of at most 2,000 terms), of the largest entry."""
    I, H = 7, 33
    p, X, T, M = random_net(I, H, O, B, O)
    p[-(O * H + O):] *= np.float32(1e-3)  # the network's own output is small beside the targets
    T = (T + np.float32(3.0)).astype(np.float32)
    T *= np.float32(scale)
    if scale < 1.0:
        p[-(O * H + O):] = 0.0  # y = 0: the error is the target
    ws = dv.dvqls_ws_create(ctx, I, H, O, p)
    try:
        g = np.zeros(p.size, np.float32)
        dv.dvqls_ws_grad(ws, B, X, T, M, g)
        g_ref = omlp.grad(p.astype(np.float64), X, T.astype(np.float64), M, I, H, O)
        assert np.isfinite(g).all()
        assert np.abs(g - g_ref).max() <= 1e-4 * np.abs(g_ref).max()
    finally:
        dv.dvqls_ws_destroy(ws)
