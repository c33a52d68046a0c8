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
