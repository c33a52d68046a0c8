"""Items of the tensor-core term kernel of every kind in one launch.

The kernel's loader warps prepare an item while the one before it runs: states of
up to 2^10 amplitudes through the load area (when the layouts leave room for it),
2^11 from global memory by registers, 2^12 and fewer than 8 amplitudes in place,
states in HBM by blocks of 2,048 (X-masks inside a block) or by gathers.  A batch
mixes them all, with one tile and pairs of tiles, so every kind follows every other
in the queue; single calls that return beta and delta take the shared memory that
the load area would need.  Bounds: the FP32 ones of the other parity tests."""
import numpy as np
import pytest
import torch

from oracle import terms as oterms
from paper_2604_14435_gb300 import workloads as wl

from test_gpu_terms import check as check_terms
from test_gpu_terms import gpu_cost_grad, random_problem
from test_gpu_tuning import check, run

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 2), (2, 1, 5), (3, 2, 8), (4, 1, 17), (5, 1, 70), (7, 1, 64), (10, 1, 66), (11, 0, 65), (12, 0, 9),
          (13, 0, 66), (14, 0, 5)]


@pytest.mark.parametrize("layout", [0, 1, 2])
@pytest.mark.parametrize("far", [True, False])
def test_every_kind_of_item_in_one_launch(dv, layout, far):
    rng = np.random.default_rng(31)
    probs = []
    for n, d, L in SHAPES:
        coef, xs, zs, b = random_problem(rng, n, L)
        if not far:
            xs = np.asarray(xs) & 2047  # states in HBM: every item inside its block
        probs.append((n, d, L, wl.random_angles(n * (d + 1), int(rng.integers(1 << 30))), coef, xs, zs, b))
    refs = [oterms.cost_grad(n, d, a, b, c, x, z) for n, d, L, a, c, x, z, b in probs]
    check(probs, refs, *run(dv, probs, 1, layout))


@pytest.mark.parametrize("n,L", [(2, 5), (3, 8), (8, 65), (9, 64), (10, 65), (11, 64), (12, 20)])
def test_readout_with_and_without_room_to_load_ahead(dv, ctx, n, L):
    rng = np.random.default_rng(1000 * n + L)
    coef, xs, zs, b = random_problem(rng, n, L)
    alpha = wl.random_angles(2 * n, n)
    ref = oterms.cost_grad(n, 1, alpha, b, coef, xs, zs)
    check_terms(gpu_cost_grad(dv, ctx, n, 1, alpha, b, coef, xs, zs, dv.DVQLS_FP32_TC), ref, dv.DVQLS_FP32_TC)
