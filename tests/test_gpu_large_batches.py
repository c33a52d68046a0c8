"""Batches of more than 65,535 instances (a grid's y extent) through the kernels
that take one row of blocks per instance: ||b||^2 by blocks and the fold of many
partial sums.

All small instances are one system, so every cost is the single call's, bit for bit
(the same split, the same order of sums)."""
import numpy as np
import pytest
import torch

from paper_2604_14435_gb300 import workloads as wl

from test_gpu_terms import cvec, random_problem

pytestmark = pytest.mark.gpu

COUNT = 65536 + 9


def system(dv, n, L, seed):
    rng = np.random.default_rng(seed)
    coef, xs, zs, b = random_problem(rng, n, L)
    t = [torch.tensor(v, device="cuda")
         for v in (cvec(coef), xs.view(np.int32), zs.view(np.int32), wl.random_angles(n, seed), cvec(b))]
    return (dv.make_ansatz(n, 0), dv.make_lcu(L, t[0], t[1], t[2]), t[3], t[4]), t


def test_fold_of_a_large_batch(dv, ctx):
    n = 9  # 10 flavours x 8 parts of the amplitudes: folded
    item, keep = system(dv, n, 2, 1)
    dv.dvqls_set_tuning(ctx, 8, 0)
    try:
        one, all_ = (torch.zeros(m, device="cuda", dtype=torch.float64) for m in (1, COUNT))
        dv.dvqls_local_cost_grad_batched(ctx, dv.make_instances([item]), dv.DVQLS_FP32, one, None)
        dv.dvqls_local_cost_grad_batched(ctx, dv.make_instances([item] * COUNT), dv.DVQLS_FP32, all_, None)
        dv.dvqls_sync(ctx)
        assert np.isfinite(one.item()) and bool((all_ == one).all())
    finally:
        dv.dvqls_set_tuning(ctx, 0, -1)


@pytest.mark.parametrize("prec", [0, 1])
def test_state_in_hbm_in_a_large_batch(dv, ctx, prec):
    big, keep_big = system(dv, 17, 3, 2)  # 64 parts: folded
    small, keep = system(dv, 1, 1, 3)
    dv.dvqls_set_tuning(ctx, 1, 0)
    try:
        f64 = dict(device="cuda", dtype=torch.float64)
        two_c, two_g = torch.zeros(2, **f64), torch.zeros(18, **f64)
        dv.dvqls_cost_grad_batched(ctx, dv.make_instances([small, big]), prec, two_c, two_g)
        costs, grads = torch.zeros(COUNT, **f64), torch.zeros(COUNT - 1 + 17, **f64)
        dv.dvqls_cost_grad_batched(ctx, dv.make_instances([small] * (COUNT - 1) + [big]), prec, costs, grads)
        dv.dvqls_sync(ctx)
        assert bool((costs[:-1] == two_c[0]).all()) and bool((grads[:-17] == two_g[0]).all())
        assert costs[-1] == two_c[1] and bool((grads[-17:] == two_g[1:]).all())
        assert np.isfinite(two_g.cpu().numpy()).all()
    finally:
        dv.dvqls_set_tuning(ctx, 0, -1)
