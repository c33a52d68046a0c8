"""FP64 evaluations whose term classes are dealt to several CTAs per state: few states,
and masks that put nearly every pair in a class of its own.

Tolerances as the other FP64 paths (1e-12, beta and delta 1e-13); the parts' sums
differ in their order alone from those of a batch that fills the GPU, which deals
nothing out (1e-13)."""
import numpy as np
import pytest

from oracle import terms as oterms
from paper_2604_14435_gb300 import workloads as wl

from test_gpu_terms import cvec, random_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,L,complex_b", [(6, 0, 64, True), (7, 0, 20, False), (8, 1, 64, True), (9, 0, 63, False),
                                             (10, 0, 64, True), (10, 0, 11, True), (10, 2, 64, False)])
def test_few_states_many_classes(dv, ctx, n, d, L, complex_b):
    rng = np.random.default_rng(100 * n + L)
    coef, xs, zs, b = random_problem(rng, n, L, complex_b)
    P = n * (d + 1)
    alpha, an = wl.random_angles(P, n + d), dv.make_ansatz(n, d)
    ref = oterms.cost_grad(n, d, alpha, b, coef, xs, zs)
    c, bb = cvec(coef), cvec(b)
    lcu = dv.make_lcu(L, c, xs, zs)

    def near(got, want, tol):
        assert np.all(np.abs(got - want) <= tol * np.maximum(1.0, np.abs(want)))

    for grad in (False, True):  # one state, or 2 P + 1
        cost, g, beta, delta = np.zeros(1), np.zeros(P), np.zeros(2 * L * L), np.zeros(2 * L)
        if grad:
            dv.dvqls_cost_grad(ctx, an, alpha, lcu, bb, dv.DVQLS_FP64, cost, g, beta, delta)
            near(g, ref["grad"], 1e-12)
        else:
            dv.dvqls_cost(ctx, an, alpha, lcu, bb, dv.DVQLS_FP64, cost, beta, delta)
        near(cost, np.array([ref["cost"]]), 1e-12)
        near(beta.view(np.complex128).reshape(L, L), ref["beta"], 1e-13)
        near(delta.view(np.complex128), ref["delta"], 1e-13)
    part = np.zeros(4 * (2 * P + 1))  # one shift alone
    dv.dvqls_cost_grad_partials(ctx, an, alpha, lcu, bb, dv.DVQLS_FP64, P, P + 1, part)
    many = dv.make_instances([(an, lcu, alpha, bb)] * 64)
    costs, grads = np.zeros(64), np.zeros(64 * P)
    dv.dvqls_cost_grad_batched(ctx, many, dv.DVQLS_FP64, costs, grads)
    near(costs, np.full(64, cost[0]), 1e-13)
    near(grads.reshape(64, P), np.tile(g, (64, 1)), 1e-13)
    full = np.zeros(4 * (2 * P + 1))
    dv.dvqls_cost_grad_partials(ctx, an, alpha, lcu, bb, dv.DVQLS_FP64, 0, 2 * P + 1, full)
    near(part.reshape(-1, 4)[P], full.reshape(-1, 4)[P], 1e-13)
    assert not part.reshape(-1, 4)[:P].any() and not part.reshape(-1, 4)[P + 1:].any()


@pytest.mark.parametrize("n,d,L", [(4, 0, 64), (8, 0, 64), (10, 0, 64), (10, 1, 12)])
def test_local_cost(dv, ctx, n, d, L):
    rng = np.random.default_rng(n + L)
    coef, xs, zs, _ = random_problem(rng, n, L)
    P = n * (d + 1)
    alpha, an = wl.random_angles(P, 5), dv.make_ansatz(n, d)
    c = cvec(coef)
    lcu = dv.make_lcu(L, c, xs, zs)
    one, cost, g = np.zeros(1), np.zeros(1), np.zeros(P)
    dv.dvqls_local_cost_grad(ctx, an, alpha, lcu, dv.DVQLS_FP64, one)
    dv.dvqls_local_cost_grad(ctx, an, alpha, lcu, dv.DVQLS_FP64, cost, g)
    costs, grads = np.zeros(80), np.zeros(80 * P)
    dv.dvqls_local_cost_grad_batched(ctx, dv.make_instances([(an, lcu, alpha, c)] * 80), dv.DVQLS_FP64, costs, grads)
    ref = oterms.local_cost_grad(n, d, alpha, coef, xs, zs)
    tol = 1e-12 * max(1.0, abs(ref["cost"]))
    assert abs(one[0] - ref["cost"]) <= tol and abs(cost[0] - ref["cost"]) <= tol
    assert np.all(np.abs(g - ref["grad"]) <= 1e-12 * np.maximum(1.0, np.abs(ref["grad"])))
    assert np.abs(costs - cost[0]).max() <= 1e-13 and np.abs(grads.reshape(80, P) - g).max() <= 1e-13
