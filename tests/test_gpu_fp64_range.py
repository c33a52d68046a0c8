"""FP64 evaluations at the ends of the range of a double: large coefficients, and
right-hand sides whose norm is not finite."""
import numpy as np
import pytest
import torch

from paper_2604_14435_gb300 import workloads as wl

from test_gpu_terms import cvec, random_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,L", [(3, 8), (6, 20), (10, 64)])
@pytest.mark.parametrize("scale", [2.0 ** 490, 2.0 ** -490])  # |c|^2 near 1e295 and 1e-295
def test_large_and_small_coefficients(dv, ctx, n, L, scale):
    """The cost does not depend on the size of A; its sums are scaled by an exact power of two (1e-13: the sums
    themselves are the same, up to the last bits of what is subnormal)."""
    rng = np.random.default_rng(n)
    coef, xs, zs, b = random_problem(rng, n, L)
    alpha, an = wl.random_angles(n * 2, 8), dv.make_ansatz(n, 1)
    S = 2 * alpha.size + 1
    got = []
    for c in (cvec(coef), cvec(coef * scale)):
        lcu, cost, local, part = dv.make_lcu(L, c, xs, zs), np.zeros(1), np.zeros(1), np.zeros(4 * S)
        dv.dvqls_cost(ctx, an, alpha, lcu, cvec(b), dv.DVQLS_FP64, cost)
        dv.dvqls_local_cost_grad(ctx, an, alpha, lcu, dv.DVQLS_FP64, local)
        dv.dvqls_cost_grad_partials(ctx, an, alpha, lcu, cvec(b), dv.DVQLS_FP64, 0, S, part)
        got.append((cost[0], local[0], part.reshape(S, 4)))
    assert abs(got[1][0] - got[0][0]) <= 1e-13 * max(1.0, abs(got[0][0]))
    assert abs(got[1][1] - got[0][1]) <= 1e-13 * max(1.0, abs(got[0][1]))
    assert np.all(np.abs(got[1][2][:, 2] / scale / scale - got[0][2][:, 2]) <= 1e-13 * np.abs(got[0][2][:, 2]))
    assert np.all(np.abs(got[1][2][:, :2] / scale - got[0][2][:, :2]) <= 1e-13 * np.abs(got[0][2][:, :2]).max())
