"""FP64 evaluations at the ends of the range of a double: large coefficients, and
right-hand sides whose norm is not finite."""
import numpy as np
import pytest
import torch

from oracle import terms as oterms
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


@pytest.mark.parametrize("bad", [np.inf, np.nan, 1e200, 0.0])  # an entry; 1e200: ||b||^2 overflows; 0: all of b
@pytest.mark.parametrize("n", [3, 6, 10])
def test_bad_norm_gives_nan(dv, ctx, n, bad):
    """A right-hand side without a finite, positive norm is reported and its instance's outputs are NaN; the other
    instance of the batch is right."""
    d, L = 1, 12
    P = n * (d + 1)
    rng = np.random.default_rng(n)
    coef, xs, zs, b = random_problem(rng, n, L)
    ref = oterms.cost_grad(n, d, wl.random_angles(P, 3), b, coef, xs, zs)
    wrong = b.copy()
    if bad == 0.0:
        wrong[:] = 0.0
    else:
        wrong[1] = bad
    dev = [torch.tensor(v, device="cuda") for v in (cvec(coef), xs.view(np.int32), zs.view(np.int32),
                                                    wl.random_angles(P, 3), cvec(wrong), cvec(b))]
    an, lcu = dv.make_ansatz(n, d), dv.make_lcu(L, dev[0], dev[1], dev[2])
    costs, grads = (torch.zeros(m, device="cuda", dtype=torch.float64) for m in (2, 2 * P))
    arr = dv.make_instances([(an, lcu, dev[3], dev[4]), (an, lcu, dev[3], dev[5])])
    with pytest.raises(dv.DvqlsError) as e:
        dv.dvqls_cost_grad_batched(ctx, arr, dv.DVQLS_FP64, costs, grads)
        dv.dvqls_sync(ctx)
    assert e.value.code == dv.DVQLS_ERR_INVALID_ARG
    c, g = costs.cpu().numpy(), grads.cpu().numpy()
    assert np.isnan(c[0]) and np.isnan(g[:P]).all()
    assert abs(c[1] - ref["cost"]) <= 1e-12 * max(1.0, abs(ref["cost"]))
    assert np.all(np.abs(g[P:] - ref["grad"]) <= 1e-12 * np.maximum(1.0, np.abs(ref["grad"])))
