"""FP64 evaluations by Walsh-Hadamard classes in fixed point (L <= 64, n <= 10)
against the oracle and against the FP64 tiles.

Tolerance 1e-13 absolute on beta and delta (at most 1 in size): an amplitude
is the product of up to n (d + 1) <= 60 roundings of 2^-53, 1e-14 at worst, and
the fixed-point roundings add 2^10 x 2^-62 = 2e-16.  Cost and gradient are
quotients of sums of at most 64^2 weighted terms: 1e-12 as the other FP64 paths."""
import numpy as np
import pytest
import torch

from oracle import terms as oterms
from paper_2604_14435_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def cvec(a):
    return np.ascontiguousarray(np.asarray(a, dtype=np.complex128)).view(np.float64)


def problem(n, L, seed, masks="random", bscale=1.0, real_b=False):
    rng = np.random.default_rng(seed)
    N = 1 << n
    if masks == "random":  # nearly every pair a class of its own
        xs, zs = rng.integers(0, N, L), rng.integers(0, N, L)
    elif masks == "one":  # every term in one class
        xs, zs = np.full(L, rng.integers(0, N)), rng.integers(0, N, L)
    else:  # a tridiagonal matrix's masks
        xs, zs = (1 << rng.integers(0, n + 1, L)) - 1, rng.integers(0, N, L)
    b = rng.normal(size=N) + (0 if real_b else 1j * rng.normal(size=N))
    return (rng.normal(size=L) + 1j * rng.normal(size=L), xs.astype(np.uint32), zs.astype(np.uint32),
            b * bscale)


@pytest.mark.parametrize("n,d,L,masks,bscale,real_b", [
    (1, 3, 1, "random", 1.0, False), (2, 0, 4, "random", 1.0, True), (4, 2, 64, "one", 1.0, False),
    (5, 1, 33, "band", 1e-140, False), (6, 3, 64, "random", 1.0, False), (7, 2, 63, "band", 1e140, True),
    (8, 1, 2, "random", 1.0, False), (9, 2, 64, "band", 3.0, False), (10, 3, 64, "random", 1.0, False),
    (10, 5, 7, "one", 1.0, True)])
def test_against_the_oracle(dv, ctx, n, d, L, masks, bscale, real_b):
    coef, xs, zs, b = problem(n, L, 10 * n + L, masks, bscale, real_b)
    alpha = wl.random_angles(n * (d + 1), n + L)
    ref = oterms.cost_grad(n, d, alpha, b / np.linalg.norm(b), coef, xs, zs)
    an, lcu = dv.make_ansatz(n, d), dv.make_lcu(L, cvec(coef), xs, zs)
    c, bb = cvec(coef), cvec(b)
    lcu = dv.make_lcu(L, c, xs, zs)
    cost, grad, beta, delta = np.zeros(1), np.zeros(alpha.size), np.zeros(2 * L * L), np.zeros(2 * L)
    dv.dvqls_cost_grad(ctx, an, alpha, lcu, bb, dv.DVQLS_FP64, cost, grad, beta, delta)
    assert np.abs(beta.view(np.complex128).reshape(L, L) - ref["beta"]).max() <= 1e-13
    assert np.abs(delta.view(np.complex128) - ref["delta"]).max() <= 1e-13
    assert abs(cost[0] - ref["cost"]) <= 1e-12 * max(1.0, abs(ref["cost"]))
    assert np.all(np.abs(grad - ref["grad"]) <= 1e-12 * np.maximum(1.0, np.abs(ref["grad"])))


def test_states_with_single_amplitudes(dv, ctx):
    """Zero angles: amplitudes of exactly 0 and 1, the ends of the fixed-point range."""
    for n in (3, 10):
        coef, xs, zs, b = problem(n, 20, n, "band")
        alpha = np.zeros(2 * n)
        alpha[0] = np.pi
        ref = oterms.cost_grad(n, 1, alpha, b / np.linalg.norm(b), coef, xs, zs)
        c, bb = cvec(coef), cvec(b)
        cost, grad = np.zeros(1), np.zeros(2 * n)
        beta = np.zeros(2 * 400)
        dv.dvqls_cost_grad(ctx, dv.make_ansatz(n, 1), alpha, dv.make_lcu(20, c, xs, zs), bb, dv.DVQLS_FP64, cost, grad,
                           beta)
        assert np.abs(beta.view(np.complex128).reshape(20, 20) - ref["beta"]).max() <= 1e-13
        assert abs(cost[0] - ref["cost"]) <= 1e-12 * max(1.0, abs(ref["cost"]))
        assert np.all(np.abs(grad - ref["grad"]) <= 1e-12 * np.maximum(1.0, np.abs(ref["grad"])))


@pytest.mark.parametrize("n,d,L", [(3, 2, 10), (7, 4, 64), (10, 2, 40)])
def test_against_the_tiles(dv, ctx, n, d, L):
    """The allocation-free call evaluates the same FP64 terms on the tiles."""
    coef, xs, zs, b = problem(n, L, 77 + n)
    alpha = wl.random_angles(n * (d + 1), 5)
    t = [torch.from_numpy(a).cuda() for a in (cvec(coef), xs.view(np.int32), zs.view(np.int32), alpha, cvec(b))]
    an, lcu = dv.make_ansatz(n, d), dv.make_lcu(L, t[0], t[1], t[2])
    out = [torch.zeros(1 + alpha.size, device="cuda", dtype=torch.float64) for _ in range(2)]
    dv.dvqls_cost_grad(ctx, an, t[3], lcu, t[4], dv.DVQLS_FP64, out[0], out[0][1:])
    st = torch.cuda.current_stream().cuda_stream
    assert dv.dvqls_cost_grad_noalloc(st, an, t[3], lcu, t[4], dv.DVQLS_FP64, out[1], out[1][1:]) == dv.DVQLS_OK
    a, r = out[0].cpu().numpy(), out[1].cpu().numpy()
    assert np.all(np.abs(a - r) <= 1e-12 * np.maximum(1.0, np.abs(r)))


def test_table_follows_the_precision(dv, ctx):
    """FP32 and FP64 calls on one LCU in turn: neither uses the other's weights."""
    n, d, L = 6, 2, 30
    coef, xs, zs, b = problem(n, L, 3, "band")
    alpha = wl.random_angles(n * (d + 1), 4)
    ref = oterms.cost_grad(n, d, alpha, b / np.linalg.norm(b), coef, xs, zs)
    c, bb = cvec(coef), cvec(b)
    an, lcu = dv.make_ansatz(n, d), dv.make_lcu(L, c, xs, zs)
    for prec, tol in ((0, 1e-12), (3, 1e-6), (0, 1e-12), (3, 1e-6)):
        cost, grad = np.zeros(1), np.zeros(alpha.size)
        dv.dvqls_cost_grad(ctx, an, alpha, lcu, bb, prec, cost, grad)
        assert abs(cost[0] - ref["cost"]) <= tol * max(1.0, abs(ref["cost"])), prec


def test_non_finite_angles_give_nan(dv, ctx):
    """Fixed point holds no NaN: an instance with one is reported and its outputs are NaN; the others are right."""
    n, d, L = 6, 2, 20
    P = n * (d + 1)
    coef, xs, zs, b = problem(n, L, 3, "band")
    alpha = wl.random_angles(2 * P, 5)
    alpha[3] = np.nan
    ref = oterms.cost_grad(n, d, alpha[P:], b / np.linalg.norm(b), coef, xs, zs)
    dev = [torch.tensor(v, device="cuda") for v in (cvec(coef), xs.view(np.int32), zs.view(np.int32), cvec(b), alpha)]
    an, lcu = dv.make_ansatz(n, d), dv.make_lcu(L, dev[0], dev[1], dev[2])
    for local in (False, True):
        costs, grads = torch.zeros(2, device="cuda", dtype=torch.float64), torch.zeros(2 * P, device="cuda", dtype=torch.float64)
        arr = dv.make_instances([(an, lcu, dev[4][:P], dev[3]), (an, lcu, dev[4][P:], dev[3])])
        call = dv.dvqls_local_cost_grad_batched if local else dv.dvqls_cost_grad_batched
        with pytest.raises(dv.DvqlsError) as e:
            call(ctx, arr, dv.DVQLS_FP64, costs, grads)
            dv.dvqls_sync(ctx)
        assert e.value.code == dv.DVQLS_ERR_INVALID_ARG
        c, g = costs.cpu().numpy(), grads.cpu().numpy()
        assert np.isnan(c[0]) and np.isnan(g[:P]).all()
        if not local:
            assert abs(c[1] - ref["cost"]) <= 1e-12 and np.abs(g[P:] - ref["grad"]).max() <= 1e-12
        else:
            assert np.isfinite(c[1]) and np.isfinite(g[P:]).all()
