"""The classical solve of several right-hand sides at n = 12, the largest instance of
the kernel on X-mask diagonals (16 amplitudes per thread), and term by term beside it.

The true residual is checked: the solves stop at 1e-13 by their own recurrence, which
for matrices of condition number 3 (the normal equations: 20) is off by a few roundings of
|x| per iteration: 1e-12 (1e-11) of |b|."""
import numpy as np
import pytest

from oracle import terms as oterms

from test_gpu_solve_diagonals import cv, lcu_terms

pytestmark = pytest.mark.gpu

N_Q = 12


def residual(coef, xs, zs, x, b):
    r = b.astype(np.complex128).copy()
    for c, px, pz in zip(coef, xs, zs):
        r -= c * oterms.apply_pauli(int(px), int(pz), x)
    return np.linalg.norm(r) / np.linalg.norm(b)


@pytest.mark.parametrize("nrhs,masks,per,complex_b,complex_c", [
    (2, 1, 1, False, False), (3, 8, 4, False, False), (2, 8, 4, True, False), (2, 5, 3, False, True), (5, 63, 1, True, False),
    (2, 100, 1, False, False)])  # 101 masks: term by term
def test_positive_definite(dv, ctx, nrhs, masks, per, complex_b, complex_c):
    rng = np.random.default_rng(masks + nrhs)
    coef, xs, zs = lcu_terms(rng, N_Q, masks, per, 2.0)
    if complex_c:  # strings with an odd number of Y: real coefficients, complex diagonals
        zs[1:] |= xs[1:] & (~xs[1:] + 1)
    N = 1 << N_Q
    B = rng.normal(size=(nrhs, N)) + (1j * rng.normal(size=(nrhs, N)) if complex_b else 0)
    B[0] = 0.0 if nrhs == 5 else B[0]  # one system with nothing to solve
    x, c = np.zeros(2 * nrhs * N), cv(coef)
    it, rr = dv.dvqls_lcu_solve_batched(ctx, N_Q, dv.make_lcu(len(xs), c, xs, zs), nrhs, cv(B), 1e-13, 500, x)
    x = x.view(np.complex128).reshape(nrhs, N)
    for k in range(nrhs):
        if not B[k].any():
            assert it[k] == 0 and not x[k].any()
            continue
        assert rr[k] <= 1e-13 and it[k] >= 1
        assert residual(coef, xs, zs, x[k], B[k]) <= 1e-12


@pytest.mark.parametrize("complex_b", [False, True])
def test_normal_equations(dv, ctx, complex_b):
    """One solve breaks down on an indefinite matrix and goes on with A^dag A x = A^dag b, beside others."""
    rng = np.random.default_rng(4)
    coef, xs, zs = lcu_terms(rng, N_Q, 4, 3, 0.0)
    coef = np.append(coef * 0.3, -1.0)
    xs, zs = np.append(xs, 0).astype(np.uint32), np.append(zs, 1).astype(np.uint32)  # - Z_0
    N, nrhs = 1 << N_Q, 3
    B = rng.normal(size=(nrhs, N)) + (1j * rng.normal(size=(nrhs, N)) if complex_b else 0)
    x, c = np.zeros(2 * nrhs * N), cv(coef)
    dv.dvqls_lcu_solve_batched(ctx, N_Q, dv.make_lcu(len(xs), c, xs, zs), nrhs, cv(B), 1e-13, 5000, x)
    x = x.view(np.complex128).reshape(nrhs, N)
    for k in range(nrhs):
        assert residual(coef, xs, zs, x[k], B[k]) <= 1e-11
