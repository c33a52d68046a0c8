"""The classical solve on X-mask diagonals (dvqls_lcu_solve_batched, n <= 12)
against dense solves, and where its diagonals are not formed.

Tolerance: the solves stop at a residual of 1e-13 and the systems' condition
numbers are below 1e3 (1e-10), below 1e4 through the normal equations (1e-8)."""
import numpy as np
import pytest

from oracle import terms as oterms

pytestmark = pytest.mark.gpu


def cv(a):
    return np.ascontiguousarray(np.asarray(a, dtype=np.complex128)).view(np.float64).reshape(-1)


def lcu_terms(rng, n, masks, per, shift):
    """shift I plus `per` random strings of small real weight on each of `masks` X-masks (Hermitian)."""
    N = 1 << n
    xs = np.repeat(rng.choice(N, size=masks, replace=False), per)
    zs = rng.integers(0, N, masks * per)
    order = rng.permutation(masks * per)
    coef = rng.uniform(-1, 1, masks * per) / (masks * per)
    return (np.concatenate([[shift], coef[order]]), np.concatenate([[0], xs[order]]).astype(np.uint32),
            np.concatenate([[0], zs[order]]).astype(np.uint32))


@pytest.mark.parametrize("n,nrhs,masks,per,complex_b", [
    (1, 1, 2, 1, False), (3, 4, 8, 2, True), (7, 3, 5, 6, False), (8, 2, 1, 9, True), (9, 2, 9, 4, False),
    (10, 3, 11, 8, True), (11, 1, 3, 3, False), (7, 2, 100, 1, True), (7, 2, 64, 3, False)])
def test_positive_definite(dv, ctx, n, nrhs, masks, per, complex_b):
    rng = np.random.default_rng(n * 100 + masks)
    coef, xs, zs = lcu_terms(rng, n, masks, per, 2.0)
    N = 1 << n
    B = rng.normal(size=(nrhs, N)) + (1j * rng.normal(size=(nrhs, N)) if complex_b else 0)
    x, c = np.zeros(2 * nrhs * N), cv(coef)
    it, rr = dv.dvqls_lcu_solve_batched(ctx, n, dv.make_lcu(len(xs), c, xs, zs), nrhs, cv(B), 1e-13, 2000, x)
    ref = np.linalg.solve(oterms.lcu_matrix(coef, xs, zs, n), B.T).T
    x = x.view(np.complex128).reshape(nrhs, N)
    assert np.linalg.norm(x - ref) <= 1e-10 * np.linalg.norm(ref)
    assert rr.max() <= 1e-13 and it.min() >= 1


@pytest.mark.parametrize("n,complex_c", [(4, False), (6, True), (9, False)])
def test_normal_equations(dv, ctx, n, complex_c):
    """CG breaks down on an indefinite (or non-Hermitian) matrix: A^dag A x = A^dag b."""
    rng = np.random.default_rng(n)
    coef, xs, zs = lcu_terms(rng, n, 4, 3, 0.0)
    coef = coef * (0.3 + 1j * rng.uniform(-0.3, 0.3, len(xs)) if complex_c else 0.3)
    coef[0] = 1j if complex_c else 0.0
    coef = np.append(coef, -1.0)
    xs, zs = np.append(xs, 0).astype(np.uint32), np.append(zs, 1).astype(np.uint32)  # - Z_0
    N = 1 << n
    b = rng.normal(size=N) + (1j * rng.normal(size=N) if complex_c else 0)
    x, c = np.zeros(2 * N), cv(coef)
    dv.dvqls_lcu_solve(ctx, n, dv.make_lcu(len(xs), c, xs, zs), cv(b), 1e-13, 20000, x)
    ref = np.linalg.solve(oterms.lcu_matrix(coef, xs, zs, n), b)
    assert np.linalg.norm(x.view(np.complex128) - ref) <= 1e-8 * np.linalg.norm(ref)


def test_not_converged_reports(dv, ctx):
    rng = np.random.default_rng(0)
    coef, xs, zs = lcu_terms(rng, 8, 6, 4, 1.2)
    x, c = np.zeros(2 << 8), cv(coef)
    with pytest.raises(dv.DvqlsError) as e:
        dv.dvqls_lcu_solve(ctx, 8, dv.make_lcu(len(xs), c, xs, zs), cv(rng.normal(size=256)), 1e-14, 2, x)
    assert e.value.code == dv.DVQLS_ERR_NUMERIC and np.any(x != 0)
