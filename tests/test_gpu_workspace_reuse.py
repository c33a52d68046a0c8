"""Equal cost passes with another kind of call in between: every call plans the
context's workspace for itself, so the cost pass has to bring its instance table
again (the table holds shapes and addresses only, so two systems of one shape in
host arrays have equal tables).

The passes before and after are the same sums on the same inputs: equal bits."""
import numpy as np
import pytest

from oracle import terms as oterms
from paper_2604_14435_gb300 import workloads as wl

from test_gpu_terms import check, cvec, random_problem

pytestmark = pytest.mark.gpu

N_Q, D, L = 6, 2, 20


def fidelity(dv, ctx, p):
    n, d, alpha, b, coef, xs, zs = p
    dv.dvqls_fidelity(ctx, dv.make_ansatz(n, d), alpha, cvec(b), np.zeros(1))


def fidelity_hbm(dv, ctx, p):
    n = 13
    x = np.zeros(2 << n)
    x[0] = 1.0
    dv.dvqls_fidelity(ctx, dv.make_ansatz(n, 0), wl.random_angles(n, 1), x, np.zeros(1))


def solve(dv, ctx, p):
    q = np.full(1 << N_Q, 0.5)
    c, xs, zs = cvec([2.0, 0.25]), np.array([0, 1], np.uint32), np.array([0, 2], np.uint32)
    dv.dvqls_lcu_solve(ctx, N_Q, dv.make_lcu(2, c, xs, zs), cvec(q), 1e-10, 100, np.zeros(2 << N_Q))


def decompose(dv, ctx, p):
    A = wl.toeplitz_dense(N_Q, 2.5, -1.0)
    dv.dvqls_pauli_decompose(ctx, A, N_Q, 0.0, 8, np.zeros(16), np.zeros(8, np.uint32), np.zeros(8, np.uint32))


def decompose_banded(dv, ctx, p):
    off, bands = wl.toeplitz_bands(N_Q, [2.5, -1.0])
    dv.dvqls_pauli_decompose_banded(ctx, N_Q, off, bands, 0.0, 8, np.zeros(16), np.zeros(8, np.uint32),
                                    np.zeros(8, np.uint32))


def circuit(dv, ctx, p):
    c, xs, zs = cvec([1.0, 0.5]), np.array([0, 1], np.uint32), np.array([0, 1], np.uint32)
    dv.dvqls_circuit_cost_grad_fp64(ctx, dv.make_ansatz(2, 0), wl.random_angles(2, 3), dv.make_lcu(2, c, xs, zs),
                                    cvec(wl.plus_state(2)), np.zeros(1), np.zeros(2))


def combine(dv, ctx, p):
    dv.dvqls_combine_partials(ctx, 4, 1, np.ones(4 * 17), np.zeros(1), np.zeros(8))


def optimize(dv, ctx, p):
    n, d, alpha, b, coef, xs, zs = p
    inst = dv.make_instances([(dv.make_ansatz(n, d), dv.make_lcu(L, cvec(coef), xs, zs), alpha, cvec(b))])
    dv.dvqls_optimize(ctx, inst, cvec(b), dv.make_adam(max_iter=1, precision=dv.DVQLS_FP64), np.zeros(alpha.size))


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("between", [fidelity, fidelity_hbm, solve, decompose, decompose_banded, circuit, combine,
                                     optimize])
def test_cost_pass_after_another_call(dv, ctx, prec, between):
    rng = np.random.default_rng(11)
    problems = []
    for i in range(2):  # two systems of one shape: one table
        coef, xs, zs, b = random_problem(rng, N_Q, L)
        problems.append((N_Q, D, wl.random_angles(N_Q * (D + 1), 20 + i), b, coef, xs, zs))
    dv.dvqls_set_tuning(ctx, 1, 0)
    try:
        def run(p):
            n, d, alpha, b, coef, xs, zs = p
            c, bb = cvec(coef), cvec(b)
            out = {"cost": np.zeros(1), "grad": np.zeros(alpha.size), "beta": np.zeros(2 * L * L), "delta": np.zeros(2 * L)}
            dv.dvqls_cost_grad(ctx, dv.make_ansatz(n, d), alpha, dv.make_lcu(L, c, xs, zs), bb, prec, out["cost"],
                               out["grad"], out["beta"], out["delta"])
            return out
        first = [run(p) for p in problems]
        for p, f in zip(problems, first):
            between(dv, ctx, p)
            again = run(p)
            for k in f:
                assert np.array_equal(f[k], again[k]), k
            n, d, alpha, b, coef, xs, zs = p
            got = {"cost": again["cost"][0], "grad": again["grad"], "beta": again["beta"].view(np.complex128).reshape(L, L),
                   "delta": again["delta"].view(np.complex128)}
            check(got, oterms.cost_grad(n, d, alpha, b, coef, xs, zs), prec)
    finally:
        dv.dvqls_set_tuning(ctx, 0, -1)
