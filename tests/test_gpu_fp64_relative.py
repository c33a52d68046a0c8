"""FP64 evaluations and fidelities keep their relative accuracy where the values are
small: angles near zero leave amplitudes of 1e-3 down to 1e-40, and so are the
overlaps that they enter.

Reference in extended precision (numpy longdouble).  Bound: the usual one of FP64
sums, gamma times the same value formed with the absolute values of all factors and
terms.  An amplitude takes P = n (d + 1) rotations of at most four roundings each, an
overlap two amplitudes, one product and a sum whose terms lie next to their largest:
gamma = (8 P + 64) 2^-53."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

LD = np.longdouble


def state(n, d, alpha, absolute):
    """psi(alpha), or the sum over paths of the absolute values of their factors."""
    N = 1 << n
    i = np.arange(N)
    par = sum(((i >> q) & 1) * ((i >> ((q + 1) % n)) & 1) for q in (range(n) if n >= 3 else range(n - 1)))
    ring = np.where(par & 1, -1, 1) if not absolute and n > 1 else np.ones(N, int)
    psi = np.zeros(N, LD)
    psi[0] = 1
    for layer in range(d + 1):
        if layer:
            psi = psi * ring
        for q in range(n):
            h = LD(alpha[layer * n + q]) / 2
            c, s = np.cos(h), np.sin(h)
            v = psi.reshape(N >> (q + 1), 2, 1 << q)
            lo, hi = v[:, 0].copy(), v[:, 1].copy()
            if absolute:
                c, s = abs(c), abs(s)
                v[:, 0], v[:, 1] = c * lo + s * hi, s * lo + c * hi
            else:
                v[:, 0], v[:, 1] = c * lo - s * hi, s * lo + c * hi
    return psi


def parity(v):
    return np.array([bin(int(k)).count("1") & 1 for k in v])


def angles(P, scale, seed):
    return np.random.default_rng(seed).uniform(scale, 3 * scale, P)


@pytest.mark.parametrize("n,d,scale,real_b", [(1, 0, 1e-9, True), (3, 1, 1e-3, False), (5, 2, 1e-4, False),
                                              (7, 0, 1e-4, True), (8, 1, 1e-3, True), (8, 2, 1e-6, False),
                                              (9, 1, 1e-3, False), (10, 2, 1e-3, False), (10, 0, 1e-4, True)])
def test_small_overlaps(dv, ctx, n, d, scale, real_b):
    rng = np.random.default_rng(40 + n)
    N, L, P = 1 << n, 14, n * (d + 1)
    xs = rng.integers(0, N, L).astype(np.uint32)
    zs = rng.integers(0, N, L).astype(np.uint32)
    xs[0], xs[1] = 0, N - 1
    coef = rng.normal(size=L) + 1j * rng.normal(size=L)
    b = rng.normal(size=N) + (0 if real_b else 1j * rng.normal(size=N))
    b[: N // 2] *= 1e-8  # and a right-hand side of two sizes
    alpha = angles(P, scale, n + d)
    c, bb = coef.view(np.float64).copy(), np.asarray(b, np.complex128).view(np.float64).copy()
    cost, grad, beta, delta = np.zeros(1), np.zeros(P), np.zeros(2 * L * L), np.zeros(2 * L)
    dv.dvqls_cost_grad(ctx, dv.make_ansatz(n, d), alpha, dv.make_lcu(L, c, xs, zs), bb, dv.DVQLS_FP64, cost, grad, beta,
                       delta)
    beta, delta = beta.view(np.complex128).reshape(L, L), delta.view(np.complex128)
    psi, size = state(n, d, alpha, False), state(n, d, alpha, True)
    gamma = LD(8 * P + 64) * LD(2) ** -53
    i = np.arange(N)
    norm = np.sqrt(np.sum(b.real.astype(LD) ** 2 + b.imag.astype(LD) ** 2))
    br, bi = b.real.astype(LD) / norm, b.imag.astype(LD) / norm

    def string(l):  # sigma_l psi = i^k phi, phi real
        k = bin(int(xs[l] & zs[l])).count("1") % 4
        src = i ^ int(xs[l])
        return k, psi[src] * (1 - 2 * parity(src & int(zs[l]))), size[src]

    for l in range(L):
        kl, pl, al = string(l)
        for m in range(L):
            km, pm, am = string(m)
            ref = np.sum(pl * pm)
            got = beta[l, m] * (-1j) ** ((km - kl) % 4)  # exact
            assert abs(LD(got.real) - ref) <= gamma * np.sum(al * am), (l, m)
            assert got.imag == 0
        got = delta[l] * (-1j) ** kl
        assert abs(LD(got.real) - np.sum(br * pl)) <= gamma * np.sum(abs(br) * al), l
        assert abs(LD(got.imag) + np.sum(bi * pl)) <= gamma * np.sum(abs(bi) * al), l


@pytest.mark.parametrize("n,d,scale", [(1, 0, 1e-9), (4, 1, 1e-3), (7, 0, 1e-4), (8, 2, 1e-4), (10, 1, 1e-3), (11, 1, 1e-3),
                                       (12, 0, 1e-3), (12, 1, 1e-2)])
def test_small_fidelity(dv, ctx, n, d, scale):
    N, P = 1 << n, n * (d + 1)
    alpha = angles(P, scale, 3 * n + d)
    x = np.zeros(N, np.complex128)
    x[N - 1], x[N // 2] = 0.25 - 0.5j, 1e-12
    F = np.zeros(1)
    dv.dvqls_fidelity(ctx, dv.make_ansatz(n, d), alpha, x.view(np.float64), F)
    psi, size = state(n, d, alpha, False), state(n, d, alpha, True)
    re, im = np.sum(x.real * psi), np.sum(x.imag * psi)
    nx = np.sum(x.real.astype(LD) ** 2 + x.imag.astype(LD) ** 2)
    bound = np.sum(abs(x.real) * size) ** 2 + np.sum(abs(x.imag) * size) ** 2
    assert abs(LD(F[0]) - (re * re + im * im) / nx) <= 2 * LD(8 * P + 64) * LD(2) ** -53 * bound / nx
    assert F[0] > 0


@pytest.mark.parametrize("n", [3, 10])
def test_deep_circuits(dv, ctx, n):
    """Many layers: the norm stays one, and a state of one path has one amplitude."""
    d = 1024 // n - 1
    P = n * (d + 1)
    alpha = np.random.default_rng(n).uniform(-np.pi, np.pi, P)
    psi = state(n, d, alpha, False)
    x = psi.astype(np.float64).astype(np.complex128)
    F = np.zeros(1)
    dv.dvqls_fidelity(ctx, dv.make_ansatz(n, d), alpha, x.view(np.float64), F)
    assert abs(F[0] - 1) <= (8 * P + 64) * 2.0 ** -53
    coef, xs, zs = np.ones(2, np.complex128), np.zeros(2, np.uint32), np.array([0, 1], np.uint32)
    cost, beta, delta = np.zeros(1), np.zeros(8), np.zeros(4)
    dv.dvqls_cost(ctx, dv.make_ansatz(n, d), alpha, dv.make_lcu(2, coef.view(np.float64), xs, zs), x.view(np.float64),
                  dv.DVQLS_FP64, cost, beta, delta)
    assert abs(beta[0] - 1) <= (8 * P + 64) * 2.0 ** -53 and abs(delta[0] - 1) <= (8 * P + 64) * 2.0 ** -53
