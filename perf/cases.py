"""Workloads whose time on the GPU is followed, as calls of the public binding.

Each case is one call (or one step) that a program built on this library makes
again and again: the evaluations of an optimizer, the set-up of a system, a
step of the warm-start network.  `listed()` names the workloads of the
repository's own configurations, `draw()` gives others of the same ranges,
`prepare()` what a program holds before the call, `run()` the call itself,
`work()` the bytes and operations it cannot do without and `exact()` its
results in 64 bits by plain torch.

Where the term kernel sums in FP32, the amplitude split and the state layout
are pinned (dvqls_set_tuning), as a program does that wants the same bits from
one run to the next: the tuner's choice follows its timings, and the splits
differ in the order of the sums.
"""
import math

import numpy as np
import torch

from paper_2604_14435_gb300 import dvqls as D
from paper_2604_14435_gb300 import warmstart
from paper_2604_14435_gb300 import workloads as wl

PRECISION = {"fp64": D.DVQLS_FP64, "fp32": D.DVQLS_FP32, "tc": D.DVQLS_FP32_TC}
HS_L, SMALL_SIZES = 256, (4, 6, 8, 10, 12)


def listed():
    return [
        # The validation system (n = 3, every Pauli term, depth 2): the smallest
        # evaluation, in FP64 and with all its beta and delta, as a check of a set-up does.
        {"name": "eval_n3_fp64", "kind": "terms", "n": 3, "d": 2},
        # One evaluation of the host L-BFGS-B loop on the throughput system (its
        # default precision, host arrays in and out).
        {"name": "eval_n10_fp64", "kind": "batch", "precision": "fp64", "count": 1, "n_min": 10, "n_max": 10,
         "L": 64, "d": 4, "host": True},
        # One round of the lock-step L-BFGS that makes the warm start's training
        # targets: systems of n = 6..10 in FP64, host arrays.
        {"name": "lockstep_n6_10_fp64", "kind": "batch", "precision": "fp64", "count": 48, "n_min": 6, "n_max": 10,
         "L": 64, "d": 4, "host": True},
        # The throughput workload: cost and gradient of 32 systems held on the GPU.
        {"name": "batch32_n10_tc", "kind": "batch", "precision": "tc", "count": 32, "n_min": 10, "n_max": 10,
         "L": 64, "d": 4, "host": False},
        # Its local cost, the cost function that the paper times.
        {"name": "local_n10_tc", "kind": "local", "precision": "tc", "count": 32, "n_min": 10, "n_max": 10,
         "L": 64, "d": 4},
        # The Hele-Shaw-type pressure system: many terms, a deeper ansatz, a real source.
        {"name": "hele_shaw_n10_tc", "kind": "hele_shaw", "grid": 32, "count": 8, "d": 6, "L": HS_L},
        # The uneven batch: 62 small systems and two whose states live in HBM.
        {"name": "uneven_n4_20_tc", "kind": "uneven", "count": 62, "big": 2, "big_n": 20},
        # Set-up of a large banded system: decomposition to its top 64 terms.
        {"name": "decompose_n20_banded", "kind": "banded", "n": 20, "bands": 1, "L": 64, "tau": 0.01},
        # Set-up of the pressure system from its matrix: top 256 terms.
        {"name": "decompose_n10_dense", "kind": "dense", "grid": 32, "L": HS_L, "tau": 0.001},
        # The pruning sweep's classical solves: 64 right-hand sides of one LCU, host arrays.
        {"name": "solve_n10_rhs64", "kind": "solve", "n": 10, "nrhs": 64, "L": 64},
        # Adam on a group of held-out systems (the warm-start evaluation's FP32 cost pass).
        {"name": "adam_n10_fp32", "kind": "adam", "n": 10, "count": 16, "steps": 5, "L": 64, "d": 4},
        # One full-batch training step of the warm-start network.
        {"name": "train_b2000_h256", "kind": "train", "batch": 2000, "hidden": 256},
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    kind = rng.choice(["terms", "batch", "batch", "local", "hele_shaw", "uneven", "banded", "dense", "solve", "adam",
                       "train"])
    if kind == "terms":
        return {"kind": kind, "n": rng.randint(1, 5), "d": rng.randint(0, 8)}
    if kind in ("batch", "local"):
        lo = rng.randint(4, 11)
        hi = min(11, rng.randint(lo, lo + 3))
        c = {"kind": kind, "precision": rng.choice(["fp64", "tc"]) if kind == "batch" else "tc",
             "count": _log(rng, 1, 48 if kind == "batch" else 16), "n_min": lo, "n_max": hi, "L": rng.randint(9, 64),
             "d": rng.randint(1, 5)}
        if kind == "batch":
            c["host"] = rng.random() < 0.5
        return c
    if kind == "hele_shaw":
        return {"kind": kind, "grid": rng.choice([16, 32]), "count": _log(rng, 1, 8), "d": rng.randint(2, 6),
                "L": rng.randint(65, HS_L)}
    if kind == "uneven":
        return {"kind": kind, "count": _log(rng, 4, 62), "big": rng.randint(0, 2), "big_n": rng.randint(13, 18)}
    if kind == "banded":
        return {"kind": kind, "n": rng.randint(3, 19), "bands": rng.randint(1, 3), "L": _log(rng, 4, 512),
                "tau": rng.choice([0.0, 0.001, 0.01])}
    if kind == "dense":
        return {"kind": kind, "grid": rng.choice([4, 8, 16, 32]), "L": _log(rng, 5, 1024),
                "tau": rng.choice([0.0, 0.001, 0.01])}
    if kind == "solve":
        return {"kind": kind, "n": rng.randint(4, 11), "nrhs": _log(rng, 1, 64), "L": rng.randint(9, 64)}
    if kind == "adam":
        return {"kind": kind, "n": rng.randint(6, 10), "count": _log(rng, 1, 16), "steps": rng.randint(1, 5),
                "L": rng.randint(33, 64), "d": rng.randint(2, 4)}
    return {"kind": kind, "batch": _log(rng, 1, 4000), "hidden": rng.choice([33, 64, 128, 200, 256, 384])}


# ------------------------------------------------------------------- inputs


class Handle:
    """A context that goes with its state."""

    def __init__(self):
        self.ctx = D.dvqls_create(0, torch.cuda.current_stream().cuda_stream)

    def __del__(self):
        if D is not None:
            D.dvqls_destroy(self.ctx)


def _lcu_banded(ctx, inst, L_max, tau=0.0):
    coef, xm, zm = np.zeros(2 * L_max), np.zeros(L_max, np.uint32), np.zeros(L_max, np.uint32)
    L, _, _ = D.dvqls_pauli_decompose_banded(ctx, inst["n"], inst["offsets"], np.ascontiguousarray(inst["bands"]),
                                             tau, L_max, coef, xm, zm)
    return L, coef[: 2 * L].copy(), xm[:L].copy(), zm[:L].copy()


def _lcu_dense(ctx, A, n, L_max, tau):
    coef, xm, zm = np.zeros(2 * L_max), np.zeros(L_max, np.uint32), np.zeros(L_max, np.uint32)
    L, _, _ = D.dvqls_pauli_decompose(ctx, np.ascontiguousarray(A), n, tau, L_max, coef, xm, zm)
    return L, coef[: 2 * L].copy(), xm[:L].copy(), zm[:L].copy()


def _system(n, d, lcu, alpha, b):
    return {"n": n, "d": d, "L": lcu[0], "coef": lcu[1], "x": lcu[2], "z": lcu[3],
            "alpha": np.ascontiguousarray(alpha, dtype=np.float64),
            "b": np.ascontiguousarray(b, dtype=np.complex128).view(np.float64).copy()}


def _systems(ctx, case, seed):
    """The systems of a cost case (host arrays), from the seed alone."""
    kind, out = case["kind"], []
    if kind == "terms":  # tridiagonal Toeplitz with every one of its terms; the angles by the seed
        n, d = case["n"], case["d"]
        rng = np.random.default_rng(seed)
        A = wl.toeplitz_dense(n, 2.5, -rng.uniform(0.5, 1.2))
        A = A / np.linalg.norm(A, 2)
        lcu = _lcu_dense(ctx, A, n, 1 << (2 * n), 0.0)
        return [_system(n, d, lcu, wl.random_angles(n * (d + 1), 1000 + seed), wl.plus_state(n))]
    if kind in ("batch", "local", "adam"):
        lo, hi = (case["n"], case["n"]) if kind == "adam" else (case["n_min"], case["n_max"])
        for i in range(case["count"]):
            n = hi - i % (hi - lo + 1)  # the mix of sizes is the case's, the systems are the seed's
            q = wl.throughput_instance(1000 * seed + i, n=n, d=case["d"], L_max=case["L"])
            out.append(_system(n, case["d"], _lcu_banded(ctx, q, case["L"]), q["alpha"], q["b"]))
    elif kind == "hele_shaw":
        n = 2 * int(math.log2(case["grid"]))
        for i in range(case["count"]):
            q = wl.hele_shaw_pressure(100 * seed + i, grid=case["grid"], d=case["d"], L_max=case["L"])
            out.append(_system(n, case["d"], _lcu_dense(ctx, q["A"], n, case["L"], 0.0), q["alpha"], q["b"]))
    elif kind == "uneven":
        for i in range(case["count"] + case["big"]):
            if i < case["count"]:  # tri- and pentadiagonal in turn
                q = wl.uneven_batch(1000 * seed + i, 2, 0, (SMALL_SIZES[i % len(SMALL_SIZES)],))[i % 2]
            else:
                q = wl.uneven_batch(1000 * seed + i, 0, 1, big_n=case["big_n"])[0]
            out.append(_system(q["n"], q["d"], _lcu_banded(ctx, q, q["L_max"], q["tau"]), q["alpha"], q["b"]))
    return out


def _on_gpu(s):
    t = dict(s)
    for k in ("coef", "alpha", "b"):
        t[k] = torch.from_numpy(s[k]).cuda()
    for k in ("x", "z"):
        t[k] = torch.from_numpy(s[k].view(np.int32)).cuda()
    return t


def _items(systems):
    return [(D.make_ansatz(s["n"], s["d"]), D.make_lcu(s["L"], s["coef"], s["x"], s["z"]), s["alpha"], s["b"])
            for s in systems]


def _matrix(case, seed):
    """The matrix of a dense decomposition: the pressure system's."""
    q = wl.hele_shaw_pressure(seed, grid=case["grid"])
    return int(math.log2(case["grid"])) * 2, np.ascontiguousarray(q["A"])


def _bands(case, seed):
    """Toeplitz bands of a large system, drawn as in the uneven batch."""
    rng = np.random.default_rng(seed)
    off = rng.uniform(-1.5, 4.0, case["bands"])
    a = max(rng.uniform(-1.5, 4.0), 1.05 * 2.0 * float(np.sum(np.abs(off))))
    k = min(case["bands"], (1 << case["n"]) - 1)
    return wl.toeplitz_bands(case["n"], [a] + list(off[:k]))


def _training(case, seed):
    """Features, angle targets and masks of the warm-start family (n = 6..10)."""
    rng = np.random.default_rng(seed)
    B = case["batch"]
    X = np.zeros((B, warmstart.FEATURES), np.float32)
    Y = np.zeros((B, warmstart.P_MAX), np.float32)
    M = np.zeros((B, warmstart.P_MAX), np.float32)
    n = rng.integers(warmstart.N_MIN, warmstart.N_MAX + 1, B)
    X[:, 0] = rng.uniform(2.0, 4.0, B) / 4.0
    X[:, 1] = rng.uniform(-1.5, -0.5, B) / 1.5
    X[np.arange(B), 2 + n - warmstart.N_MIN] = 1.0
    M[:] = np.arange(warmstart.P_MAX)[None, :] < (n * (warmstart.DEPTH + 1))[:, None]
    Y[:] = M * (rng.normal(0.0, 0.3, Y.shape) + 0.5 * np.pi * (np.arange(warmstart.P_MAX)[None, :] < n[:, None]))
    return X, Y, M, warmstart.init_params(case["hidden"], seed)


LR = 2e-3  # the training run's step size


def prepare(case, seed):
    h, kind = Handle(), case["kind"]
    st = {"case": case, "handle": h}
    if kind in ("terms", "batch", "local", "hele_shaw", "uneven", "adam"):
        systems = _systems(h.ctx, case, seed)
        P = [s["n"] * (s["d"] + 1) for s in systems]
        if kind == "adam":
            xhat = []
            for s in systems:
                x = np.zeros(2 << s["n"])
                D.dvqls_lcu_solve(h.ctx, s["n"], D.make_lcu(s["L"], s["coef"], s["x"], s["z"]), s["b"], 1e-12, 20000, x)
                xhat.append(x)
            D.dvqls_set_tuning(h.ctx, 1, 0)
            st["xhat"] = np.concatenate(xhat)
            st["adam"] = D.make_adam(lr=0.02, max_iter=case["steps"], target_fidelity=2.0, precision=D.DVQLS_FP32)
            st["alpha"] = np.zeros(sum(P))
        else:
            if kind != "terms" and case.get("precision", "tc") == "tc":
                D.dvqls_set_tuning(h.ctx, 1, 0)
            if not case.get("host"):
                systems = [_on_gpu(s) for s in systems]
            if case.get("host"):
                st["costs"], st["grads"] = np.zeros(len(P)), np.zeros(sum(P))
            else:
                st["costs"] = torch.zeros(len(P), dtype=torch.float64, device="cuda")
                st["grads"] = torch.zeros(sum(P), dtype=torch.float64, device="cuda")
            if kind == "terms":
                L = systems[0]["L"]
                st["beta"] = torch.zeros(L * L, dtype=torch.complex128, device="cuda")
                st["delta"] = torch.zeros(L, dtype=torch.complex128, device="cuda")
        st["systems"] = systems
        st["items"] = _items(systems)
        st["inst"] = D.make_instances(st["items"])
    elif kind in ("banded", "dense"):
        if kind == "dense":
            n, A = _matrix(case, seed)
            st["in"] = torch.from_numpy(A).cuda()
        else:
            n = case["n"]
            st["offsets"], bands = _bands(case, seed)
            st["in"] = torch.from_numpy(np.ascontiguousarray(bands)).cuda()
        st["n"] = n
        st["coef"] = torch.zeros(case["L"], dtype=torch.complex128, device="cuda")
        st["x"] = torch.zeros(case["L"], dtype=torch.int32, device="cuda")
        st["z"] = torch.zeros(case["L"], dtype=torch.int32, device="cuda")
    elif kind == "solve":
        n, k = case["n"], case["nrhs"]
        q = wl.throughput_instance(seed, n=n, L_max=case["L"])
        st["lcu"] = _lcu_banded(h.ctx, q, case["L"])
        st["b"] = np.ascontiguousarray(wl.gaussian_rhs(1 << n, k, seed).astype(np.complex128)).view(np.float64).reshape(-1)
        st["x"] = np.zeros(2 * k << n)
    else:
        X, Y, M, p = _training(case, seed)
        st["net"] = D.dvqls_ws_create(h.ctx, warmstart.FEATURES, case["hidden"], warmstart.P_MAX, p)
        st["data"] = [torch.from_numpy(v).cuda() for v in (X, Y, M)]
        st["params"] = torch.zeros(p.size, dtype=torch.float32, device="cuda")
        st["keep"] = Network(st["net"], h)
    return st


class Network:
    """A warm-start network that goes with its state (before its context)."""

    def __init__(self, net, handle):
        self.net, self.handle = net, handle

    def __del__(self):
        if D is not None:
            D.dvqls_ws_destroy(self.net)


# --------------------------------------------------------------------- call


def run(st):
    case, ctx = st["case"], st["handle"].ctx
    kind = case["kind"]
    if kind == "terms":
        an, lcu, alpha, b = st["items"][0]
        D.dvqls_cost_grad(ctx, an, alpha, lcu, b, D.DVQLS_FP64, st["costs"], st["grads"], st["beta"], st["delta"])
        return {"cost": st["costs"], "grad": st["grads"], "beta": st["beta"], "delta": st["delta"]}
    if kind == "batch" and case["count"] == 1 and case["host"]:
        an, lcu, alpha, b = st["items"][0]
        D.dvqls_cost_grad(ctx, an, alpha, lcu, b, PRECISION[case["precision"]], st["costs"], st["grads"])
        return {"cost": st["costs"], "grad": st["grads"]}
    if kind in ("batch", "hele_shaw", "uneven"):
        D.dvqls_cost_grad_batched(ctx, st["inst"], PRECISION[case.get("precision", "tc")], st["costs"], st["grads"])
        return {"cost": st["costs"], "grad": st["grads"]}
    if kind == "local":
        D.dvqls_local_cost_grad_batched(ctx, st["inst"], PRECISION[case["precision"]], st["costs"], st["grads"])
        return {"cost": st["costs"], "grad": st["grads"]}
    if kind == "dense":
        got = D.dvqls_pauli_decompose(ctx, st["in"], st["n"], case["tau"], case["L"], st["coef"], st["x"], st["z"])
        return {"counts": list(got), "coef": st["coef"], "x": st["x"], "z": st["z"]}
    if kind == "banded":
        got = D.dvqls_pauli_decompose_banded(ctx, st["n"], st["offsets"], st["in"], case["tau"], case["L"],
                                             st["coef"], st["x"], st["z"])
        return {"counts": list(got), "coef": st["coef"], "x": st["x"], "z": st["z"]}
    if kind == "solve":
        L, coef, x, z = st["lcu"]
        iters, _ = D.dvqls_lcu_solve_batched(ctx, case["n"], D.make_lcu(L, coef, x, z), case["nrhs"], st["b"], 1e-12,
                                             20000, st["x"])
        return {"x": st["x"], "iters": iters}
    if kind == "adam":
        res = D.dvqls_optimize(ctx, st["inst"], st["xhat"], st["adam"], st["alpha"])
        return {"alpha": st["alpha"], "cost": np.array([r.cost for r in res]),
                "fidelity": np.array([r.fidelity for r in res]), "iters": np.array([r.iters for r in res])}
    X, Y, M = st["data"]
    loss = D.dvqls_ws_train_step(st["net"], case["batch"], X, Y, M, LR)
    D.dvqls_ws_get_params(st["net"], st["params"])
    return {"loss": loss, "params": st["params"]}


# --------------------------------------------------------------------- work


def _cost_work(n, d, L, flavours=1):
    """One cost and gradient: 2P + 1 shifted evaluations of every term, a real
    product-sum of 2^n amplitudes each (beta_lm = conj beta_ml formed once), and
    the state of each evaluation by n (depth + 1) rotations."""
    N, P = 1 << n, n * (d + 1)
    S = 2 * P + 1
    return {"bytes": 24 * L + 16 * N + 8 * P + 8 * (P + 1),
            "flops": S * (2 * N * (flavours * L * (L + 1) // 2 + L) + 3 * N * P)}


def work(case):
    kind = case["kind"]
    if kind == "terms":
        n = case["n"]
        L = n * (n + 1) // 2 + 1  # about the terms of a tridiagonal matrix
        w = _cost_work(n, case["d"], 1 << n if n < 3 else L)
        w["bytes"] += 16 * L * (L + 1)
        return w
    if kind in ("batch", "local"):
        ns = [case["n_max"] - i % (case["n_max"] - case["n_min"] + 1) for i in range(case["count"])]
        ws = [_cost_work(n, case["d"], min(case["L"], 1 << n), n + 1 if kind == "local" else 1) for n in ns]
    elif kind == "hele_shaw":
        ws = [_cost_work(2 * int(math.log2(case["grid"])), case["d"], case["L"])] * case["count"]
    elif kind == "uneven":
        ns = [SMALL_SIZES[i % len(SMALL_SIZES)] for i in range(case["count"])] + [case["big_n"]] * case["big"]
        ws = [_cost_work(n, n // 2, min(48, 1 << n)) for n in ns]
        if case["big"] and case["big_n"] > 12:  # every shifted state once, in FP32
            P = case["big_n"] * (case["big_n"] // 2 + 1)
            ws[-1] = dict(ws[-1], bytes=ws[-1]["bytes"] + case["big"] * (2 * P + 1) * (8 << case["big_n"]))
    elif kind == "adam":
        w = _cost_work(case["n"], case["d"], case["L"])
        return {k: v * case["count"] * (case["steps"] + 1) for k, v in w.items()}
    elif kind == "banded":
        N, masks = 1 << case["n"], 1 + case["n"] * case["bands"]
        return {"bytes": 8 * N * (2 * case["bands"] + 1) + 24 * case["L"], "flops": masks * N * case["n"]}
    elif kind == "dense":
        N = case["grid"] ** 2
        n = 2 * int(math.log2(case["grid"]))
        return {"bytes": 8 * N * N + 24 * case["L"], "flops": (2 * n + 1) * N * n}
    elif kind == "solve":
        N = 1 << case["n"]
        distinct = min(case["L"], case["n"] + 1)  # X-masks; a complex vector by a real diagonal each
        return {"bytes": 32 * N * case["nrhs"] + 24 * case["L"],
                "flops": 40 * case["nrhs"] * N * (4 * distinct + 20)}
    else:
        B, I, H, O = case["batch"], warmstart.FEATURES, case["hidden"], warmstart.P_MAX
        p = H * I + H + H * H + H + O * H + O
        return {"bytes": 4 * (B * (I + 2 * O) + 7 * p), "flops": 2 * B * (3 * (H * H + O * H) + 2 * H * I) + 12 * p}
    return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}


# -------------------------------------------------------------------- exact


def _cplx(a, dev="cuda"):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.complex128).copy()).to(dev)


def _states(n, d, al):
    """psi(alpha) for rows of angles: Ry layers and CZ rings, real FP64 [rows, 2^n]."""
    N, B = 1 << n, al.shape[0]
    i = torch.arange(N, device="cuda")
    par = torch.zeros(N, dtype=torch.int64, device="cuda")
    pairs = [(q, q + 1) for q in range(n - 1)] + ([(n - 1, 0)] if n >= 3 else [])
    for p, q in pairs:
        par += ((i >> p) & 1) * ((i >> q) & 1)
    ring = (1 - 2 * (par & 1)).double()
    psi = torch.zeros(B, N, dtype=torch.float64, device="cuda")
    psi[:, 0] = 1.0
    for layer in range(d + 1):
        if layer:
            psi = psi * ring
        for k in range(n):
            t = 0.5 * al[:, layer * n + k]
            c, s = torch.cos(t)[:, None, None], torch.sin(t)[:, None, None]
            v = psi.view(B, N >> (k + 1), 2, 1 << k)
            lo, hi = v[:, :, 0], v[:, :, 1]
            psi = torch.stack((c * lo - s * hi, s * lo + c * hi), dim=2).view(B, N)
    return psi


def _parity(v):
    for k in (16, 8, 4, 2, 1):
        v = v ^ (v >> k)
    return v & 1


def _apply_all(n, s, psi):
    """A~ psi = sum_l c_l sigma_l psi, split into real and imaginary parts."""
    i = torch.arange(1 << n, device="cuda")
    c = s["coef"].view(np.complex128)
    re, im = torch.zeros_like(psi), None
    for l in range(s["L"]):
        x, z = int(s["x"][l]), int(s["z"][l])
        w = complex(c[l]) * 1j ** (bin(x & z).count("1") % 4)
        src = i ^ x
        v = psi[:, src] * (1 - 2 * _parity(src & z)).double()
        if w.real:
            re += w.real * v
        if w.imag:
            im = torch.zeros_like(psi) if im is None else im
            im += w.imag * v
    return re, im


def _cost_exact(s, local, base=None):
    """Cost and parameter-shift gradient of one system."""
    n, d = s["n"], s["d"]
    P, N = n * (d + 1), 1 << n
    al = torch.from_numpy(s["alpha"]).cuda() if base is None else base
    rows = al.repeat(2 * P + 1, 1)
    k = torch.arange(P, device="cuda")
    rows[1 + 2 * k, k] += 0.5 * math.pi
    rows[2 + 2 * k, k] -= 0.5 * math.pi
    b = _cplx(s["b"])
    b = b / torch.linalg.norm(b)
    num, den = [], []
    step = max(1, (1 << 25) >> n)
    for r in rows.split(step):
        re, im = _apply_all(n, s, _states(n, d, r))
        D_ = (re * re).sum(1) + (0 if im is None else (im * im).sum(1))
        if local:
            E = torch.zeros_like(D_)
            i = torch.arange(N, device="cuda")
            for j in range(n):
                E += (re * re[:, i ^ (1 << j)]).sum(1)
                if im is not None:
                    E += (im * im[:, i ^ (1 << j)]).sum(1)
            num.append(E / n)
        else:
            T = re @ b.real.contiguous() + 1j * -(re @ b.imag.contiguous())
            if im is not None:
                T = T + 1j * (im @ b.real.contiguous()) + im @ b.imag.contiguous()
            num.append(T.real ** 2 + T.imag ** 2)
        den.append(D_)
    num, den = torch.cat(num), torch.cat(den)
    f = (0.5, 0.5) if local else (1.0, 1.0)
    cost = f[0] - f[1] * num[0] / den[0]
    dn, dd = 0.5 * (num[1::2] - num[2::2]), 0.5 * (den[1::2] - den[2::2])
    grad = -f[1] * (dn * den[0] - num[0] * dd) / den[0] ** 2
    return cost.reshape(1), grad


def _terms_exact(s):
    n, N = s["n"], 1 << s["n"]
    psi = _states(n, s["d"], torch.from_numpy(s["alpha"]).cuda()[None])[0]
    i = torch.arange(N, device="cuda")
    phi = []
    for l in range(s["L"]):
        x, z = int(s["x"][l]), int(s["z"][l])
        src = i ^ x
        phi.append(1j ** (bin(x & z).count("1") % 4) * psi[src] * (1 - 2 * _parity(src & z)).double())
    phi = torch.stack(phi).to(torch.complex128)
    b = _cplx(s["b"])
    b = b / torch.linalg.norm(b)
    return (phi.conj() @ phi.T).reshape(-1), phi @ b.conj()


def _dense_of(s):
    """The matrix that an LCU (L, coef, x, z) of n qubits encodes."""
    n = s["n"]
    eye = torch.eye(1 << n, dtype=torch.float64, device="cuda")
    re, im = _apply_all(n, s, eye)  # row k: A~ e_k
    A = re.to(torch.complex128)
    return (A if im is None else torch.complex(re, im)).T.contiguous()


def _decompose_exact(case, seed):
    n, L_max = (_matrix(case, seed)[0], case["L"]) if case["kind"] == "dense" else (case["n"], case["L"])
    N = 1 << n
    i = torch.arange(N, device="cuda")
    diag = {}
    if case["kind"] == "dense":
        A = torch.from_numpy(_matrix(case, seed)[1]).cuda()
        at = torch.nonzero(A)
        for x in torch.unique(at[:, 0] ^ at[:, 1]).tolist():
            diag[x] = A[i ^ x, i]
    else:
        offsets, bands = _bands(case, seed)
        for o, row in zip(offsets, bands):  # A[r, r + o] = row[r]: column c = r + o is d_x(c) of x = r ^ c
            r = torch.arange(N, device="cuda")
            c = r + int(o)
            ok = (c >= 0) & (c < N)
            v = torch.from_numpy(row).cuda()
            r, c, v = r[ok], c[ok], v[ok]
            for x in torch.unique(r ^ c).tolist():
                m = ((r ^ c) == x) & (v != 0)
                if bool(m.any()):
                    d = diag.setdefault(x, torch.zeros(N, dtype=torch.float64, device="cuda"))
                    d[c[m]] = v[m]
    keys, vals, where = [], [], []
    for x in sorted(diag):
        w = diag[x].clone()
        h = 1
        while h < N:
            v = w.view(N // (2 * h), 2, h)
            w = torch.stack((v[:, 0] + v[:, 1], v[:, 0] - v[:, 1]), dim=1).reshape(N)
            h *= 2
        w = w / N
        vals.append(w)
        keys.append(w * w)
        where.append((x << n) | i)
    keys, vals, where = torch.cat(keys), torch.cat(vals), torch.cat(where)
    thr = case["tau"] * case["tau"] * keys.max()
    order = torch.argsort(where)
    order = order[torch.argsort(keys[order], descending=True, stable=True)]
    L = min(L_max, int((keys > thr).sum()))
    top = order[:L]
    x, z, v = where[top] >> n, where[top] & (N - 1), vals[top]
    k = torch.zeros_like(x)
    for q in range(n):
        k += ((x & z) >> q) & 1
    ph = torch.tensor([1, -1j, -1, 1j], dtype=torch.complex128, device="cuda")[k % 4]
    coef = torch.zeros(L_max, dtype=torch.complex128, device="cuda")
    coef[:L] = v * ph
    return coef


def _train_exact(case, seed):
    X, Y, M, p = _training(case, seed)
    I, H, O = warmstart.FEATURES, case["hidden"], warmstart.P_MAX
    X, Y, M = (torch.from_numpy(v).cuda().double() for v in (X, Y, M))
    sizes = [(H, I), (H,), (H, H), (H,), (O, H), (O,)]
    parts, at = [], 0
    p = torch.from_numpy(p).cuda().double()
    for sh in sizes:
        m = math.prod(sh)
        parts.append(p[at:at + m].view(sh).clone().requires_grad_())
        at += m
    W1, b1, W2, b2, W3, b3 = parts
    gelu = torch.nn.functional.gelu
    y = gelu(gelu(X @ W1.T + b1) @ W2.T + b2) @ W3.T + b3
    loss = (M * (y - Y) ** 2).sum() / M.sum()
    g = torch.cat([t.reshape(-1) for t in torch.autograd.grad(loss, parts)])
    return {"loss": float(loss), "params": p - LR * g / (g.abs() + 1e-8)}  # Adam's first step: m^ = g, v^ = g^2


def _adam_exact(case, systems):
    alphas, costs, fids = [], [], []
    for s in systems:
        x = torch.linalg.solve(_dense_of(s), _cplx(s["b"]))
        al = torch.from_numpy(s["alpha"]).cuda()
        m, v = torch.zeros_like(al), torch.zeros_like(al)
        for t in range(case["steps"] + 1):
            cost, g = _cost_exact(s, False, al)
            psi = _states(s["n"], s["d"], al[None])[0].to(torch.complex128)
            F = torch.abs(torch.vdot(x, psi)) ** 2 / torch.linalg.norm(x) ** 2
            if t < case["steps"]:
                m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
                al = al - 0.02 * (m / (1 - 0.9 ** (t + 1))) / (torch.sqrt(v / (1 - 0.999 ** (t + 1))) + 1e-8)
        alphas.append(al)
        costs.append(cost)
        fids.append(F.reshape(1))
    return {"alpha": torch.cat(alphas), "cost": torch.cat(costs), "fidelity": torch.cat(fids), "iters": None}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("banded", "dense"):
        return {"counts": None, "coef": _decompose_exact(case, seed), "x": None, "z": None}
    if kind == "train":
        return _train_exact(case, seed)
    h = Handle()  # the masks and coefficients are the case's input
    if kind == "solve":
        q = wl.throughput_instance(seed, n=case["n"], L_max=case["L"])
        L, coef, x, z = _lcu_banded(h.ctx, q, case["L"])
        A = _dense_of({"n": case["n"], "L": L, "coef": coef, "x": x, "z": z})
        B = torch.from_numpy(wl.gaussian_rhs(1 << case["n"], case["nrhs"], seed)).cuda().to(torch.complex128)
        return {"x": torch.view_as_real(torch.linalg.solve(A, B.T).T.contiguous()).reshape(-1), "iters": None}
    systems = _systems(h.ctx, case, seed)
    if kind == "adam":
        return _adam_exact(case, systems)
    got = [_cost_exact(s, kind == "local") for s in systems]
    out = {"cost": torch.cat([c for c, _ in got]), "grad": torch.cat([g for _, g in got])}
    if kind == "terms":
        out["beta"], out["delta"] = _terms_exact(systems[0])
    return out
