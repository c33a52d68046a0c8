"""Cost passes that the caller captures into a CUDA graph of its own: the graph
brings its instance table with every launch, whatever the context has done since,
and a direct call after the capture uploads its own (the captured pass has not
run yet)."""
import numpy as np
import pytest
import torch

from oracle import terms as oterms
from paper_2604_14435_gb300 import workloads as wl

from test_gpu_terms import cvec, random_problem

pytestmark = pytest.mark.gpu

TOL = {0: (1e-12, 1e-12), 2: (1e-6, 1e-5), 3: (1e-6, 1e-5)}  # cost, gradient: as the direct calls


@pytest.mark.parametrize("prec,count", [(0, 1), (0, 33), (2, 3), (3, 3)])  # 33 records: more than one chunk of arguments
def test_captured_pass(dv, prec, count):
    n, d, L = 6, 1, 12
    P = n * (d + 1)
    rng = np.random.default_rng(5)
    probs, dev = [], []
    for i in range(count):
        coef, xs, zs, b = random_problem(rng, n, L)
        probs.append((coef, xs, zs, b))
        dev.append([torch.tensor(v, device="cuda") for v in (cvec(coef), xs.view(np.int32), zs.view(np.int32), cvec(b))])
    alpha = [wl.random_angles(count * P, 60 + k) for k in range(2)]
    al = torch.tensor(alpha[0], device="cuda")
    costs, grads = (torch.zeros(m, device="cuda", dtype=torch.float64) for m in (count, count * P))
    an = dv.make_ansatz(n, d)
    inst = dv.make_instances([(an, dv.make_lcu(L, t[0], t[1], t[2]), al[i * P:(i + 1) * P], t[3])
                              for i, t in enumerate(dev)])
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    ctx = dv.dvqls_create(0, stream.cuda_stream)

    def right(k):
        torch.cuda.synchronize()
        dv.dvqls_sync(ctx)
        c, g = costs.cpu().numpy(), grads.cpu().numpy()
        for i, (coef, xs, zs, b) in enumerate(probs):
            ref = oterms.cost_grad(n, d, alpha[k][i * P:(i + 1) * P], b, coef, xs, zs)
            assert abs(c[i] - ref["cost"]) <= TOL[prec][0] * max(1.0, abs(ref["cost"]))
            bound = TOL[prec][1] * (np.maximum(1.0, np.abs(ref["grad"])) if prec == 0 else 1.0)
            assert np.all(np.abs(g[i * P:(i + 1) * P] - ref["grad"]) <= bound)
        costs.zero_()
        grads.zero_()
        torch.cuda.synchronize()

    try:
        dv.dvqls_set_tuning(ctx, 1, 0)
        x = np.zeros(2 << 17)  # the workspace grows before the capture
        x[0] = 1.0
        dv.dvqls_fidelity(ctx, dv.make_ansatz(17, 0), np.zeros(17), x, np.zeros(1))
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
            dv.dvqls_cost_grad_batched(ctx, inst, prec, costs, grads)
        dv.dvqls_cost_grad_batched(ctx, inst, prec, costs, grads)  # the same pass, before the graph has run
        right(0)
        dv.dvqls_fidelity(ctx, dv.make_ansatz(17, 0), np.zeros(17), x, np.zeros(1))  # writes over the table
        al.copy_(torch.tensor(alpha[1]))
        torch.cuda.synchronize()
        graph.replay()
        right(1)
        dv.dvqls_cost_grad_batched(ctx, inst, prec, costs, grads)
        right(1)
    finally:
        dv.dvqls_destroy(ctx)
