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


@pytest.mark.parametrize("prec", [0, 2, 3])
def test_direct_calls_around_a_launch_of_the_graph(dv, prec):
    """A launch of the graph leaves its own table in the workspace, and the context is not
    told: a direct call equal to the one before it brings its table again.  The same
    sums on the same inputs: equal bits."""
    n, d, L, count = 6, 1, 12, 2
    P = n * (d + 1)
    rng = np.random.default_rng(7)
    an = dv.make_ansatz(n, d)
    batches = []
    for k in range(2):  # the captured batch, and another one of the same shape
        keep, items = [], []
        for i in range(count):
            coef, xs, zs, b = random_problem(rng, n, L)
            t = [torch.tensor(v, device="cuda") for v in (cvec(coef), xs.view(np.int32), zs.view(np.int32), cvec(b),
                                                          wl.random_angles(P, 70 + 2 * k + i))]
            keep.append(t)
            items.append((an, dv.make_lcu(L, t[0], t[1], t[2]), t[4], t[3]))
        out = [torch.zeros(m, device="cuda", dtype=torch.float64) for m in (count, count * P)]
        batches.append((dv.make_instances(items), out, keep))
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    ctx = dv.dvqls_create(0, stream.cuda_stream)

    def taken(k):  # the results of batch k, which are cleared
        torch.cuda.synchronize()
        dv.dvqls_sync(ctx)
        r = [o.cpu().numpy().copy() for o in batches[k][1]]
        for o in batches[k][1]:
            o.zero_()
        torch.cuda.synchronize()
        return r

    def direct(k):
        dv.dvqls_cost_grad_batched(ctx, batches[k][0], prec, *batches[k][1])
        return taken(k)

    try:
        dv.dvqls_set_tuning(ctx, 1, 0)
        first = [direct(k) for k in range(2)]
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
            dv.dvqls_cost_grad_batched(ctx, batches[0][0], prec, *batches[0][1])
        for k in (1, 0, 1):
            for a, b in zip(first[k], direct(k)):
                assert np.array_equal(a, b)
            graph.replay()
            for a, b in zip(first[0], taken(0)):
                assert np.array_equal(a, b)
            for a, b in zip(first[k], direct(k)):
                assert np.array_equal(a, b)
    finally:
        dv.dvqls_destroy(ctx)
