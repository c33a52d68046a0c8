"""A call whose workspace just fits the free memory is served: the spare quarter that the
workspace grows by is not a condition (the chain of the unshifted state has made the
workspace of states in HBM a few percent larger than the states alone)."""
import numpy as np
import pytest
import torch

from paper_2604_14435_gb300 import workloads as wl

from test_gpu_terms import cvec

pytestmark = pytest.mark.gpu


def test_workspace_without_room_to_spare(dv):
    n, d = 18, 20
    P = n * (d + 1)
    stream = torch.cuda.current_stream().cuda_stream
    c, xs, zs = cvec([1.0]), np.array([3], np.uint32), np.array([5], np.uint32)
    b, alpha = cvec(np.full(1 << n, 2.0 ** (-n / 2))), wl.random_angles(P, 1)

    def run(hold):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        ctx = dv.dvqls_create(0, stream)
        try:
            dv.dvqls_set_tuning(ctx, 1, 0)
            before = torch.cuda.mem_get_info()[0]
            kept = torch.empty(before - hold, dtype=torch.uint8, device="cuda") if hold else None
            cost, grad = np.zeros(1), np.zeros(P)
            dv.dvqls_cost_grad(ctx, dv.make_ansatz(n, d), alpha, dv.make_lcu(1, c, xs, zs), b, dv.DVQLS_FP32, cost, grad)
            used = before - torch.cuda.mem_get_info()[0] - (before - hold if hold else 0)
            del kept
            torch.cuda.empty_cache()
            return cost, grad, used
        finally:
            dv.dvqls_destroy(ctx)

    cost, grad, used = run(0)
    need = used / 1.25  # the workspace with its spare room (and little else)
    assert need > 7e8
    cost2, grad2, _ = run(int(1.12 * need))
    assert np.array_equal(cost, cost2) and np.array_equal(grad, grad2)
