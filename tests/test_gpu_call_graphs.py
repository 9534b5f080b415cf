"""Gradient calls replayed as graphs (CallGraphs) give what the launches one by one
give: the third and later calls of a row bucket against the first, with the row
count, the inputs, the output buffers and the stream changing from call to call;
more buckets than graphs are kept; and a call recorded into a graph of the
caller's own."""

import pytest
import torch

from gpu_helpers import cuda_problem, free_theta, oracle_for, random_cube

pytestmark = pytest.mark.gpu


def _theta(p, n, seed):
    inp, _ = oracle_for("shear_tiny")
    return torch.tensor(free_theta(inp, random_cube(n, p.d, seed)), device="cuda")


@pytest.mark.parametrize("precision", ["bf16", "fp32", "fp64"])
def test_replayed_calls_equal_first_calls(precision):
    p, fresh = cuda_problem("shear_tiny", precision), cuda_problem("shear_tiny", precision)
    sizes = [20, 32, 17, 31, 20, 32, 5, 8, 7, 6]          # buckets 32 and 8
    side = torch.cuda.Stream()
    for i, n in enumerate(sizes):
        th = _theta(p, n, i)
        want_l, want_g = fresh.loglike_grad(th)
        fresh = cuda_problem("shear_tiny", precision)     # every reference call is a first call
        torch.cuda.synchronize()
        with torch.cuda.stream(side if i % 2 else torch.cuda.current_stream()):
            got_l, got_g = p.loglike_grad(th)
        torch.cuda.synchronize()
        assert torch.equal(got_l, want_l) and torch.equal(got_g, want_g)
    assert p.device_status() == 0


def test_more_buckets_than_graphs():
    p, ref = cuda_problem("shear_tiny", "bf16", max_batch=300), cuda_problem("shear_tiny", "bf16", max_batch=300)
    th = _theta(p, 300, 1)
    sizes = (1, 2, 3, 8, 16, 30, 40, 60, 100, 200, 300)
    want = {n: ref.loglike_grad(th[:n]) for n in sizes}
    for _ in range(4):
        for n in sizes:
            got = p.loglike_grad(th[:n])
            assert torch.equal(got[0], want[n][0]) and torch.equal(got[1], want[n][1])


def test_call_inside_a_callers_graph():
    p, ref = cuda_problem("shear_tiny", "bf16"), cuda_problem("shear_tiny", "bf16")
    th = _theta(p, 20, 2)
    for _ in range(4):
        p.loglike_grad(th)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out, grad = p.loglike_grad(th)
    th.copy_(_theta(p, 20, 3))
    g.replay()
    torch.cuda.synchronize()
    want = ref.loglike_grad(th)
    assert torch.equal(out, want[0]) and torch.equal(grad, want[1])
