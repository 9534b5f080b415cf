"""Gradient calls of one problem from two threads, on one stream and on a stream each:
every call reads its own parameters and writes its own results."""

import threading

import pytest
import torch

from gpu_helpers import cuda_problem, free_theta, oracle_for, random_cube

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["bf16", "fp64"])
@pytest.mark.parametrize("own_streams", [False, True])
def test_two_threads(precision, own_streams):
    p, ref = cuda_problem("shear_tiny", precision), cuda_problem("shear_tiny", precision)
    inp, _ = oracle_for("shear_tiny")
    sizes = (20, 27)                                     # one row bucket, one graph
    theta = [torch.tensor(free_theta(inp, random_cube(n, p.d, n)), device="cuda") for n in sizes]
    want = [ref.loglike_grad(t) for t in theta]
    p.loglike_grad(theta[0])                             # the gradient state is there before the threads start
    one = torch.cuda.Stream()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()] if own_streams else [one, one]
    torch.cuda.synchronize()
    bad = [None, None]

    def work(i):
        with torch.cuda.stream(streams[i]):
            wrong = 0
            for _ in range(150):
                log_l, grad = p.loglike_grad(theta[i])
                streams[i].synchronize()
                wrong += not (torch.equal(log_l, want[i][0]) and torch.equal(grad, want[i][1]))
            bad[i] = wrong

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert bad == [0, 0]
    assert p.device_status() == 0
