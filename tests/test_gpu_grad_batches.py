"""The log L that a gradient call returns does not depend on the batch that a row comes
in: on both sides of every rule by rows (K splits of the layers, rows per block of the
chi^2 stage, node ranges)."""

from dataclasses import replace

import numpy as np
import pytest
import torch

import workloads as w
from gpu_helpers import free_theta, random_cube

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["bf16", "fp32", "fp64"])
def test_log_l_of_a_gradient_call_is_its_rows_own(precision):
    from paper_2509_13307_gb300 import Problem
    rows = 1100
    inp = w.make_shear_inputs(replace(w.shear_tiny(), emu_hidden=(1024, 1024)))
    D = len(inp["noise_eps"])
    p = Problem(inp, precision, max_batch=rows, data=np.ones(D), cov=np.eye(D))
    theta = torch.tensor(free_theta(inp, random_cube(rows, p.d, 3)), device="cuda")
    whole, _ = p.loglike_grad(theta)
    for n in (1, 5, 33, 64, 100, 153, 400, 1023, 1024):
        assert torch.equal(p.loglike_grad(theta[:n])[0], whole[:n]), n
