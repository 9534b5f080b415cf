"""Batches past the 65535 blocks that a grid's second dimension holds."""

import numpy as np
import pytest
import torch

from gpu_helpers import cuda_problem, free_theta, oracle_for, random_cube

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16"])
def test_log_likelihoods_of_66000_rows(precision):
    """Every row has the bits that it has in a small batch."""
    rows = 66000
    p, small = cuda_problem("shear_tiny", precision, max_batch=rows), cuda_problem("shear_tiny", precision)
    inp, _ = oracle_for("shear_tiny")
    base = free_theta(inp, random_cube(64, p.d, 5))
    theta = torch.tensor(np.tile(base, (rows // 64 + 1, 1))[:rows], device="cuda")
    got = p.loglike(theta)
    want = small.loglike(theta[:64])
    assert p.device_status() == 0
    assert torch.equal(got, want.repeat(rows // 64 + 1)[:rows])
