"""bf16 planes of FP32 values at the top of FP32's range (tcgen05.cuh: plane_take)."""

from dataclasses import replace

import numpy as np
import pytest
import torch

import workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("where", ["input layer", "hidden layer", "weight"])
def test_values_above_the_largest_bf16(where):
    """3.4e38 lies between the largest bf16 and the largest FP32 value: as an activation
    of either kind of layer (g = 1: the identity) or as a weight it keeps its 24 bits.
    Bound: (K / 64 + 32) 2^-23 of sum |w| |h| for the plane GEMMs, as for other values; the
    factors beside it stay above 2^-109, below which planes hold fewer bits."""
    from paper_2509_13307_gb300 import Problem
    inp = w.make_cmb_inputs(replace(w.cmb6(n_ell=40), emu_hidden=(64, 64)))
    rng = np.random.default_rng(7)
    W, b = [np.zeros_like(q) for q in inp["emu_W"]], [np.ones_like(q) for q in inp["emu_b"]]
    inp.update(emu_W=W, emu_b=b, act_g=[np.ones_like(q) for q in inp["act_g"]],
               emu_out_mu=np.zeros_like(inp["emu_out_mu"]), emu_out_sig=np.ones_like(inp["emu_out_sig"]))
    big, small = 3.4e38, 1e-25
    W[2][:] = rng.standard_normal(W[2].shape)
    if where == "input layer":          # unit 0 is huge there and of order 1e13 behind
        b[0][0] = big
        W[1][:, 0] = small * rng.uniform(0.5, 1.0, 64)
    elif where == "hidden layer":
        b[1][0] = big
        W[2][:, 0] *= small
    else:
        b[1][0] = small
        W[2][:, 0] = np.where(np.arange(len(W[2])) % 2, big, -big)
    h = b[0].astype(np.float32).astype(float)
    f32 = [q.astype(np.float32).astype(float) for q in W]
    h = h @ f32[1].T + b[1].astype(np.float32)
    ref, mag = h @ f32[2].T + b[2], np.abs(h) @ np.abs(f32[2]).T + np.abs(b[2])
    D = len(ref)
    p = Problem(inp, "fp32", max_batch=3, data=np.zeros(D), cov=np.eye(D))
    theta = torch.tensor(np.tile(inp["fiducial"], (3, 1)), device="cuda")
    got = p.emulator(theta).cpu().numpy()
    assert np.all(np.abs(got - ref) <= 2 * 33 * 2.0 ** -23 * mag), np.max(np.abs(got - ref) / mag)
