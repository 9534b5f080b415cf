"""FP32 layers as bf16-plane GEMMs (gemm_planes.cu) against FP64 NumPy at the
edges of their tiles: rows around the 32 / 64 / 128 row tiles, widths that are
no multiple of 128 features, of a 64-deep k-block or of the 8-element row
pitch, one k-block up to enough of them for every split over a cluster.

Bound per layer, propagated: a k-block's 24 MMA steps and the block sums each
lose at most one unit of 2^-23 of sum_k |w| |h|, the FP32 weight and bias
2^-24, tanhf and its rounding 4 x 2^-24; tanh' <= 1."""

from dataclasses import replace

import numpy as np
import pytest
import torch

import workloads as w
from gpu_helpers import free_theta, random_cube

pytestmark = pytest.mark.gpu


def _reference(inp, full):
    h = ((full[:, inp["emu_inputs"]] - inp["emu_in_center"]) / inp["emu_in_scale"])
    e = np.abs(h) * 2.0 ** -23
    Ws, bs = inp["emu_W"], inp["emu_b"]
    for l, (W, b) in enumerate(zip(Ws, bs)):
        mag = np.abs(h) @ np.abs(W).T + np.abs(b)
        e = ((W.shape[1] + 63) // 64 + 32) * 2.0 ** -23 * mag + e @ np.abs(W).T
        h = h @ W.T + b
        if l + 1 < len(Ws):
            h, e = np.tanh(h), e + 4 * 2.0 ** -24
    t = inp["emu_out_mu"] + inp["emu_out_sigma"] * h
    return t, inp["emu_out_sigma"] * e + 2.0 ** -22 * np.abs(t)


@pytest.mark.parametrize("hidden", [(192, 192), (100, 72), (20, 136), (130, 1028), (1024, 64)])
@pytest.mark.parametrize("rows", [1, 31, 33, 64, 129, 300])
def test_fp32_emulator_tiles(hidden, rows):
    from paper_2509_13307_gb300 import Problem
    inp = w.make_shear_inputs(replace(w.shear_tiny(), emu_hidden=hidden))
    D = len(inp["noise_eps"])
    p = Problem(inp, "fp32", max_batch=max(rows, 3), data=np.zeros(D), cov=np.eye(D))
    full = free_theta(inp, random_cube(rows, p.d, 7 + rows))          # every parameter of this model is free
    got = p.emulator(torch.tensor(full, device="cuda")).cpu().numpy()
    ref, bound = _reference(inp, full)
    assert p.device_status() == 0
    assert np.all(np.abs(got - ref) <= bound), np.max(np.abs(got - ref) / bound)
