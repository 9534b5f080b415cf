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


def _bf16_weights(inp):
    """The same problem with the weights of layers >= 1 rounded to bf16: what a BF16 gradient differentiates."""
    from oracle.shear import ShearOracle
    return dict(inp, emu_W=[inp["emu_W"][0]] + [ShearOracle.to_bf16(W) for W in inp["emu_W"][1:]])


@pytest.mark.parametrize("precision,hidden", [("fp32", (100, 72)), ("fp32", (192, 192)), ("bf16", (136, 72)),
                                              ("bf16", (1024, 64))])
@pytest.mark.parametrize("rows", [1, 33, 260])
def test_gradient_tiles(precision, hidden, rows):
    """Gradients g_i = sum_a r_a J_ai / s_a^2 of a diagonal-covariance problem
    against the FP64 problem's (itself held to the complex step).  A model
    vector off by eps_m shifts g_i by eps_m sum_a |m_a J_ai| / s_a^2 (the terms
    cancel near the peak, this does not), and the adjoint's own chain is held to
    1e-5 of sum_a |r_a J_ai| / s_a^2; eps_m = 2e-6 is the FP32 stages' figure of
    the log-likelihood bounds, doubled for activations of 16 bits (BF16).  J by
    central differences of the FP64 model."""
    from paper_2509_13307_gb300 import Problem
    from paper_2509_13307_gb300.mock import diagonal_covariance
    inp = w.make_shear_inputs(replace(w.shear_tiny(), emu_hidden=hidden))
    ref_inp = _bf16_weights(inp) if precision == "bf16" else inp
    fid, D = np.asarray(inp["fiducial"], float), len(inp["noise_eps"])
    P = len(fid)
    model = Problem(ref_inp, "fp64", max_batch=2 * P, data=np.zeros(D), cov=np.eye(D))
    m0 = model.model(torch.tensor(fid[None], device="cuda"))[0].cpu().numpy()
    cov = diagonal_covariance(m0)
    sig2 = torch.tensor(np.diag(cov).copy(), device="cuda")
    data = m0 + np.sqrt(np.diag(cov)) * inp["noise_eps"]
    theta = fid + 0.1 * (free_theta(inp, random_cube(rows, P, 3 + rows)) - fid)
    theta = torch.tensor(theta, device="cuda")
    _, got = Problem(inp, precision, max_batch=rows, data=data, cov=cov).loglike_grad(theta)
    exact = Problem(ref_inp, "fp64", max_batch=rows, data=data, cov=cov)
    _, ref = exact.loglike_grad(theta)
    eps_m = 4e-6 if precision == "bf16" else 2e-6
    for b in range(0, rows, 32):                      # noise templates are free parameters too: their J counts
        h = 1e-5 * torch.clamp(theta[b].abs(), min=1e-2)
        steps = torch.diag(h)
        both = Problem(ref_inp, "fp64", max_batch=2 * P, data=data, cov=cov).model(
            torch.cat([theta[b] + steps, theta[b] - steps]))
        J = (both[:P] - both[P:]) / (2 * h[:, None])
        m = exact.model(theta[b:b + 1])[0]
        r = torch.tensor(data, device="cuda") - m
        bound = (eps_m * (m.abs() / sig2) @ J.abs().T + 1e-5 * (r.abs() / sig2) @ J.abs().T)
        ratio = float(((got[b] - ref[b]).abs() / bound).max())
        print(f"{precision} {hidden} row {b} of {rows}: error / bound = {ratio:.3f}")
        assert ratio <= 1.0


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_rows_do_not_depend_on_their_batch(precision):
    """The shards of a run evaluate their own chains: the same row gives the same
    bits in every batch size (every row tile, and both sides of the FP64 rules)."""
    from paper_2509_13307_gb300 import Problem
    inp = w.make_shear_inputs(replace(w.shear_tiny(), emu_hidden=(1024, 1024)))
    D, rows = len(inp["noise_eps"]), 400
    p = Problem(inp, precision, max_batch=rows, data=np.ones(D), cov=np.eye(D))
    theta = torch.tensor(free_theta(inp, random_cube(rows, p.d, 3)), device="cuda")
    whole = p.loglike(theta)
    for n in (1, 5, 33, 64, 100, 153, 250):
        assert torch.equal(p.loglike(theta[:n]), whole[:n])
