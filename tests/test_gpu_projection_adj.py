"""The projection adjoint (projection_adj.cu) at the edges of its splits, in FP64
against the oracle's complex-step gradient (1e-9 of the largest component, as
for the other FP64 gradients): more multipoles than lanes, multipoles that share
a clamped ln k cell, out-of-order multipoles, fewer nodes than warps, nodes that
skip z cells, and row counts on both sides of each warps-per-evaluation rule and
of the rows-per-block rule of the chi^2 stage; in FP32, where bins
and taps go in packed pairs, against the FP64 gradient."""

from dataclasses import replace

import numpy as np
import pytest
import torch

import workloads as w
from gpu_helpers import free_theta, random_cube
from oracle.shear import ShearOracle

pytestmark = pytest.mark.gpu

VARIANTS = {
    "many_ell": dict(n_ell=40),
    "clamped": dict(n_ell=9, ell_min=0.5, ell_max=60000.0),
    "few_nodes": dict(n_chi=14),
    "skipped_cells": dict(n_chi=41, n_z=38),
    "one_bin": dict(n_bins=1, nz_mean=(0.8,), nz_sigma=(0.2,), n_ell=33),
    "wide_table": dict(n_k=4700, n_z=4, n_chi=14),     # table read from global memory, one warp per CTA
}


def _check(inp, orc, rows, picks):
    from paper_2509_13307_gb300 import Problem
    p = Problem(inp, "fp64", max_batch=rows, data=orc.data, cov=orc.cov)
    th = free_theta(inp, random_cube(rows, p.d, 11 + rows, 0.1, 0.9))
    t = torch.tensor(th, device="cuda")
    log_l, g = p.loglike_grad(t)
    again = p.loglike_grad(t)
    assert torch.equal(again[0], log_l) and torch.equal(again[1], g)     # fixed-order sums
    g, ll = g.cpu().numpy(), p.loglike(t).cpu().numpy()
    assert np.allclose(log_l.cpu().numpy(), ll, rtol=1e-12, atol=0)
    for b in picks:
        ref = orc.grad_complex_step(th[b])
        err = np.max(np.abs(g[b] - ref)) / np.max(np.abs(ref))
        assert err < 1e-9, (b, err, np.argmax(np.abs(g[b] - ref)))


@pytest.mark.parametrize("name", sorted(VARIANTS))
def test_gradient_variants(name):
    inp = w.make_shear_inputs(replace(w.shear_tiny(), **VARIANTS[name]))
    _check(inp, ShearOracle(inp), 3, range(3))


def test_gradient_unsorted_multipoles():
    inp = w.make_shear_inputs(w.shear_tiny())
    order = np.array([3, 0, 5, 1, 4, 2])
    inp = dict(inp, ell=inp["ell"][order], delta_ell=inp["delta_ell"][order])
    _check(inp, ShearOracle(inp), 2, range(2))


@pytest.mark.parametrize("rows", [76, 77, 152, 153, 1023, 1025])
def test_gradient_row_splits(rows):
    inp = w.make_shear_inputs(w.shear_tiny())
    _check(inp, ShearOracle(inp), rows, (0, rows - 1))


FP32_VARIANTS = {
    "odd_ell": dict(n_ell=9),
    "ell_33": dict(n_ell=33),
    "many_ell": dict(n_ell=64),
    "few_nodes": dict(n_chi=14),
    "skipped_cells": dict(n_chi=41, n_z=38),
    "one_bin": dict(n_bins=1, nz_mean=(0.8,), nz_sigma=(0.2,), n_ell=20),
    "wide_table": dict(n_k=2000, n_z=4),           # 32 KB of columns per warp
    "unsorted": dict(),
}


@pytest.mark.parametrize("rows", [2, 77, 154])
@pytest.mark.parametrize("name", sorted(FP32_VARIANTS))
def test_fp32_gradient_variants(name, rows):
    """FP32 gradients g_i = sum_a r_a J_ai / s_a^2 of a diagonal-covariance problem
    against the FP64 problem's: a model vector off by eps_m shifts g_i by
    eps_m sum_a |m_a J_ai| / s_a^2, the reverse chain is held to 1e-5 of
    sum_a |r_a J_ai| / s_a^2; eps_m = 2e-6 (twice the FP32 stages' figure of the
    log-likelihood bounds).  Both grow with the number of ln k cells, whose
    coordinate FP32 holds to 2^-24 of the range (24 cells in the tiny problem)."""
    from paper_2509_13307_gb300 import Problem
    from paper_2509_13307_gb300.mock import diagonal_covariance
    inp = w.make_shear_inputs(replace(w.shear_tiny(), **FP32_VARIANTS[name]))
    if name == "unsorted":
        order = np.array([3, 0, 5, 1, 4, 2])
        inp = dict(inp, ell=inp["ell"][order], delta_ell=inp["delta_ell"][order])
    fid, D = np.asarray(inp["fiducial"], float), len(inp["noise_eps"])
    P, cells = len(fid), FP32_VARIANTS[name].get("n_k", 24) / 24
    model = Problem(inp, "fp64", max_batch=2 * P, data=np.zeros(D), cov=np.eye(D))
    m0 = model.model(torch.tensor(fid[None], device="cuda"))[0].cpu().numpy()
    cov = diagonal_covariance(m0)
    sig2 = torch.tensor(np.diag(cov).copy(), device="cuda")
    data = m0 + np.sqrt(np.diag(cov)) * inp["noise_eps"]
    theta = fid + 0.1 * (free_theta(inp, random_cube(rows, P, 3 + rows)) - fid)
    theta = torch.tensor(theta, device="cuda")
    p = Problem(inp, "fp32", max_batch=rows, data=data, cov=cov)
    _, got = p.loglike_grad(theta)
    assert torch.equal(p.loglike_grad(theta)[1], got)              # fixed-order sums
    exact = Problem(inp, "fp64", max_batch=max(rows, 2 * P), data=data, cov=cov)
    _, ref = exact.loglike_grad(theta)
    for b in (0, rows - 1):
        steps = torch.diag(1e-5 * torch.clamp(theta[b].abs(), min=1e-2))
        both = exact.model(torch.cat([theta[b] + steps, theta[b] - steps]))
        J = (both[:P] - both[P:]) / (2 * torch.diagonal(steps)[:, None])
        m = exact.model(theta[b:b + 1])[0]
        r = torch.tensor(data, device="cuda") - m
        bound = cells * (2e-6 * (m.abs() / sig2) @ J.abs().T + 1e-5 * (r.abs() / sig2) @ J.abs().T)
        ratio = float(((got[b] - ref[b]).abs() / bound).max())
        print(f"{name} row {b} of {rows}: error / bound = {ratio:.3f}")
        assert ratio <= 1.0


@pytest.mark.parametrize("hidden", [(100, 72), (20, 136), (130, 1028), (64,)])
@pytest.mark.parametrize("rows", [1, 17, 33, 65])
def test_fp64_gradient_tiles(hidden, rows):
    """FP64 emulator layers around the 16, 32 and 64 row tiles of the backward pass,
    widths that are no multiple of 64 units or of a share of the contraction."""
    inp = w.make_shear_inputs(replace(w.shear_tiny(), emu_hidden=hidden))
    _check(inp, ShearOracle(inp), rows, (0, rows - 1))
