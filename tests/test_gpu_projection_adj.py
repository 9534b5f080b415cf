"""The projection adjoint (projection_adj.cu) at the edges of its splits, in FP64
against the oracle's complex-step gradient (1e-9 of the largest component, as
for the other FP64 gradients): more multipoles than lanes, multipoles that share
a clamped ln k cell, out-of-order multipoles, fewer nodes than warps, nodes that
skip z cells, and row counts on both sides of each warps-per-evaluation rule and
of the rows-per-block rule of the chi^2 stage."""

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
