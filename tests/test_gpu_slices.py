"""FP64 layers as fixed-point slices on the tensor cores (gemm_slices.cu) against
NumPy at the edges of their tiles: rows around the 32-row tile, widths that are
no multiple of 128 features, of a 32- or 128-deep block or of the 8-element row
pitch, and weight rows of very different size (one of them zero).

Bound per layer, propagated (tanh' <= 1): NumPy's own sum K 2^-53 of
sum_k |w| |h|, both operands' 2^-54 of their scale (1 for h, max |w| of the row
for w) and the dropped slice pairs, below 2^-53 of it each, over K terms."""

from dataclasses import replace

import numpy as np
import pytest
import torch

import workloads as w
from gpu_helpers import free_theta, random_cube

pytestmark = pytest.mark.gpu


def _reference(inp, full):
    h = (full[:, inp["emu_inputs"]] - inp["emu_in_center"]) / inp["emu_in_scale"]
    e = np.abs(h) * 2.0 ** -52
    Ws, bs = inp["emu_W"], inp["emu_b"]
    for l, (W, b) in enumerate(zip(Ws, bs)):
        K = W.shape[1]
        mag = np.abs(h) @ np.abs(W).T + np.abs(b)
        fixed = 4 * K * 2.0 ** -53 * np.abs(W).max(axis=1) if l else 0.0
        e = (K + 4) * 2.0 ** -53 * mag + fixed + e @ np.abs(W).T
        h = h @ W.T + b
        if l + 1 < len(Ws):
            h, e = np.tanh(h), e + 2.0 ** -51
    return inp["emu_out_mu"] + inp["emu_out_sigma"] * h, inp["emu_out_sigma"] * e + 2.0 ** -51 * np.abs(inp["emu_out_mu"])


def _problem(hidden, rows):
    from paper_2509_13307_gb300 import Problem
    inp = w.make_shear_inputs(replace(w.shear_tiny(), emu_hidden=hidden))
    W = inp["emu_W"][1]
    W *= 10.0 ** np.linspace(-3, 1, W.shape[0])[:, None]
    W[W.shape[0] // 2] = 0.0
    D = len(inp["noise_eps"])
    return inp, Problem(inp, "fp64", max_batch=max(rows, 3), data=np.zeros(D), cov=np.eye(D))


@pytest.mark.parametrize("hidden", [(192, 192), (100, 72), (20, 136), (130, 1028), (1024, 64)])
@pytest.mark.parametrize("rows", [1, 31, 33, 65])
def test_fp64_emulator_slices(hidden, rows):
    inp, p = _problem(hidden, rows)
    full = free_theta(inp, random_cube(rows, p.d, 5 + rows))
    got = p.emulator(torch.tensor(full, device="cuda")).cpu().numpy()
    ref, bound = _reference(inp, full)
    assert p.device_status() == 0
    assert np.all(np.abs(got - ref) <= bound), np.max(np.abs(got - ref) / bound)


def test_fp64_emulator_keeps_nan_in_its_row():
    inp, p = _problem((130, 1028), 5)
    full = free_theta(inp, random_cube(5, p.d, 3))
    clean = p.emulator(torch.tensor(full, device="cuda")).cpu().numpy()
    full[2, 3] = np.nan                                    # n_s: an input of the emulator only
    full[3, 3] = np.inf
    got = p.emulator(torch.tensor(full, device="cuda")).cpu().numpy()
    assert np.isnan(got[2]).all() and np.isfinite(got[3]).all()
    assert np.array_equal(got[[0, 1, 4]], clean[[0, 1, 4]])
