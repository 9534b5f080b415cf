"""FP64 slice GEMMs (gemm_slices.cu) outside the well-behaved middle of their range."""

from dataclasses import replace

import numpy as np
import pytest
import torch

import workloads as w
from gpu_helpers import free_theta, random_cube

pytestmark = pytest.mark.gpu


def _inputs(hidden, seed=0):
    """shear_tiny with random-normal layers of the given widths (fan-in scaled)."""
    inp = w.make_shear_inputs(replace(w.shear_tiny(), emu_hidden=hidden))
    rng = np.random.default_rng([seed, *hidden])
    dims = [len(inp["emu_inputs"]), *hidden, len(inp["emu_out_mu"])]
    inp["emu_W"] = [rng.standard_normal((n, k)) / np.sqrt(k) for k, n in zip(dims[:-1], dims[1:])]
    inp["emu_b"] = [0.1 * rng.standard_normal(n) for n in dims[1:]]
    return inp


def _problem(inp, rows):
    from paper_2509_13307_gb300 import Problem
    D = len(inp["noise_eps"])
    return Problem(inp, "fp64", max_batch=rows, data=np.zeros(D), cov=np.eye(D))


def _emulator(inp, full):
    h = (full[:, inp["emu_inputs"]] - inp["emu_in_center"]) / inp["emu_in_scale"]
    with np.errstate(invalid="ignore"):
        for W, b in zip(inp["emu_W"][:-1], inp["emu_b"][:-1]):
            h = np.tanh(h @ W.T + b)
        return inp["emu_out_mu"] + inp["emu_out_sigma"] * (h @ inp["emu_W"][-1].T + inp["emu_b"][-1])


@pytest.mark.parametrize("layer", [1, 2])
@pytest.mark.parametrize("rows", [1, 16, 64])
def test_nan_weight_marks_exactly_its_features(layer, rows):
    """A NaN seen by one CTA of a cluster that splits K, beside partial sums of
    either sign: a NaN weight of the output layer shows in its own outputs only, one
    of a hidden layer in all of them."""
    inp = _inputs((1024, 1024))
    W = inp["emu_W"][layer]
    rng = np.random.default_rng(layer)
    if layer == 2:
        for f in range(0, W.shape[0], 3):
            W[f, rng.integers(W.shape[1])] = np.nan
    else:
        W[700, 300] = np.nan
    p = _problem(inp, rows)
    full = free_theta(inp, random_cube(rows, p.d, rows))
    got = p.emulator(torch.tensor(full, device="cuda")).cpu().numpy()
    assert p.device_status() == 0
    assert np.array_equal(np.isnan(got), np.isnan(_emulator(inp, full)))


def _near_largest(rng, shape):
    """Values whose 9-bit digits lie in 250 .. 255 in all of the first five slices."""
    return sum(rng.integers(250, 256, shape) * 2.0 ** -(8 + 9 * i) for i in range(5))


@pytest.mark.parametrize("width", [1024, 1000])
def test_slices_near_their_largest_values(width):
    """Operands with every slice near its largest value and equal signs: the sums
    of 64 products still fit FP32's 24 bits where their unit matters, and a row's
    bits do not depend on the batch, which chooses the split of K.

    Bound, of the sum (about `width`): 2^-54 of the scale for each operand, one
    unit in the last place of tanh, the slice pairs left out (below 2^-50 of the
    scale in all), the roundings of the total, bias and output: under 2^-49."""
    inp = _inputs((width,))
    rng = np.random.default_rng(width)
    h = _near_largest(rng, width)
    inp["emu_W"][0][:] = 0.0
    inp["emu_b"][0][:] = np.arctanh(h)
    inp["emu_W"][1][:] = _near_largest(rng, inp["emu_W"][1].shape)
    inp["emu_b"][1][:] = 0.0
    inp["emu_out_mu"][:] = 0.0
    p = _problem(inp, 200)
    full = free_theta(inp, random_cube(200, p.d, 1))
    theta = torch.tensor(full, device="cuda")
    whole = p.emulator(theta)
    ld = np.longdouble
    ref = ld(inp["emu_out_sigma"]) * (np.tanh(inp["emu_b"][0]).astype(ld) @ inp["emu_W"][1].T.astype(ld))
    err = np.abs(whole.cpu().numpy().astype(ld) / ref - 1).max()
    assert err < 2.0 ** -49, float(err)
    for n in (1, 16, 17, 33, 64, 100):
        assert torch.equal(p.emulator(theta[:n]), whole[:n])


@pytest.mark.parametrize("width", [1024, 200])
@pytest.mark.parametrize("order", [1.0, 1e-3, 1e-6])
def test_small_activations_keep_fp64(width, order):
    """An output layer fed by activations of a given order: rows are scaled by their
    own power of two, so small activations keep their bits.

    Bound 2^-51 of sum |w| |h|: the digits' own error is below 2^-54 of it (K >= 200,
    normal weights and activations), tanh and the seven-term input sums of both sides
    2^-52 of each h (h's rms times 2^-52 sqrt(K) in the sum), the output 2^-53.  FP64 FMA
    chains stay near 2^-52; digits held against 1 were off by 2^-41 at order 1e-6."""
    inp = _inputs((width,))
    inp["emu_W"][0] *= order
    inp["emu_b"][0] *= order
    inp["emu_b"][1][:] = 0.0
    inp["emu_out_mu"][:] = 0.0
    rows = 40
    p = _problem(inp, rows)
    full = free_theta(inp, random_cube(rows, p.d, 3))
    got = p.emulator(torch.tensor(full, device="cuda")).cpu().numpy()
    ld = np.longdouble
    x = (full[:, inp["emu_inputs"]].astype(ld) - inp["emu_in_center"]) / inp["emu_in_scale"]
    h = np.tanh(x @ inp["emu_W"][0].T.astype(ld) + inp["emu_b"][0])
    W = inp["emu_W"][1].astype(ld)
    ref, mag = inp["emu_out_sigma"] * (h @ W.T), inp["emu_out_sigma"] * (np.abs(h) @ np.abs(W).T)
    err = float(np.max(np.abs(got - ref) / mag))
    print(f"width {width}, order {order}: {err:.2e}")
    assert err < 2.0 ** -51


def test_infinite_weights_act_as_in_fp64():
    """Infinite weights saturate tanh and make infinite outputs of the FP64 sums' signs."""
    inp = _inputs((256, 256))
    inp["emu_W"][1][17, 40] = np.inf
    inp["emu_W"][1][99, 3] = -np.inf
    inp["emu_W"][2][5, 7] = np.inf
    p = _problem(inp, 9)
    full = free_theta(inp, random_cube(9, p.d, 5))
    got = p.emulator(torch.tensor(full, device="cuda")).cpu().numpy()
    ref = _emulator(inp, full)
    assert p.device_status() == 0 and np.isinf(ref[:, 5]).all()
    assert np.allclose(got, ref, rtol=1e-11, atol=1e-11)


@pytest.mark.parametrize("large", [1e6, 1e150])
def test_outlying_weight_keeps_fp64(large):
    """One weight far above the others of its row, against an activation as far below
    its own: the other products keep their bits.  Bound 2^-49 of sum |w| |h|: sixteen
    rounding units, where an FP64 FMA chain of 1024 terms stays within three; digits held
    against the large weight are off by 2^-38 and more."""
    inp = _inputs((1024,))
    inp["emu_W"][1][:, 300] *= large
    inp["emu_W"][0][300] /= large
    inp["emu_b"][0][300] /= large
    inp["emu_b"][1][:] = 0.0
    inp["emu_out_mu"][:] = 0.0
    p = _problem(inp, 20)
    full = free_theta(inp, random_cube(20, p.d, 4))
    got = p.emulator(torch.tensor(full, device="cuda")).cpu().numpy()
    ld = np.longdouble
    x = (full[:, inp["emu_inputs"]].astype(ld) - inp["emu_in_center"]) / inp["emu_in_scale"]
    h = np.tanh(x @ inp["emu_W"][0].T.astype(ld) + inp["emu_b"][0])
    W = inp["emu_W"][1].astype(ld)
    ref, mag = inp["emu_out_sigma"] * (h @ W.T), inp["emu_out_sigma"] * (np.abs(h) @ np.abs(W).T)
    err = float(np.max(np.abs(got - ref) / mag))
    print(f"large {large}: {err:.2e}")
    assert err < 2.0 ** -49
