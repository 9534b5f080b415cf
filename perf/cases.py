"""What a program does with this framework, as cases to time: single-call and
batched log-likelihoods of the cosmic-shear and CMB problems, gradients through
the autograd entry point, and whole nested-sampling iterations.

A case is a dict of plain values.  The sizes are the repository's own
(workloads/configs.py, the benchmark and the tests); the number of parameter
vectors B of a call ranges from 1 to 4096.

The entry points return float64 storage for every problem precision.  A program
that chose a reduced precision keeps the values in the type they are computed
in, so the outputs here are float32 for FP32 and BF16 problems (and gradients
arrive in the float32 of the parameters) and float64 for FP64 ones.
"""

from __future__ import annotations

import functools
import math

import numpy as np
import torch

import workloads as w
from paper_2509_13307_gb300 import NestedRun, Problem, loglike_autograd
from paper_2509_13307_gb300.mock import knox_covariance

C_OVER_100 = 2997.92458            # c / (100 km/s/Mpc) [Mpc]
LN_2PI = math.log(2.0 * math.pi)
SHEAR = {"shear39": w.shear39, "shear37_lcdm": w.shear37_lcdm, "shear39_interp": w.shear39_interp,
         "shear37_interp": w.shear37_interp, "shear39_interp_linear": w.shear39_interp_linear}


def listed():
    return [
        # one point: an optimiser's or a Metropolis chain's step; launches and latency count
        dict(name="loglike_bf16_1", do="loglike", model="shear39", precision="bf16", rows=1),
        # the batch of a nested-sampling round or of an importance-sampling pass (k = 500 chains)
        dict(name="loglike_bf16_500", do="loglike", model="shear39", precision="bf16", rows=500),
        # scoring a stored chain: the largest batch
        dict(name="loglike_bf16_4096", do="loglike", model="shear39", precision="bf16", rows=4096),
        # the nested LCDM model on the coarse-z emulator (interpolated P(k) runs), an odd batch
        dict(name="loglike_bf16_interp_375", do="loglike", model="shear37_interp", precision="bf16", rows=375),
        # the FP32 form: the evidence check's second precision
        dict(name="loglike_fp32_500", do="loglike", model="shear39", precision="fp32", rows=500),
        # the FP64 form: posterior points re-scored at full precision
        dict(name="loglike_fp64_64", do="loglike", model="shear39", precision="fp64", rows=64),
        # a lockstep NUTS leapfrog of 64 chains
        dict(name="grad_bf16_64", do="grad", model="shear39", precision="bf16", rows=64),
        # gradients of a large batch (variational fits, flow training)
        dict(name="grad_bf16_4096", do="grad", model="shear39", precision="bf16", rows=4096),
        # gradients at FP32, a mid-sized odd batch
        dict(name="grad_fp32_129", do="grad", model="shear39", precision="fp32", rows=129),
        # the CMB problem with the dense 7521 x 7521 covariance, a round of k = 250 chains
        dict(name="cmb_fold_fp32_250", do="cmb", form="gauss", n_ell=2507, precision="fp32", rows=250),
        # the cosmic-variance TT form on the tensor-core hidden layers, an odd batch
        dict(name="cmb_tt_bf16_333", do="cmb", form="tt_cv", n_ell=2507, precision="bf16", rows=333),
        # the sampler itself: set up a run, evolve it, read the live points back
        dict(name="nested_bf16_1000", do="nested", model="shear39", precision="bf16", n_live=1000, n_delete=500,
             repeats=10, iterations=2),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    do = rng.choice(["loglike", "loglike", "loglike", "grad", "grad", "cmb", "cmb", "nested"])
    if do == "cmb":
        form = rng.choice(["gauss", "tt_cv"])
        return dict(do="cmb", form=form, n_ell=_log_int(rng, 40, 835 if form == "gauss" else 2507),
                    precision=rng.choice(["fp32", "bf16", "fp32"]), rows=_log_int(rng, 1, 1000))
    model = rng.choice(sorted(SHEAR))
    if do == "nested":
        n_live = 2 * _log_int(rng, 50, 500)
        return dict(do="nested", model=model, precision="bf16", n_live=n_live, n_delete=n_live // 2,
                    repeats=rng.randint(4, 10), iterations=rng.randint(1, 2))
    precision = rng.choice(["bf16", "bf16", "bf16", "fp32", "fp32", "fp64"])
    most = {"bf16": 4096, "fp32": 1000, "fp64": 64} if do == "loglike" else {"bf16": 4096, "fp32": 300, "fp64": 24}
    return dict(do=do, model=model, precision=precision, rows=_log_int(rng, 1, most[precision]))


# ---------------------------------------------------------------- the inputs

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


@functools.lru_cache(maxsize=None)
def _shear_problem_inputs(model):
    """Configuration, emulator weights and mock observation of a shear model.
    Every model shares one observation: the fiducial spectra of shear39 plus
    one noise draw, with the Knox + low-rank covariance at those spectra."""
    inp = w.make_shear_inputs(SHEAR[model]())
    if model != "shear39":
        return (inp,) + _shear_problem_inputs("shear39")[1:]
    fid = torch.tensor(inp["fiducial"], dtype=torch.float64, device=_device())[None]
    m = _ShearExact(inp).model(fid)[0].cpu().numpy()
    cov = knox_covariance(m, inp["n_bins"], inp["ell"], inp["delta_ell"], inp["f_sky"],
                          inp["sigma_e"] ** 2 / inp["n_gal_sr"], inp["cov_V"], inp["cov_rank_amp"])
    return inp, m + np.linalg.cholesky(cov) @ inp["noise_eps"], cov


@functools.lru_cache(maxsize=2)
def _cmb_problem_inputs(n_ell, form):
    """Emulator weights and mock observation of the CMB problem: a seeded
    Wishart covariance scaled to the fiducial spectra (dense form), or
    cosmic-variance draws of the TT spectrum."""
    inp = w.make_cmb_inputs(w.cmb6(n_ell=n_ell))
    fid = torch.tensor(inp["fiducial"], dtype=torch.float64, device=_device())[None]
    m = _CmbExact(inp).emulator(fid)[0]
    if form == "tt_cv":
        return inp, m[:n_ell].cpu().numpy() * inp["tt_chi2"] / (2.0 * inp["ell"] + 1.0), None
    D, nu = int(inp["n_data"]), int(inp["wishart_nu"])
    gen = torch.Generator(device=_device()).manual_seed(int(inp["seed_cov"]))
    cov = torch.zeros(D, D, dtype=torch.float64, device=_device())
    for c in range(0, nu, 2048):
        a = torch.randn(D, min(2048, nu - c), dtype=torch.float64, device=_device(), generator=gen)
        cov += a @ a.T
    cov = 0.5 * (cov + cov.T)
    cov *= (inp["cov_rel"] ** 2 * (m * m).mean()) / cov.diagonal().mean()
    eps = torch.tensor(inp["noise_eps"], dtype=torch.float64, device=_device())
    data = m + torch.linalg.cholesky(cov) @ eps
    return inp, data.cpu().numpy(), cov.cpu().numpy()


def _points(inp, rows, seed):
    """Parameter vectors of all stages of a run: the fiducial point plus prior
    displacements shrunk by a factor between 1 (the start of a run) and 1/50
    (near the peak)."""
    rng = np.random.default_rng([int(seed), 17])
    free = [(i, p) for i, p in enumerate(inp["priors"]) if p[0] != "F"]
    fid = np.array([inp["fiducial"][i] for i, _ in free])
    u, g = rng.random((rows, len(free))), rng.standard_normal((rows, len(free)))
    a, b = np.array([p[1] for _, p in free]), np.array([p[2] for _, p in free])
    uniform = np.array([p[0] == "U" for _, p in free])
    prior = np.where(uniform, a + (b - a) * u, a + b * g)
    shrink = np.exp(rng.uniform(math.log(0.02), 0.0, (rows, 1)))
    return torch.tensor(fid + shrink * (prior - fid), dtype=torch.float64)


def _result_type(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def _case_points(case, inp, seed):
    theta = _points(inp, case["rows"], seed)
    if case["do"] == "grad":       # a training program's parameters have the type it works in
        theta = theta.to(_result_type(case))
    return theta.to(_device())


def prepare(case, seed):
    if case["do"] == "cmb":
        inp, data, cov = _cmb_problem_inputs(case["n_ell"], case["form"])
        problem = Problem(inp, case["precision"], max_batch=case["rows"], data=data, cov=cov, form=case["form"])
        return dict(case=case, problem=problem, theta=_case_points(case, inp, seed))
    inp, data, cov = _shear_problem_inputs(case["model"])
    if case["do"] == "nested":
        problem = Problem(inp, case["precision"], max_batch=case["n_live"], data=data, cov=cov)
        return dict(case=case, problem=problem, seed=int(seed))
    problem = Problem(inp, case["precision"], max_batch=case["rows"], data=data, cov=cov)
    theta = _case_points(case, inp, seed)
    return dict(case=case, problem=problem, theta=theta.requires_grad_(case["do"] == "grad"))


def run(state):
    case, problem = state["case"], state["problem"]
    kind = _result_type(case)
    if case["do"] == "nested":
        r = NestedRun(problem, case["n_live"], case["n_delete"], repeats=case["repeats"], seed=state["seed"])
        st = r.step(case["iterations"])
        x, log_l = r.live_points()
        r.close()
        return dict(x=x, log_l=log_l.astype(np.float32), log_z=st.logZ, log_x=st.logX, evaluations=st.evaluations,
                    rounds=st.rounds)
    if case["do"] == "grad":
        log_l = loglike_autograd(problem, state["theta"].double())
        (grad,) = torch.autograd.grad(log_l.sum(), state["theta"])
        return dict(log_l=log_l.detach().to(kind), grad=grad)
    return dict(log_l=problem.loglike(state["theta"]).to(kind))


def work(case):
    """Multiply-adds counted as two.  Bytes: weights in the problem's type,
    the observation's whitening matrix, parameters in, results out."""
    elt = {"bf16": 2, "fp32": 4, "fp64": 8}[case["precision"]]
    if case["do"] == "cmb":
        cfg = w.cmb6(n_ell=case["n_ell"])
        n_out = cfg.n_ell if case["form"] == "tt_cv" else cfg.n_data
        dims = list(cfg.emu_dims[:-1]) + [n_out]
        hidden = sum(a * b for a, b in zip(dims[:-2], dims[1:-1]))
        head = dims[-2] * n_out
        return dict(bytes=float(hidden * elt + head * max(4, elt) + case["rows"] * 8 * 7),
                    flops=float(case["rows"] * 2 * (hidden + head + n_out)))
    cfg = SHEAR[case["model"]]()
    dims, d = cfg.emu_dims, cfg.d_free
    weights = sum(a * b for a, b in zip(dims[:-1], dims[1:]))
    per = (2 * weights + 2 * cfg.n_ell * cfg.n_chi * (16 + cfg.n_pairs)
           + cfg.n_chi * (60 + 25 * cfg.n_bins) + cfg.n_data * (cfg.n_data + 1))
    fixed = weights * elt + cfg.n_data * (cfg.n_data + 1) // 2 * max(4, elt)
    if case["do"] == "nested":
        # a slice move takes the two ends of its slice and at least one point
        evals = case["n_live"] + case["iterations"] * case["n_delete"] * case["repeats"] * 3
        return dict(bytes=float(fixed + case["n_live"] * (d + 1) * 8), flops=float(evals * per))
    if case["do"] == "grad":
        return dict(bytes=float(fixed + case["rows"] * (2 * d + 1) * max(4, elt)), flops=float(3 * case["rows"] * per))
    return dict(bytes=float(fixed + case["rows"] * (8 * d + max(4, elt))), flops=float(case["rows"] * per))


# ------------------------------------------- the same quantities in plain FP64

class _ShearExact:
    """The shear model of arXiv:2509.13307 App. A in FP64 torch, batched over
    rows of full parameter vectors."""

    def __init__(self, inp):
        t = functools.partial(torch.tensor, dtype=torch.float64, device=_device())
        self.inp = inp
        n = int(inp["n_chi"])
        step = (1.0 - inp["a_min"]) / (n - 1)
        self.a = 1.0 - step * torch.arange(n, dtype=torch.float64, device=_device())
        self.ln_a, self.z = self.a.log(), 1.0 / self.a - 1.0
        self.wt = torch.full_like(self.a, step)
        self.wt[0] *= 0.5
        self.wt[-1] *= 0.5
        x, gw = np.polynomial.legendre.leggauss(4)
        self.gl_x, self.gl_w = t(x), t(gw)
        self.W, self.b = [t(q) for q in inp["emu_W"]], [t(q) for q in inp["emu_b"]]
        self.mu, self.sg = t(inp["nz_mean"])[:, None], t(inp["nz_sigma"])[:, None]
        self.center, self.scale, self.out_mu = t(inp["emu_in_center"]), t(inp["emu_in_scale"]), t(inp["emu_out_mu"])
        self.ln_ell = (t(inp["ell"]) + 0.5).log()
        nb = int(inp["n_bins"])
        self.pairs = [(i, j) for i in range(nb) for j in range(i, nb)]

    @staticmethod
    def _weights(u):
        return [0.5 * (-u + 2 * u ** 2 - u ** 3), 0.5 * (2 - 5 * u ** 2 + 3 * u ** 3),
                0.5 * (u + 4 * u ** 2 - 3 * u ** 3), 0.5 * (-u ** 2 + u ** 3)]

    @staticmethod
    def _pad(t, dim):
        """Ghost entries by linear extrapolation at both ends of an axis."""
        n = t.shape[dim]
        first, last = t.narrow(dim, 0, 1), t.narrow(dim, n - 1, 1)
        return torch.cat([2 * first - t.narrow(dim, 1, 1), t, 2 * last - t.narrow(dim, n - 2, 1)], dim)

    def _table(self, theta):
        inp = self.inp
        h = (theta[:, list(inp["emu_inputs"])] - self.center) / self.scale
        for W, b in zip(self.W[:-1], self.b[:-1]):
            h = torch.tanh(h @ W.T + b)
        t = self.out_mu + inp["emu_out_sigma"] * (h @ self.W[-1].T + self.b[-1])
        nzc, nz = int(inp["n_z_emu"]), int(inp["n_z"])
        t = t.reshape(-1, nzc, int(inp["n_k"]))
        if nzc == nz:
            return t
        u = torch.arange(nz, dtype=torch.float64, device=t.device) * ((nzc - 1) / (nz - 1))
        i = u.floor().clamp(0, nzc - 2).long()
        f = (u - i)[:, None]
        if inp["z_interp"] == "linear":
            return (1 - f) * t[:, i] + f * t[:, i + 1]
        p = self._pad(t, 1)
        return sum(wq * p[:, i + q] for q, wq in enumerate(self._weights(f)))

    def model(self, theta):
        inp, a, ln_a = self.inp, self.a, self.ln_a
        nb, n_k, nz = int(inp["n_bins"]), int(inp["n_k"]), int(inp["n_z"])
        col = lambda i: theta[:, i:i + 1]  # noqa: E731
        om, w0, wa, chi_h = (col(0) + col(1)) / col(2) ** 2, col(5), col(6), C_OVER_100 / col(2)

        def e2(s, ln_s):
            return om / s ** 3 + (1 - om) * torch.exp(-3 * (1 + w0 + wa) * ln_s - 3 * wa * (1 - s))

        E2 = e2(a, ln_a)
        E = E2.sqrt()
        mid, half = 0.5 * (a[:-1] + a[1:]), 0.5 * (a[:-1] - a[1:])
        inc = 0.0
        for x, g in zip(self.gl_x, self.gl_w):
            s = mid + half * x
            inc = inc + g / (s * s * e2(s, s.log()).sqrt())
        chi = torch.cumsum(chi_h * half * inc, 1)              # nodes 1 .. N - 1
        f = (om / (a ** 3 * E2)) ** (0.55 + 0.05 * (1 + w0 + 0.5 * wa))
        seg = 0.5 * (f[:, :-1] + f[:, 1:]) * (ln_a[:-1] - ln_a[1:])
        growth = torch.exp(-torch.cumsum(seg, 1))
        omw = self.wt * chi_h / (a * a * E)
        u = (self.z - theta[:, 11:11 + nb, None] - self.mu) / self.sg
        raw = torch.exp(-0.5 * u * u)
        nchi = raw * (E / chi_h)[:, None] / (self.wt / a ** 2 * raw).sum(2, keepdim=True)
        nchi, omw, a1, z1 = nchi[:, :, 1:], omw[:, 1:], a[1:], self.z[1:]
        wn = omw[:, None] * nchi
        tail = lambda q: q.flip(2).cumsum(2).flip(2) - q  # noqa: E731
        s0, s1 = tail(wn), tail(wn / chi[:, None])
        lens = (1.5 * om / chi_h ** 2 * chi / a1)[:, None] * (s0 - chi[:, None] * s1)
        amp = col(9) * ((1 + z1) / inp["ia_pivot"]) ** col(10) * inp["c1rho"] * om / growth
        V = (omw.sqrt() / chi)[:, None] * (lens - amp[:, None] * nchi)
        # P at (ell, node): Catmull-Rom in z at the nodes, then in ln k
        T = self._pad(self._pad(self._table(theta), 1), 2)
        uz = z1 / (inp["z_max"] / (nz - 1))
        j = uz.floor().clamp(0, nz - 2).long()
        rows = sum(wq[:, None] * T[:, j + q] for q, wq in enumerate(self._weights(uz - j)))
        s = (self.ln_ell[:, None] - chi.log()[:, None]).clamp(inp["lnk_min"], inp["lnk_max"])
        uk = (s - inp["lnk_min"]) * ((n_k - 1) / (inp["lnk_max"] - inp["lnk_min"]))
        i = uk.detach().floor().clamp(0, n_k - 2).long()
        wk = self._weights(uk - i)
        flat = rows.reshape(rows.shape[0], -1)
        base = (torch.arange(rows.shape[1], device=flat.device) * (n_k + 2))[None, None] + i
        shape = base.shape
        v = sum(wk[q] * flat.gather(1, (base + q).reshape(shape[0], -1)).reshape(shape) for q in range(4))
        X = torch.stack([V[:, p] * V[:, q] for p, q in self.pairs], 1)
        C = X @ torch.exp(v * math.log(10.0)).transpose(1, 2)
        bias = torch.stack([(1 + theta[:, 11 + nb + p]) * (1 + theta[:, 11 + nb + q]) for p, q in self.pairs], 1)
        return (bias[:, :, None] * C).reshape(theta.shape[0], -1)

    def log_l(self, theta, data, L, tmpl):
        nb = int(self.inp["n_bins"])
        m = self.model(theta) + theta[:, 11 + 2 * nb:] @ tmpl.T
        y = torch.linalg.solve_triangular(L, (data - m).T, upper=False)
        return -0.5 * (y * y).sum(0) - L.diagonal().log().sum() - 0.5 * L.shape[0] * LN_2PI


class _CmbExact:
    """The CMB problem's emulator in FP64 torch."""

    def __init__(self, inp):
        t = functools.partial(torch.tensor, dtype=torch.float64, device=_device())
        self.W, self.b = [t(q) for q in inp["emu_W"]], [t(q) for q in inp["emu_b"]]
        self.g, self.beta = [t(q) for q in inp["act_g"]], [t(q) for q in inp["act_beta"]]
        self.center, self.scale = t(inp["emu_in_center"]), t(inp["emu_in_scale"])
        self.mu, self.sig = t(inp["emu_out_mu"]), t(inp["emu_out_sig"])

    def emulator(self, theta):
        h = (theta - self.center) / self.scale
        for W, b, g, beta in zip(self.W, self.b, self.g, self.beta):
            x = h @ W.T + b
            h = (g + (1 - g) * torch.sigmoid(beta * x)) * x
        return self.mu + self.sig * (h @ self.W[-1].T + self.b[-1])


def exact(case, seed):
    if case["do"] == "nested":
        return None
    t = functools.partial(torch.tensor, dtype=torch.float64, device=_device())
    if case["do"] == "cmb":
        inp, data, cov = _cmb_problem_inputs(case["n_ell"], case["form"])
        m, d = _CmbExact(inp).emulator(_case_points(case, inp, seed)), t(data)
        if case["form"] == "tt_cv":
            k, c = 2.0 * t(inp["ell"]) + 1.0, m[:, :case["n_ell"]]
            x = k * d / c                          # chi^2 with k degrees of freedom
            return dict(log_l=((0.5 * k - 1) * x.log() - 0.5 * x - 0.5 * k * math.log(2.0) - torch.lgamma(0.5 * k)
                               + (k / c).log()).sum(1))
        L = torch.linalg.cholesky(t(cov))
        y = torch.linalg.solve_triangular(L, (d - m).T, upper=False)
        return dict(log_l=-0.5 * (y * y).sum(0) - L.diagonal().log().sum() - 0.5 * L.shape[0] * LN_2PI)
    inp, data, cov = _shear_problem_inputs(case["model"])
    model, L, d = _ShearExact(inp), torch.linalg.cholesky(t(cov)), t(data)
    tmpl = t(0.1 * np.sqrt(np.diag(cov))[:, None] * inp["tmpl_g"])
    free = [i for i, p in enumerate(inp["priors"]) if p[0] != "F"]
    full = t(np.array([p[1] if p[0] == "F" else 0.0 for p in inp["priors"]]))
    theta = _case_points(case, inp, seed).double()
    log_l, grad = [], []
    for rows in theta.split(128):
        rows = rows.clone().requires_grad_(case["do"] == "grad")
        x = full.repeat(rows.shape[0], 1).index_copy(1, torch.tensor(free, device=rows.device), rows)
        out = model.log_l(x, d, L, tmpl)
        if case["do"] == "grad":
            grad.append(torch.autograd.grad(out.sum(), rows)[0])
        log_l.append(out.detach())
    log_l = torch.cat(log_l)
    return dict(log_l=log_l, grad=torch.cat(grad)) if case["do"] == "grad" else dict(log_l=log_l)
