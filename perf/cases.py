"""The work that users of this library have it do, as cases that can be timed one by one.

Every case goes through the public Python entry points (``api``, ``autograd``, ``fit``) on
seeded synthetic EM stacks (``synthetic``).  Sizes are those of the library's own
configurations, tests and benchmark, or odd ones between them.  ``exact`` restates the method in
64-bit PyTorch, without the library.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1506_02079_gb300 import api, autograd, fit
from paper_1506_02079_gb300.synthetic import evaluate_stack, make_ragged_batch, stack_params


def listed():
    return [
        # The plain configuration: a stack small enough that launches and latency are the cost.
        {"name": "correct_16x256x256", "kind": "correct", "nz": 16, "ny": 256, "nx": 256, "dtype": "f32",
         "alpha": 0.01, "tol": 1e-6, "kappa": 0.0, "host": False},
        # The headline configuration: both phases on a stack resident on the GPU, the paper's alpha.
        {"name": "correct_64x2048x2048", "kind": "correct", "nz": 64, "ny": 2048, "nx": 2048, "dtype": "f32",
         "alpha": 0.001, "tol": 1e-6, "kappa": 0.0, "host": False},
        # A cropped 8-bit volume: odd width and height, so rows are unaligned and every level is ragged.
        {"name": "correct_u8_21x1187x1531", "kind": "correct", "nz": 21, "ny": 1187, "nx": 1531, "dtype": "u8",
         "alpha": 0.01, "tol": 1e-6, "kappa": 0.0, "host": False},
        # A volume that lives on the host: 8-bit in, float out, both in page-locked memory.
        {"name": "correct_host_u8_32x2048", "kind": "correct", "nz": 32, "ny": 2048, "nx": 2048, "dtype": "u8",
         "alpha": 0.001, "tol": 1e-6, "kappa": 0.0, "host": True},
        # The batched configuration (slices of mixed sizes in one packed call), a fifth of its slices.
        {"name": "solve_ragged_96", "kind": "batch", "nslices": 96, "lo": 256, "hi": 4096, "sizes": 2,
         "alpha": 0.001, "tol": 1e-6, "precision": "mixed"},
        # Fitting alpha and sigma_z: one forward and backward pass of the differentiation configuration.
        {"name": "train_32x512x512", "kind": "train", "nz": 32, "ny": 512, "nx": 512, "alpha": 0.001, "sigma_z": 2.5},
        # Phase 1 alone on an 8-bit volume, as a preprocessing pass.
        {"name": "smooth_u8_32x4096x3072", "kind": "smooth", "nz": 32, "ny": 4096, "nx": 3072, "dtype": "u8",
         "sigma_xy": 1.0, "sigma_z": 3.0, "kappa": 0.0},
        # Phase 1 with robust averaging on a stack with missing slices.
        {"name": "smooth_robust_48x1024x1536", "kind": "smooth", "nz": 48, "ny": 1024, "nx": 1536, "dtype": "f32",
         "sigma_xy": 1.0, "sigma_z": 3.0, "kappa": 2.0},
        # Colour / monochrome fusion of two images.
        {"name": "color_2x2048x3072", "kind": "color", "n": 2, "ny": 2048, "nx": 3072, "alpha": 0.001},
        # The direct (transform) solver on a uniform batch.
        {"name": "direct_16x1024x1024", "kind": "direct", "n": 16, "ny": 1024, "nx": 1024, "alpha": 0.001,
         "precision": "fp32"},
        # The 3-D gradient-domain smoothing, by transforms and by multigrid.
        {"name": "gd_direct_32x1024x1024", "kind": "gd_direct", "nz": 32, "ny": 1024, "nx": 1024, "dtype": "u8",
         "alpha": 0.1, "precision": "fp32"},
        {"name": "gd_multigrid_32x1024x1024", "kind": "gd_mg", "nz": 32, "ny": 1024, "nx": 1024, "dtype": "f32",
         "alpha": 0.1, "tol": 1e-6},
    ]


def _log(rng: random.Random, lo: float, hi: float) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _plane(rng: random.Random, lo: int, hi: int):
    """A slice: sides over [lo, hi], half of the time multiples of 4 (camera formats), else as cropped."""
    ny, nx = _log(rng, lo, hi), _log(rng, lo, hi)
    if rng.random() < 0.5:
        ny, nx = max(4, ny // 4 * 4), max(4, nx // 4 * 4)
    return ny, nx


def _depth(rng: random.Random, ny: int, nx: int, lo: int, hi: int, voxels: float) -> int:
    return max(1, min(_log(rng, lo, hi), int(voxels / (ny * nx))))


def draw(rng: random.Random):
    kind = rng.choice(["correct", "correct", "correct_host", "batch", "train", "smooth", "smooth", "robust", "color",
                       "direct", "gd_direct", "gd_mg"])
    alpha = rng.choice([0.001, 0.01, 0.1])
    dtype = rng.choice(["u8", "f32"])
    if kind == "correct":
        ny, nx = _plane(rng, 128, 4096)
        return {"kind": "correct", "nz": _depth(rng, ny, nx, 4, 96, 1.5e8), "ny": ny, "nx": nx, "dtype": dtype,
                "alpha": alpha, "tol": 1e-6, "kappa": rng.choice([0.0, 0.0, 0.0, 2.0]), "host": False}
    if kind == "correct_host":
        ny, nx = _plane(rng, 256, 4096)
        return {"kind": "correct", "nz": _depth(rng, ny, nx, 4, 64, 1.0e8), "ny": ny, "nx": nx, "dtype": dtype,
                "alpha": alpha, "tol": 1e-6, "kappa": 0.0, "host": True}
    if kind == "batch":
        precision = rng.choice(["mixed", "mixed", "mixed", "fp64"])
        hi = rng.choice([1024, 2048, 4096]) if precision == "mixed" else 512
        return {"kind": "batch", "nslices": _log(rng, 4, 96 if hi < 4096 else 48), "lo": 64, "hi": hi,
                "sizes": rng.randrange(1 << 20), "alpha": alpha,
                "tol": rng.choice([1e-6, 1e-6, 1e-9]) if precision == "mixed" else 1e-6, "precision": precision}
    if kind == "train":
        ny, nx = _plane(rng, 64, 768)
        return {"kind": "train", "nz": _depth(rng, ny, nx, 4, 48, 1.0e7), "ny": ny, "nx": nx,
                "alpha": rng.choice([0.001, 0.01]), "sigma_z": rng.choice([1.5, 2.5, 3.2])}
    if kind in ("smooth", "robust"):
        ny, nx = _plane(rng, 128, 6144)
        rob = kind == "robust"
        return {"kind": "smooth", "nz": _depth(rng, ny, nx, 4, 96, 7.5e7 if rob else 3.5e8), "ny": ny, "nx": nx,
                "dtype": dtype, "sigma_xy": rng.choice([1.0, 1.0, 0.5, 1.3]), "sigma_z": rng.choice([3.0, 3.0, 1.5, 2.5]),
                "kappa": 2.0 if rob else 0.0}
    if kind == "color":
        ny, nx = _plane(rng, 128, 4096)
        return {"kind": "color", "n": max(1, min(_log(rng, 1, 8), int(1.6e7 / (ny * nx)))), "ny": ny, "nx": nx,
                "alpha": alpha}
    ny, nx = _plane(rng, 96, 2048)
    if kind == "direct":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        return {"kind": "direct", "n": _depth(rng, ny, nx, 1, 64, 3.0e7 if precision == "fp32" else 6.0e6), "ny": ny,
                "nx": nx, "alpha": alpha, "precision": precision}
    nz = _depth(rng, ny, nx, 4, 96, 3.3e7)
    if kind == "gd_direct":
        return {"kind": "gd_direct", "nz": nz, "ny": ny, "nx": nx, "dtype": dtype, "alpha": rng.choice([0.01, 0.1]),
                "precision": "fp32"}
    return {"kind": "gd_mg", "nz": nz, "ny": ny, "nx": nx, "dtype": dtype, "alpha": rng.choice([0.05, 0.1]), "tol": 1e-6}


# ---------------------------------------------------------------- inputs
_DEV = "cuda"
_PRECISION = {"fp32": api.PREC_FP32, "mixed": api.PREC_MIXED, "fp64": api.PREC_FP64}


def _stack(case, seed):
    return evaluate_stack(stack_params(case["nz"], case["ny"], case["nx"], seed), device=_DEV, dtype=torch.float32,
                          out_dtype=torch.uint8 if case.get("dtype", "f32") == "u8" else torch.float32)


def _drop_slices(stack, seed):
    """Robust averaging is for stacks with damaged slices: one in sixteen is missing (zero)."""
    nz = stack.shape[0]
    for z in random.Random(seed).sample(range(nz), max(1, nz // 16)):
        stack[z].zero_()
    return stack


def _sides(case):
    r = random.Random(case["sizes"])
    return [(n, n) for n in (_log(r, case["lo"], case["hi"]) for _ in range(case["nslices"]))]


def _images(n, ny, nx, seed):
    """n colour images and their monochrome counterparts: the grey image has the fine structure,
    the colour channels are gained and offset versions of it."""
    grey = evaluate_stack(stack_params(n, ny, nx, seed), device=_DEV, dtype=torch.float32)
    rng = np.random.default_rng(seed)
    g = torch.as_tensor(rng.uniform(0.7, 1.2, size=(n, 3, 1, 1)), device=_DEV, dtype=torch.float32)
    c = torch.as_tensor(rng.uniform(-25.0, 25.0, size=(n, 3, 1, 1)), device=_DEV, dtype=torch.float32)
    rgb = (g * grey[:, None] + c).clamp_(0.0, 255.0)
    return rgb.contiguous(), grey


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("correct", "smooth", "gd_direct", "gd_mg"):
        st["stack"] = _stack(case, seed)
        if case.get("kappa", 0.0) > 0:
            _drop_slices(st["stack"], seed)
    if kind == "correct":
        st["opts"] = api.default_opts(tol=case["tol"], robust_kappa=case["kappa"])
        if case["host"]:
            host = torch.empty(st["stack"].shape, dtype=st["stack"].dtype, pin_memory=True)
            host.copy_(st["stack"])
            st["stack"] = host
            st["out"] = torch.empty(host.shape, dtype=torch.float32, pin_memory=True)
    elif kind == "batch":
        st["s"], st["o"], st["ny"], st["nx"], st["offsets"] = make_ragged_batch(
            case["nslices"], seed, device=_DEV, dtype=torch.float32, sides=_sides(case))
        st["opts"] = api.default_opts(tol=case["tol"], precision=_PRECISION[case["precision"]])
    elif kind == "train":
        st["stack"] = _stack(case, seed).requires_grad_(True)
        st["alpha"] = torch.tensor(case["alpha"], device=_DEV, requires_grad=True)
        st["sigma_z"] = torch.tensor(case["sigma_z"], device=_DEV, requires_grad=True)
    elif kind == "color":
        st["rgb"], st["grey"] = _images(case["n"], case["ny"], case["nx"], seed)
    elif kind == "direct":
        p = stack_params(case["n"], case["ny"], case["nx"], seed)
        st["s"] = evaluate_stack(p, device=_DEV, dtype=torch.float32, per_slice_gain=False)
        st["o"] = evaluate_stack(p, device=_DEV, dtype=torch.float32)
    elif kind == "gd_mg":
        st["opts"] = api.default_opts(tol=case["tol"])
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "correct":
        return api.emfuse_correct_stack(st["stack"], 1.0, 3.0, case["alpha"], st["opts"], out=st.get("out"))
    if kind == "smooth":
        if case["kappa"] > 0:
            return api.emfuse_smooth_z_robust(st["stack"], case["sigma_xy"], case["sigma_z"], case["kappa"])
        return api.emfuse_smooth_z(st["stack"], case["sigma_xy"], case["sigma_z"])
    if kind == "batch":
        return api.emfuse_screened_poisson(st["s"], st["o"], case["alpha"], st["opts"], nx=st["nx"], ny=st["ny"],
                                           offsets=st["offsets"])
    if kind == "train":
        f = autograd.correct_stack(st["stack"], st["alpha"], st["sigma_z"])
        loss = fit.interslice_loss(f)
        g = torch.autograd.grad(loss, (st["stack"], st["alpha"], st["sigma_z"]))
        return {"f": f.detach(), "loss": loss.detach(), "d_stack": g[0], "d_alpha": g[1], "d_sigma_z": g[2]}
    if kind == "color":
        return api.emfuse_fuse_color(st["rgb"], st["grey"], case["alpha"])
    if kind == "direct":
        return api.emfuse_screened_poisson_dct(st["s"], st["o"], case["alpha"], _PRECISION[case["precision"]])
    if kind == "gd_direct":
        return api.emfuse_smooth_gradient_domain(st["stack"], case["alpha"], _PRECISION[case["precision"]])
    return api.emfuse_smooth_gradient_domain_mg(st["stack"], case["alpha"], st["opts"])


def work(case):
    """Bytes: every input read once, every output written once.  Flops: the taps of the smoothing,
    and for the solves the multiplications and additions of one 5-point (7-point) operator and its
    update per cell, which no solver can do without."""
    kind = case["kind"]
    inp = 1 if case.get("dtype", "f32") == "u8" else 4
    if kind == "batch":
        cells = sum(a * b for a, b in _sides(case))
        return {"bytes": 12.0 * cells, "flops": 12.0 * cells}
    n = float(case["ny"]) * case["nx"] * (case.get("nz") or case["n"])
    taps = 2.0 * (2 * (2 * math.floor(3 * case.get("sigma_xy", 1.0) + 1e-9) + 1)
                  + 2 * math.floor(3 * case.get("sigma_z", 3.0) + 1e-9) + 1)
    if kind == "smooth":
        return {"bytes": (inp + 4.0) * n, "flops": taps * n}
    if kind == "correct":
        return {"bytes": (inp + 4.0) * n, "flops": (taps + 12.0) * n}
    if kind == "train":  # the stack in; f and the stack's gradient out
        return {"bytes": 12.0 * n, "flops": 2.0 * (taps + 12.0) * n}
    if kind == "color":  # three channels and the grey image in, three channels out
        return {"bytes": 28.0 * n, "flops": 36.0 * n}
    if kind == "direct":
        return {"bytes": 12.0 * n, "flops": 12.0 * n}
    return {"bytes": (inp + 4.0) * n, "flops": 16.0 * n}


# ---------------------------------------------------------------- 64-bit restatement
def _taps(sigma):
    sigma = float(np.float32(sigma))
    R = int(math.floor(3.0 * sigma + 1e-9))
    d = torch.arange(-R, R + 1, dtype=torch.float64)
    return R, (torch.exp(-d * d / (2.0 * sigma * sigma)) if sigma > 0 else torch.ones(1, dtype=torch.float64))


def _shifted_sum(x, axis, w, R):
    n = x.shape[axis]
    out = torch.zeros_like(x)
    for d in range(-R, R + 1):
        if abs(d) >= n:
            continue
        a, b = max(0, -d), min(n, n - d)
        out.narrow(axis, a, b - a).add_(x.narrow(axis, a + d, b - a), alpha=float(w[d + R]))
    return out


def _norms(n, w, R, axis, dev):
    v = _shifted_sum(torch.ones(n, dtype=torch.float64), 0, w, R)
    shape = [1, 1, 1]
    shape[axis] = n
    return v.view(shape).to(dev)


def _blur(x, axis, sigma, transpose=False):
    R, w = _taps(sigma)
    N = _norms(x.shape[axis], w, R, axis, x.device)
    return _shifted_sum(x / N, axis, w, R) if transpose else _shifted_sum(x, axis, w, R) / N


def _smooth(x, sigma_xy, sigma_z):
    return _blur(_blur(_blur(x, 2, sigma_xy), 1, sigma_xy), 0, sigma_z)


def _smooth_robust(x, sigma_xy, sigma_z, kappa):
    x = _blur(_blur(x, 2, sigma_xy), 1, sigma_xy)
    R, w = _taps(sigma_z)
    nz = x.shape[0]
    W = _norms(nz, w, R, 0, x.device)
    mu = _shifted_sum(x, 0, w, R) / W
    out = torch.empty_like(x)
    for z in range(nz):
        lo, hi = max(0, z - R), min(nz, z + R + 1)
        win, ww = x[lo:hi], w[lo - z + R:hi - z + R].to(x.device).view(-1, 1, 1)
        dev2 = (win - mu[z]) ** 2
        var = (ww * dev2).sum(0) / W[z]
        k = torch.where(dev2 <= kappa * kappa * var, ww, torch.zeros_like(ww))
        out[z] = (k * win).sum(0) / k.sum(0)
    return out


def _lap(x):
    """L x per slice: graph Laplacian on 4 neighbours, no flux across the slice's edges."""
    out = torch.zeros_like(x)
    for axis in (-1, -2):
        d = torch.diff(x, dim=axis)
        n = x.shape[axis]
        out.narrow(axis, 0, n - 1).sub_(d)
        out.narrow(axis, 1, n - 1).add_(d)
    return out


def _lam(n, m, dev):
    k = torch.arange(m, dtype=torch.float64, device=dev)
    return 4.0 * torch.sin(math.pi * k / (2.0 * n)) ** 2


def _solve(x, shift):
    """(shift I + L)^{-1} x of one slice, by the Fourier transform of its mirror extension."""
    ny, nx = x.shape
    e = torch.cat((x, x.flip(1)), 1)
    e = torch.cat((e, e.flip(0)), 0)
    F = torch.fft.rfft2(e)
    F /= shift + _lam(ny, 2 * ny, x.device)[:, None] + _lam(nx, nx + 1, x.device)[None, :]
    return torch.fft.irfft2(F, s=(2 * ny, 2 * nx))[:ny, :nx].contiguous()


def _poisson(s, o, alpha):
    """Eq. (1) per slice, f = o + alpha A^{-1}(s - o)."""
    f = torch.empty_like(o)
    for j in range(o.shape[0]):
        f[j] = o[j] + alpha * _solve(s[j] - o[j], alpha)
    return f


def _gradient_domain(x, alpha):
    """x + d with (alpha I + L_xy + L_z) d = -L_z x: the cosine transform along z, then slices."""
    nz = x.shape[0]
    k = torch.arange(nz, dtype=torch.float64, device=x.device)
    C = torch.cos(math.pi * k[:, None] * (2 * k[None, :] + 1) / (2 * nz)) * math.sqrt(2.0 / nz)
    C[0] /= math.sqrt(2.0)
    lz = _lam(nz, nz, x.device)
    y = (C @ x.reshape(nz, -1)).view(x.shape)
    for j in range(nz):
        y[j] = _solve(-lz[j] * y[j], alpha + float(lz[j]))
    return x + (C.T @ y.reshape(nz, -1)).view(x.shape)


def _train(x, alpha, sigma_z):
    alpha, sigma_z = float(np.float32(alpha)), float(np.float32(sigma_z))
    s = _smooth(x, 1.0, sigma_z)
    f = _poisson(s, x, alpha)
    d = f[1:] - f[:-1]
    loss = (d * d).mean()
    g = torch.zeros_like(f)
    g[1:] += 2.0 * d / d.numel()
    g[:-1] -= 2.0 * d / d.numel()
    lam = torch.stack([_solve(g[j], alpha) for j in range(g.shape[0])])
    t = alpha * lam
    dx = _lap(lam) + _blur(_blur(_blur(t, 0, sigma_z, True), 1, 1.0, True), 2, 1.0, True)
    # dK/dsigma_z at a fixed support: w'(d) = w(d) d^2 / sigma^3
    xy = _blur(_blur(x, 2, 1.0), 1, 1.0)
    R, w = _taps(sigma_z)
    dw = w * torch.arange(-R, R + 1, dtype=torch.float64) ** 2 / sigma_z ** 3
    N, dN = _norms(x.shape[0], w, R, 0, x.device), _norms(x.shape[0], dw, R, 0, x.device)
    dk = _shifted_sum(xy, 0, dw, R) / N - _shifted_sum(xy, 0, w, R) * dN / (N * N)
    return {"f": f, "loss": loss, "d_stack": dx, "d_alpha": (lam * (s - f)).sum(), "d_sigma_z": (t * dk).sum()}


def exact(case, seed):
    kind = case["kind"]
    st = prepare(case, seed)
    if kind == "smooth":
        x = st["stack"].double()
        if case["kappa"] > 0:
            return _smooth_robust(x, case["sigma_xy"], case["sigma_z"], case["kappa"])
        return _smooth(x, case["sigma_xy"], case["sigma_z"])
    if kind == "correct":
        x = st["stack"].to(_DEV).double()
        s = _smooth_robust(x, 1.0, 3.0, case["kappa"]) if case["kappa"] > 0 else _smooth(x, 1.0, 3.0)
        f = _poisson(s, x, case["alpha"])
        return f.cpu() if case["host"] else f
    if kind == "batch":
        f = torch.empty_like(st["s"], dtype=torch.float64)
        for (h, w), a in zip(_sides(case), st["offsets"].tolist()):
            s, o = (t[a:a + h * w].view(1, h, w).double() for t in (st["s"], st["o"]))
            f[a:a + h * w] = _poisson(s, o, case["alpha"]).reshape(-1)
        return f
    if kind == "train":
        return _train(st["stack"].detach().double(), case["alpha"], case["sigma_z"])
    if kind == "color":
        rgb, grey = st["rgb"].double(), st["grey"].double()
        return torch.stack([_poisson(rgb[:, c].contiguous(), grey, case["alpha"]) for c in range(3)], 1)
    if kind == "direct":
        return _poisson(st["s"].double(), st["o"].double(), case["alpha"])
    return _gradient_domain(st["stack"].double(), case["alpha"])
