"""The work that users of this library have it do, as cases that can be timed.

Every case goes through the public entry points (``paper_2406_18356_gb300``)
the way a program of a user does: a plan (or network) is built once, then the
calls of the method run on images and visibilities that already are on the
GPU.  The sizes are those of the repository's own workloads (``synth``,
``bench.py``): the 128-pixel FP64 observation of 31,744 rows, the 512-pixel
paper-like study of 241,920 rows, the 1024-pixel SKA-Mid-like observation of
9,266,880 rows and its multi-channel form, the 4096-pixel SKA-Low-like layout,
and the warm-start network at its configured shape (6 levels, width 6).

``exact`` states the same results in 64 bits with plain torch, without any of
the library's code: the gridded operator A = G F Z D with the
exponential-of-semicircle kernel, the concatenated Daubechies dictionary,
FISTA, the two-step method, and the U-Net.
"""
import functools
import math

import numpy as np
import torch

import paper_2406_18356_gb300 as ms

DEC, LAT = math.radians(-30.0), math.radians(-30.7)


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # one major-cycle residual image of the small plain-FP64 observation:
        # a call of a few short kernels, where launches and latency count
        {"name": "residual_128_fp64", "kind": "residual", "npix": 128, "precision": "fp64",
         "part": "ALL", "antennas": 32, "dumps": 64, "core": 0},
        # the major cycle of the SKA-Mid-like observation (9,266,880 rows):
        # where a reconstruction touches its visibilities
        {"name": "residual_1024_fp32", "kind": "residual", "npix": 1024, "precision": "fp32",
         "part": "ALL", "antennas": 197, "dumps": 480, "core": 1},
        # wide field with compensated sums (the precision form of the large
        # configuration): the biggest grid, rows of the long baselines only
        {"name": "residual_4096_kahan", "kind": "residual", "npix": 4096,
         "precision": "fp32_kahan", "part": "H", "antennas": 512, "dumps": 30, "core": 1},
        # multi-channel operator: both partitions of 8 unevenly flagged
        # channels through the batched calls (a major cycle of the channels)
        {"name": "channels_8x1024_fp32", "kind": "channels", "npix": 1024, "precision": "fp32",
         "channels": 8, "antennas": 197, "dumps": 60},
        # minor cycle of the small plain-FP64 observation (step one)
        {"name": "minor_low_128_fp64", "kind": "minor", "npix": 128, "precision": "fp64",
         "step": "low", "convolution": "circular", "iterations": 100, "warm": False,
         "antennas": 32, "dumps": 64, "core": 0},
        # the paper's 100 FISTA iterations on step two's problem at 1024
        # pixels, from a given start and with the coefficients returned: what
        # a reconstruction spends nearly all of its time on
        {"name": "minor_full_1024_fp32", "kind": "minor", "npix": 1024, "precision": "fp32",
         "step": "full", "convolution": "circular", "iterations": 100, "warm": True,
         "antennas": 64, "dumps": 120, "core": 1},
        # single-step problem on a wide image (coefficients well beyond L2)
        {"name": "minor_single_2048_fp32", "kind": "minor", "npix": 2048, "precision": "fp32",
         "step": "single", "convolution": "circular", "iterations": 25, "warm": False,
         "antennas": 64, "dumps": 120, "core": 1},
        # the linear reading of the PSF operator (the one with which the major
        # cycles converge), on an image side that is no power of two
        {"name": "minor_linear_448_fp32", "kind": "minor", "npix": 448, "precision": "fp32",
         "step": "low", "convolution": "linear", "iterations": 50, "warm": False,
         "antennas": 64, "dumps": 120, "core": 1},
        # step-one minor cycles of 8 channels in one batched call
        {"name": "minor_batch_8x1024_fp32", "kind": "minor_batch", "npix": 1024,
         "precision": "fp32", "channels": 8, "iterations": 50, "antennas": 64, "dumps": 24},
        # a whole two-step reconstruction at the study's size
        {"name": "two_step_512_fp32", "kind": "two_step", "npix": 512, "precision": "fp32",
         "majors": 2, "iterations": 50, "antennas": 64, "dumps": 120, "core": 1},
        # the warm-start network: inference on an evaluation image, and the
        # forward and backward pass of training with its gradients
        {"name": "net_forward_1024", "kind": "net_forward", "height": 1024, "width": 1024,
         "levels": 6, "channels": 6},
        {"name": "net_gradients_512", "kind": "net_gradients", "height": 512, "width": 512,
         "levels": 6, "channels": 6},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _side(rng, lo, hi, step):
    """An image side: half of them powers of two, the others multiples of `step`
    (16 for the operator; 64 for four wavelet levels on whole vectors)."""
    if rng.random() < 0.5:
        return 1 << rng.randint(math.ceil(math.log2(lo)), int(math.log2(hi)))
    return max(lo, _log_int(rng, lo, hi) // step * step)


def draw(rng):
    kind = rng.choice(["residual", "residual", "channels", "minor", "minor", "minor_batch",
                       "two_step", "net"])
    precision = rng.choice(["fp64", "fp32", "fp32", "fp32_kahan"])
    antennas, core = rng.randint(24, 96), rng.choice([0, 1])
    if kind == "residual":
        return {"kind": kind, "npix": _side(rng, 96, 2048, 16), "precision": precision,
                "part": rng.choice(["L", "H", "ALL"]), "antennas": rng.randint(24, 160),
                "dumps": _log_int(rng, 8, 240), "core": core}
    if kind == "channels":
        return {"kind": kind, "npix": _side(rng, 128, 1024, 16), "precision": precision,
                "channels": rng.randint(2, 8), "antennas": rng.randint(24, 128),
                "dumps": _log_int(rng, 8, 60)}
    if kind == "minor":
        linear = rng.random() < 0.25
        return {"kind": kind,
                "npix": _side(rng, 128, 512 if linear or precision == "fp64" else 1024, 64),
                "precision": precision, "step": rng.choice(["low", "full", "single"]),
                "convolution": "linear" if linear else "circular",
                "iterations": rng.randint(20, 60), "warm": rng.random() < 0.3,
                "antennas": antennas, "dumps": rng.randint(24, 120), "core": core}
    if kind == "minor_batch":   # (the batched form takes powers of two)
        return {"kind": kind, "npix": 1 << rng.randint(7, 10), "precision": "fp32",
                "channels": rng.randint(2, 8), "iterations": rng.randint(20, 50),
                "antennas": rng.randint(24, 64), "dumps": rng.randint(12, 24)}
    if kind == "two_step":
        return {"kind": kind, "npix": _side(rng, 128, 512, 64), "precision": "fp32",
                "majors": rng.randint(1, 2), "iterations": rng.randint(20, 50),
                "antennas": antennas, "dumps": rng.randint(24, 120), "core": core}
    levels, channels = rng.choice([(3, 16), (6, 6)])
    unit = 4 << (levels - 1)
    side = lambda hi: max(1, _log_int(rng, 128, hi) // unit) * unit  # noqa: E731
    kind = rng.choice(["net_forward", "net_gradients"])
    hi = 1024 if kind == "net_forward" else 512
    return {"kind": kind, "height": side(hi), "width": side(hi), "levels": levels,
            "channels": channels}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _rows(case):
    return case["antennas"] * (case["antennas"] - 1) // 2 * case["dumps"]


def _observation(case, seed, channels=1):
    """Earth-rotation tracks of a random array, one row per baseline and dump:
    u, v [channels, rows] in wavelengths, the pixel size that puts the longest
    baseline at npix / 3 cells of the image's DFT grid, and flags."""
    rng = np.random.default_rng(seed)
    n = case["antennas"]
    r = np.exp(rng.uniform(math.log(50.0), math.log(150e3), n)) if case.get("core", 1) else \
        1000.0 * np.sqrt(rng.random(n))
    th = 2 * np.pi * rng.random(n)
    i, j = np.triu_indices(n, k=1)
    e, nn = r * np.cos(th), r * np.sin(th)
    e, nn = e[j] - e[i], nn[j] - nn[i]
    ha = ((np.arange(case["dumps"]) + 0.5) / case["dumps"] * 8.0 - 4.0) * (2 * np.pi / 24.0)
    sh, ch = np.sin(ha)[:, None], np.cos(ha)[:, None]
    x, z = -math.sin(LAT) * nn, math.cos(LAT) * nn
    u = (sh * x + ch * e).ravel()
    v = (-math.sin(DEC) * ch * x + math.sin(DEC) * sh * e + math.cos(DEC) * z).ravel()
    scale = np.linspace(1.0 / 3.0, 1.0, channels) if channels > 1 else np.ones(1)
    u, v = u[None] * scale[:, None] * 4.27, v[None] * scale[:, None] * 4.27   # 1.28 GHz
    pixel = 1.0 / (3.0 * float(np.max(np.hypot(u, v))))
    flags = None
    if channels > 1:   # an uneven share of the rows of each channel is flagged
        share = rng.uniform(0.0, 0.5, channels)
        flags = (rng.random(u.shape) < share[:, None]).astype(np.uint8)
    return u, v, pixel, flags


def _split(case):
    """Partition centre and half width in pixels of the image's DFT grid."""
    frac = 0.10 if case["npix"] >= 1024 else 0.205
    return frac * case["npix"] / 3.0, 3.0


def _types(case):
    return (torch.float64, torch.complex128) if case["precision"] == "fp64" else \
        (torch.float32, torch.complex64)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _sky(npix, gen):
    """A few point sources per 64 x 64 pixels and some blobs, in the central half."""
    img = torch.zeros((npix, npix), dtype=torch.float64, device="cuda")
    count = max(4, (npix // 64) ** 2)
    at = torch.randint(npix // 4, 3 * npix // 4, (2, count), generator=gen, device="cuda")
    flux = 0.01 * torch.exp(math.log(100.0) * torch.rand(count, generator=gen, device="cuda",
                                                         dtype=torch.float64))
    img[at[0], at[1]] = flux
    k = torch.fft.rfftfreq(npix, device="cuda", dtype=torch.float64)
    k2 = torch.fft.fftfreq(npix, device="cuda", dtype=torch.float64)[:, None] ** 2 + k[None] ** 2
    blob = torch.fft.irfft2(torch.fft.rfft2(img.roll((npix // 9, npix // 7), (0, 1)))
                            * torch.exp(-2 * (math.pi * 1.5) ** 2 * k2), s=img.shape)
    return img + 2.0 * blob


def _visibilities(u, v, pixel, npix, dtype, gen):
    """Exact visibilities of a dozen point sources plus noise at SNR 30, and
    the model image of a later major cycle (most of their flux)."""
    lm = torch.randint(npix // 4, 3 * npix // 4, (12, 2), generator=gen, device="cuda")
    flux = 0.05 + torch.rand(12, generator=gen, device="cuda", dtype=torch.float64)
    model = torch.zeros((npix, npix), dtype=torch.float64, device="cuda")
    ud, vd = torch.as_tensor(u, device="cuda"), torch.as_tensor(v, device="cuda")
    vis = torch.zeros(ud.shape, dtype=torch.complex128, device="cuda")
    for s in range(12):
        p, q = int(lm[s, 0]), int(lm[s, 1])
        ph = (ud * (q - npix // 2) + vd * (p - npix // 2)) * (-2 * math.pi * pixel)
        vis += torch.polar(flux[s].expand_as(ph), ph)
        model[p, q] += 0.8 * float(flux[s])
    sigma = float(vis.abs().square().mean().sqrt()) / 30.0
    noise = torch.randn(ud.shape + (2,), generator=gen, device="cuda", dtype=torch.float64)
    vis += torch.view_as_complex(noise) * (sigma / math.sqrt(2))
    return vis.to(dtype).contiguous(), model


def _dirty(u, v, pixel, npix, dtype, gen):
    """A dirty image: the sky seen through the observation's own uv coverage
    (nearest cells of the image's DFT grid) plus noise."""
    at = [torch.remainder(torch.round(torch.as_tensor(a, device="cuda") * npix * pixel).long(), npix)
          for a in (v, u)]
    cover = torch.bincount(at[0] * npix + at[1], minlength=npix * npix).double()
    cover = cover.reshape(npix, npix) / u.size
    img = torch.fft.ifft2(torch.fft.fft2(_sky(npix, gen)) * cover).real
    noise = torch.randn((npix, npix), generator=gen, device="cuda", dtype=torch.float64)
    return (img + 0.02 * img.std() * noise).to(dtype).contiguous()


def _noise_variance(image):
    """Mean variance of the 5 x 5 windows (the method's noise estimate)."""
    x = image.double()[None, None]
    mean = torch.nn.functional.avg_pool2d(x, 5, 1)
    return float((torch.nn.functional.avg_pool2d(x * x, 5, 1) - mean * mean).mean())


def _plan(case, u, v, pixel, flags=None):
    ell, delta = _split(case)
    return ms.Plan(u, v, case["npix"], pixel, ell, delta, flags=flags,
                   precision=case["precision"], convolution=case.get("convolution", "circular"))


def _images(case, seed):
    """The images of a minor cycle, its lambda and (step two) its variances."""
    real, _ = _types(case)
    u, v, pixel, _ = _observation(case, seed)
    gen = _generator(seed)
    res = _dirty(u[0], v[0], pixel, case["npix"], real, gen)
    got = {"u": u, "v": v, "pixel": pixel, "residual": res,
           "lam": 0.05 * float(res.double().norm()) * 2.0, "l_low": None, "sigma2": 0.0,
           "eta2": 0.0, "beta": None}
    if case["step"] == "full":
        got["l_low"] = _dirty(u[0] * 0.2, v[0] * 0.2, pixel, case["npix"], real, gen)
        got["sigma2"] = _noise_variance(res)
        got["eta2"] = 1e-3 * got["sigma2"]
    if case["warm"]:
        start = torch.randn((8, case["npix"], case["npix"]), generator=gen, device="cuda")
        got["beta"] = (start * float(res.abs().mean()) * (start.abs() > 1.5)).to(real)
    return got


def _channel_jobs(case):
    return [(c, p) for c in range(case["channels"]) for p in ("L", "H")]


def _channel_inputs(case, seed):
    u, v, pixel, flags = _observation(case, seed, case["channels"])
    gen = _generator(seed)
    real, cplx = _types(case)
    vis, models = [], []
    for c in range(case["channels"]):
        a, b = _visibilities(u[c], v[c], pixel, case["npix"], cplx, gen)
        vis.append(a)
        models.append(b.to(real))
    return u, v, pixel, flags, vis, models


def _batch_inputs(case, seed):
    """Several channels' step-one problems: residual images and lambdas."""
    u, v, pixel, flags = _observation(case, seed, case["channels"])
    gen = _generator(seed)
    real, _ = _types(case)
    res = [_dirty(u[c], v[c], pixel, case["npix"], real, gen) for c in range(case["channels"])]
    return u, v, pixel, flags, res, [0.05 * float(r.double().norm()) * 2.0 for r in res]


def _net_parameters(case, seed):
    """He-normal weights and small biases, conv after conv in execution order."""
    rng = np.random.default_rng(seed)
    parts = []
    for co, ci in _net_shapes(case):
        parts.append(rng.standard_normal(co * 9 * ci) * math.sqrt(2.0 / (9 * ci)))
        parts.append(0.01 * rng.standard_normal(co))
    return np.concatenate(parts).astype(np.float32)


def _net_shapes(case):
    c, levels = case["channels"], case["levels"]
    shapes, ci = [], 2
    for lv in range(levels):
        shapes += [(c << lv, ci), (c << lv, c << lv)]
        ci = c << lv
    for lv in range(levels - 2, -1, -1):
        shapes += [(c << lv, (c << (lv + 1)) + (c << lv)), (c << lv, c << lv)]
    return shapes + [(1, c)]


def _net_images(case, seed):
    """[step-one image, long-baseline dirty image] at unit peak, and the sky."""
    gen = _generator(seed)
    n = max(case["height"], case["width"])
    sky = _sky(n, gen)
    k = torch.fft.rfftfreq(n, device="cuda", dtype=torch.float64)
    k2 = torch.fft.fftfreq(n, device="cuda", dtype=torch.float64)[:, None] ** 2 + k[None] ** 2
    low = torch.fft.irfft2(torch.fft.rfft2(sky) * torch.exp(-2 * (math.pi * 3.0) ** 2 * k2),
                           s=sky.shape)
    pair = torch.stack([low, sky - low], dim=-1)
    pair = pair + 0.02 * pair.std() * torch.randn(pair.shape, generator=gen, device="cuda",
                                                  dtype=torch.float64)
    peak = pair.abs().max()
    crop = lambda a: (a / peak)[:case["height"], :case["width"]].float().contiguous()  # noqa: E731
    return crop(pair), crop(sky)


# ---------------------------------------------------------------------------
# what a program has in hand, and what it calls
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    state = {"case": case}
    if kind in ("residual", "two_step"):
        real, cplx = _types(case)
        u, v, pixel, _ = _observation(case, seed)
        state["plan"] = _plan(case, u, v, pixel)
        state["vis"], model = _visibilities(u[0], v[0], pixel, case["npix"], cplx,
                                            _generator(seed))
        state["model"] = model.to(real)
    elif kind == "channels":
        u, v, pixel, flags, state["vis"], models = _channel_inputs(case, seed)
        state["plan"] = _plan(case, u, v, pixel, flags)
        state["jobs"] = _channel_jobs(case)
        state["models"] = [models[c] for c, _ in state["jobs"]]
        state["obs"] = [state["vis"][c] for c, _ in state["jobs"]]
        state["res"] = [torch.zeros_like(a) for a in state["obs"]]
    elif kind == "minor":
        state.update(_images(case, seed))
        state["plan"] = _plan(case, state.pop("u"), state.pop("v"), state.pop("pixel"))
    elif kind == "minor_batch":
        u, v, pixel, flags, res, lams = _batch_inputs(case, seed)
        state["plan"] = _plan(case, u, v, pixel, flags)
        state["jobs"] = [{"step": "low", "chan": c, "residual": r, "lam": lam}
                         for c, (r, lam) in enumerate(zip(res, lams))]
    else:
        state["net"] = ms.WarmStartNet(case["levels"], case["channels"],
                                       max(case["height"], case["width"]))
        state["net"].set_params(_net_parameters(case, seed))
        state["x"], state["target"] = _net_images(case, seed)
    return state


def run(state):
    case, plan = state["case"], state.get("plan")
    kind = case["kind"]
    if kind == "residual":
        return plan.residual_image(case["part"], state["vis"], state["model"])
    if kind == "channels":
        plan.degrid_batch(state["jobs"], state["models"], state["obs"], outs=state["res"])
        return {"images": plan.grid_batch(state["jobs"], state["res"]), "residuals": state["res"]}
    if kind == "minor":
        beta = state["beta"].clone() if case["warm"] else None
        model, _ = plan.minor_cycle(case["step"], state["residual"], state["lam"],
                                    case["iterations"], l_low=state["l_low"],
                                    sigma2=state["sigma2"], eta2=state["eta2"], beta=beta)
        return {"model": model, "beta": beta}
    if kind == "minor_batch":
        models, _ = plan.minor_cycle_batch(state["jobs"], case["iterations"])
        return {"models": models}
    if kind == "two_step":
        opts = ms.ReconOptions(n_major=case["majors"], fista_iters=case["iterations"])
        low, image, _ = plan.reconstruct_two_step(state["vis"], opts)
        return {"low": low, "image": image}
    if kind == "net_forward":
        return state["net"].forward(state["x"])
    out, loss, grads = state["net"].gradients(state["x"], state["target"])
    return {"out": out, "loss": loss, "grads": grads}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _operator_work(case, rows):
    """Residual image: the rows' places (one packed cell, two offsets), the
    observed values, two grids' worth of FFT and the images; 7 x 7 taps each
    way and the transforms' butterflies."""
    size = 8 if case["precision"] == "fp64" else 4
    n = case["npix"]
    grid = 4 * n * n
    taps = 2 * rows * 49 * 4 + 2 * rows * 14 * 12
    fft = 2 * 5 * grid * math.log2(grid)
    return rows * (4 + 2 * size + 2 * size) + 2 * n * n * size, taps + fft


def _iteration_work(case):
    """One FISTA iteration on M = 8 bases: the coefficients of this and the
    last iteration read, the next written; both transforms' taps (72 per
    output over the 8 bases, two directions, 4/3 for the coarser levels) and
    two image FFTs."""
    size = 8 if case["precision"] == "fp64" else 4
    n = case["npix"]
    flops = 2 * (4 * 72 * 4 / 3) * n * n + 16 * 8 * n * n + 2 * 2.5 * n * n * math.log2(n * n)
    if case.get("convolution") == "linear":
        flops += 4 * 2.5 * 4 * n * n * math.log2(4 * n * n)
    return 3 * 8 * n * n * size, flops


def work(case):
    kind = case["kind"]
    if kind in ("residual", "channels"):
        b, f = _operator_work(case, _rows(case))
        return {"bytes": b * case.get("channels", 1), "flops": f * case.get("channels", 1)}
    if kind in ("minor", "minor_batch"):
        b, f = _iteration_work(case)
        times = case["iterations"] * case.get("channels", 1)
        return {"bytes": b * times, "flops": f * times}
    if kind == "two_step":
        b, f = _iteration_work(case)
        ob, of = _operator_work(case, _rows(case))
        times, images = 2 * case["majors"] * case["iterations"], case["majors"] + 1
        return {"bytes": b * times + ob * images, "flops": f * times + of * images}
    # every layer's bfloat16 activations written and read once, its weights read
    size, flops, params = 0, 0, 0
    pixels = case["height"] * case["width"]
    levels = [lv for lv in range(case["levels"]) for _ in (0, 1)]
    levels += [lv for lv in range(case["levels"] - 2, -1, -1) for _ in (0, 1)] + [0]
    for (co, ci), lv in zip(_net_shapes(case), levels):
        p = pixels >> (2 * lv)
        size += 2 * p * (co + ci)
        flops += 2 * 9 * ci * co * p
        params += co * 9 * ci + co
    back = 3 if kind == "net_gradients" else 1
    return {"bytes": back * size + 12 * pixels + 4 * params * (1 + (back > 1)),
            "flops": back * flops}


# ---------------------------------------------------------------------------
# the same in 64 bits, with plain torch
# ---------------------------------------------------------------------------
class _Operator:
    """The gridded measurement operator of some rows: ES kernel of 7 cells,
    twofold oversampling, beta = 2.3 x 7."""

    def __init__(self, u, v, npix, pixel):
        self.n, self.ng, beta = npix, 2 * npix, 2.30 * 7
        t, w = np.polynomial.legendre.leggauss(400)
        a = np.arange(npix) - npix // 2
        phi = np.exp(beta * (np.sqrt(1.0 - t * t) - 1.0))
        psi = (np.cos(2 * np.pi * np.outer(a, 3.5 * t) / self.ng) * (3.5 * w * phi)).sum(1)
        self.psi = torch.as_tensor(np.outer(psi, psi), device="cuda")
        self.place = torch.as_tensor(a % self.ng, device="cuda")
        self.axes = []
        for x in (v, u):
            g = torch.as_tensor(x, device="cuda") * (self.ng * pixel)
            first = torch.floor(g - 3.5).long() + 1
            self.axes.append((first, g - first, beta))

    def _tap(self, axis, i):
        first, off, beta = self.axes[axis]
        z = (off - i) / 3.5
        return torch.remainder(first + i, self.ng), \
            torch.exp(beta * (torch.sqrt((1.0 - z * z).clamp_min(0.0)) - 1.0))

    def _taps(self):
        us = [self._tap(1, i) for i in range(7)]
        for j in range(7):
            cv, wv = self._tap(0, j)
            for cu, wu in us:
                yield cv * self.ng + cu, wv * wu

    def forward(self, image):
        pad = torch.zeros((self.ng, self.ng), dtype=torch.complex128, device="cuda")
        pad[self.place[:, None], self.place[None]] = (image / self.psi).to(torch.complex128)
        grid = torch.fft.fft2(pad).reshape(-1)
        out = torch.zeros(self.axes[0][0].shape, dtype=torch.complex128, device="cuda")
        for at, w in self._taps():
            out += w * grid[at]
        return out

    def dirty(self, vis):
        grid = torch.zeros((self.ng * self.ng, 2), dtype=torch.float64, device="cuda")
        pairs = torch.view_as_real(vis)
        for at, w in self._taps():
            grid.index_add_(0, at, w[:, None] * pairs)
        img = torch.fft.ifft2(torch.view_as_complex(grid).reshape(self.ng, self.ng),
                              norm="forward")
        img = img[self.place[:, None], self.place[None]].real
        return img / self.psi / max(1, vis.numel())

    def psf_spectrum(self):
        delta = torch.zeros((self.n, self.n), dtype=torch.float64, device="cuda")
        delta[self.n // 2, self.n // 2] = 1.0
        psf = self.dirty(self.forward(delta))
        return torch.fft.rfft2(torch.fft.ifftshift(psf)).real


def _part(u, v, case, pixel, part, flags=None):
    """Rows of a baseline partition."""
    ell, delta = _split(case)
    r = np.hypot(u, v) * case["npix"] * pixel
    keep = {"L": r <= ell + delta, "H": r >= ell - delta, "ALL": r >= 0}[part]
    return keep if flags is None else keep & (flags == 0)


@functools.lru_cache(None)
def _daubechies(p):
    """The 2p taps of db_p: the roots of sum_k C(p-1+k, k) y^k give the zeros
    outside the unit circle of z + 1/z = 2 - 4 y, beside p zeros at -1."""
    zeros = np.full(p, -1.0 + 0j)
    if p > 1:
        poly = np.array([math.comb(p - 1 + k, k) for k in range(p)][::-1], dtype=float)
        y = np.roots(poly)
        for _ in range(4):
            y = y - np.polyval(poly, y) / np.polyval(np.polyder(poly), y)
        s = 1.0 - 2.0 * y
        z = s + np.sqrt(s * s - 1.0)
        zeros = np.concatenate([zeros, np.where(np.abs(z) < 1.0, 1.0 / z, z)])
    h = np.poly(zeros).real[::-1]
    return h * (math.sqrt(2.0) / h.sum())


def _taps_of(m):
    """Low- and high-pass taps of basis m (db_m+1)."""
    h = _daubechies(m + 1)
    return h, [(-1) ** k * h[len(h) - 1 - k] for k in range(len(h))]


def _split_axis(x, m):
    """One periodized analysis level along the last axis: [low | high]."""
    n, (h, g) = x.shape[-1], _taps_of(m)
    wrapped = x[..., torch.arange(n + len(h), device="cuda") % n]
    halves = torch.zeros((2,) + x.shape[:-1] + (n // 2,), dtype=x.dtype, device="cuda")
    for k in range(len(h)):
        part = wrapped[..., k:k + n:2]
        halves[0].add_(part, alpha=float(h[k]))
        halves[1].add_(part, alpha=float(g[k]))
    return torch.cat([halves[0], halves[1]], -1)


def _join_axis(y, m):
    """The transpose of _split_axis."""
    n, (h, g) = y.shape[-1], _taps_of(m)
    room = -(-(n + len(h)) // n) * n
    out = torch.zeros(y.shape[:-1] + (room,), dtype=y.dtype, device="cuda")
    for k in range(len(h)):
        out[..., k:k + n:2].add_(y[..., :n // 2], alpha=float(h[k]))
        out[..., k:k + n:2].add_(y[..., n // 2:], alpha=float(g[k]))
    return out.reshape(y.shape[:-1] + (room // n, n)).sum(-2)


def _analysis(x, levels=4):
    y = x.expand(8, *x.shape).clone()
    for m in range(8):
        n = x.shape[0]
        for _ in range(levels):
            y[m, :n, :n] = _split_axis(_split_axis(y[m, :n, :n], m).T, m).T
            n //= 2
    return y


def _synthesis(a, levels=4):
    out = torch.zeros(a.shape[1:], dtype=a.dtype, device="cuda")
    for m in range(8):
        y = a[m].clone()
        n = a.shape[1] >> (levels - 1)
        for _ in range(levels):
            y[:n, :n] = _join_axis(_join_axis(y[:n, :n].T, m).T, m)
            n *= 2
        out += y
    return out


def _filters(case, sigma2, eta2):
    """g_L^2, g_H^2 on the half plane: the sine transition around ell."""
    ell, delta = _split(case)
    n = case["npix"]
    kx = torch.fft.rfftfreq(n, device="cuda", dtype=torch.float64) * n
    ky = torch.fft.fftfreq(n, device="cuda", dtype=torch.float64) * n
    r = torch.sqrt(ky[:, None] ** 2 + kx[None] ** 2)
    s = torch.sin(math.pi * ((r - ell) / delta).clamp(-1, 1) / 2)
    a2 = 1.0 / (eta2 * (1 - s) ** 2 + sigma2 * (1 + s) ** 2)
    return a2 * (1 - s) ** 2, a2 * (1 + s) ** 2


def _filtered(x, response):
    return torch.fft.irfft2(torch.fft.rfft2(x) * response, s=x.shape)


def _psf_operator(case, u, v, pixel):
    """The PSF operator H, and its spectrum in the circular reading."""
    n = case["npix"]
    if case.get("convolution") == "linear":
        spec = _Operator(u, v, 2 * n, pixel).psf_spectrum()

        def linear(x):
            y = torch.zeros((2 * n, 2 * n), dtype=torch.float64, device="cuda")
            y[:n, :n] = x
            return _filtered(y, spec)[:n, :n]
        return linear, None
    spec = _Operator(u, v, n, pixel).psf_spectrum()
    return lambda x: _filtered(x, spec), spec


def _power_start(count):
    """SplitMix64 (Steele, Lea and Flood 2014) from 12345, mapped to [-1, 1)."""
    with np.errstate(over="ignore"):
        z = np.uint64(12345) + np.uint64(0x9E3779B97F4A7C15) * np.arange(1, count + 1, dtype=np.uint64)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    z = z ^ (z >> np.uint64(31))
    return torch.as_tensor((z >> np.uint64(11)).astype(np.float64) * 2.0 ** -52 - 1.0, device="cuda")


def _fista(case, psf, residual, lam, iterations, l_low=None, sigma2=0.0, eta2=0.0, beta=None):
    """Algorithm 1 on the LowRes / FullRes problem: (model, beta)."""
    H, spec = psf
    res = residual.double()
    if l_low is None:
        normal = lambda x: H(H(x))  # noqa: E731
        b = H(res)
        top = None if spec is None else float((spec * spec).max())
    else:
        gl2, gh2 = _filters(case, sigma2, eta2)
        low = l_low.double()
        normal = lambda x: H(_filtered(H(x), gh2)) + _filtered(x, gl2)  # noqa: E731
        b = H(_filtered(res, gh2)) + _filtered(low, gl2)
        top = None if spec is None else float((gh2 * spec * spec + gl2).max())
    shape = (8,) + tuple(res.shape)
    if top is not None:
        theta = 2.0 * 8 * top
    else:   # not circulant: 100 power iterations from a fixed start
        w = _power_start(8 * res.numel()).reshape(shape)
        for _ in range(100):
            x = w / w.norm()
            w = _analysis(normal(_synthesis(x)))
            theta = 2.0 * float((x * w).sum())
    cur = torch.zeros(shape, dtype=torch.float64, device="cuda") if beta is None else beta.double()
    prev = cur
    for k in range(iterations):
        t = (k - 1.0) / (k + 2.0) if k > 1 else 0.0
        alpha = cur + t * (cur - prev)
        z = alpha - (2.0 / theta) * _analysis(normal(_synthesis(alpha)) - b)
        prev, cur = cur, torch.sign(z) * (z.abs() - lam / theta).clamp_min(0.0)
    return _synthesis(cur), cur


def _exact_two_step(case, seed):
    u, v, pixel, _ = _observation(case, seed)
    vis, _ = _visibilities(u[0], v[0], pixel, case["npix"], _types(case)[1], _generator(seed))
    vis = vis.to(torch.complex128)
    done = {}
    for part in ("L", "H"):
        keep = _part(u[0], v[0], case, pixel, part)
        op = _Operator(u[0][keep], v[0][keep], case["npix"], pixel)
        obs = vis[torch.as_tensor(keep, device="cuda")]
        psf = _psf_operator(case, u[0][keep], v[0][keep], pixel)
        model = torch.zeros((case["npix"],) * 2, dtype=torch.float64, device="cuda")
        more = {}
        for n in range(1, case["majors"] + 1):
            res = op.dirty(obs - op.forward(model))
            if part == "H":
                s2 = _noise_variance(res) if n == 1 else more["sigma2"]
                more = {"l_low": done["L"] - model, "sigma2": s2, "eta2": 1e-3 * s2}
            lam = 0.05 * float(res.norm()) * 2.0 ** n
            model = model + _fista(case, psf, res, lam, case["iterations"], **more)[0]
        done[part] = op.dirty(obs - op.forward(model)) + model
    return {"low": done["L"], "image": done["H"]}


def _exact_net(case, seed):
    F = torch.nn.functional
    params = torch.as_tensor(_net_parameters(case, seed), device="cuda").double().requires_grad_()
    x, target = _net_images(case, seed)
    shapes, at = iter(_net_shapes(case)), [0]

    def conv(a):
        co, ci = next(shapes)
        w = params[at[0]:at[0] + co * 9 * ci].reshape(co, 3, 3, ci).permute(0, 3, 1, 2)
        bias = params[at[0] + co * 9 * ci:at[0] + co * (9 * ci + 1)]
        at[0] += co * (9 * ci + 1)
        # the 3 x 3 window as nine products over the channels
        pad = F.pad(a, (1, 1, 1, 1))
        h, wd = a.shape[1:]
        return bias[:, None, None] + sum(
            torch.einsum("oc,chw->ohw", w[:, :, i, j], pad[:, i:i + h, j:j + wd])
            for i in range(3) for j in range(3))

    a = x.double().permute(2, 0, 1)
    skips = []
    for lv in range(case["levels"]):
        a = torch.relu(conv(torch.relu(conv(a))))
        if lv < case["levels"] - 1:
            skips.append(a)
            a = F.avg_pool2d(a[None], 2)[0]
    for skip in reversed(skips):
        a = a.repeat_interleave(2, 1).repeat_interleave(2, 2)
        a = torch.relu(conv(torch.relu(conv(torch.cat([a, skip])))))
    out = conv(a)[0] + x[..., 0].double()
    if case["kind"] == "net_forward":
        return out.detach()
    loss = (out - target.double()).square().mean()
    loss.backward()
    return {"out": out.detach(), "loss": float(loss.detach()), "grads": params.grad}


def exact(case, seed):
    kind = case["kind"]
    if kind == "residual":
        u, v, pixel, _ = _observation(case, seed)
        vis, model = _visibilities(u[0], v[0], pixel, case["npix"], _types(case)[1],
                                   _generator(seed))
        keep = _part(u[0], v[0], case, pixel, case["part"])
        op = _Operator(u[0][keep], v[0][keep], case["npix"], pixel)
        obs = vis.to(torch.complex128)[torch.as_tensor(keep, device="cuda")]
        return op.dirty(obs - op.forward(model.to(_types(case)[0]).double()))
    if kind == "channels":
        u, v, pixel, flags, vis, models = _channel_inputs(case, seed)
        images, residuals = [], []
        for c, part in _channel_jobs(case):
            keep = _part(u[c], v[c], case, pixel, part, flags[c])
            op = _Operator(u[c][keep], v[c][keep], case["npix"], pixel)
            keep = torch.as_tensor(keep, device="cuda")
            r = torch.zeros(vis[c].shape, dtype=torch.complex128, device="cuda")
            r[keep] = vis[c].to(torch.complex128)[keep] - op.forward(models[c].double())
            images.append(op.dirty(r[keep]))
            residuals.append(r)
        return {"images": images, "residuals": residuals}
    if kind == "minor":
        s = _images(case, seed)
        part = {"low": "L", "full": "H", "single": "ALL"}[case["step"]]
        keep = _part(s["u"][0], s["v"][0], case, s["pixel"], part)
        psf = _psf_operator(case, s["u"][0][keep], s["v"][0][keep], s["pixel"])
        model, beta = _fista(case, psf, s["residual"], s["lam"], case["iterations"],
                             s["l_low"], s["sigma2"], s["eta2"], s["beta"])
        return {"model": model, "beta": beta if case["warm"] else None}
    if kind == "minor_batch":
        u, v, pixel, flags, res, lams = _batch_inputs(case, seed)
        models = []
        for c in range(case["channels"]):
            keep = _part(u[c], v[c], case, pixel, "L", flags[c])
            psf = _psf_operator(case, u[c][keep], v[c][keep], pixel)
            models.append(_fista(case, psf, res[c], lams[c], case["iterations"])[0])
        return {"models": models}
    if kind == "two_step":
        return _exact_two_step(case, seed)
    return _exact_net(case, seed)
