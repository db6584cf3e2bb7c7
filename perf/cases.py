"""The work whose speed is measured: what users of this library have it do, through its
public entry points, over the range of sizes its configurations, tests and benchmark use.

Each case names a kind of work:

  reconstruct       a whole reconstruction on device buffers (``clamp.reconstruct``)
  reconstruct_host  the same from and to host memory (``clamp.reconstruct_host``)
  iterate           iterations of a running reconstruction (``clamp.iterate``)
  step              a caller's own iteration: forward agents, prior agent, MACE step
  batch             scenes of uneven sizes as one graph (``clamp.Batch``)
  data              training data: looks simulated, speckle average formed
  denoise           the CNN prior agent alone (``clamp.denoise``)
  warm_start        the U-Net's initial reflectance (``UNet.warm_start``)
  train             forward and backward of the U-Net on a mini-batch (``UNet.backward``)

Inputs are synthetic scenes and looks made with plain torch from the seed; reflectances of
one surface per (x, y) column, circular Gaussian speckle, a circular pupil and a Hann range
window, additive noise.  Residuals and losses are returned in 32 bits: they are sums of
values that the library computes in 32 bits.
"""
from __future__ import annotations

import math
import os
import random

import numpy as np
import torch

from paper_2406_13651_gb300 import clamp as C
from paper_2406_13651_gb300 import inputs as I

PROX_VAR = 1e-4
SIGMA = 0.8              # Gaussian prior
CHANNELS = (16, 32, 64)  # U-Net
AXES = (32, 64, 96, 128, 192, 256)
LARGEST = 256 * 256 * 128 * 32   # voxel-looks of the largest volume


# ------------------------------------------------------------------------------ the cases

def listed():
    return [
        # a small scene from start to end: every launch counts (20 iterations, Gaussian prior)
        dict(name="reconstruct 32x32x16 L4", kind="reconstruct", nx=32, ny=32, nz=16, looks=4, radius=0.5,
             snr=10.0, iters=20),
        # data of the paper's size (128^3, nine looks) handed over in host memory
        dict(name="host 128x128x128 L9", kind="reconstruct_host", nx=128, ny=128, nz=128, looks=9, radius=0.5,
             snr=10.0, iters=10),
        # the FP32 CNN prior's configuration, iterations in the middle of a run
        dict(name="iterate cnn 128x128x64 L16", kind="iterate", nx=128, ny=128, nz=64, looks=16, radius=0.4,
             snr=15.0, iters=4, prior="cnn", layers=5, channels=32, dtype="fp32"),
        # the largest scene (warm-start comparison's configuration), Gaussian prior
        dict(name="iterate 256x256x128 L32", kind="iterate", nx=256, ny=256, nz=128, looks=32, radius=0.4,
             snr=1.5, iters=2, prior="gauss"),
        # a caller's own loop on a zero-padded grid (q = 1.5, radix-3 lengths), nine looks
        dict(name="step 192x192x96 L9", kind="step", nx=192, ny=192, nz=96, looks=9, radius=0.27, snr=10.0, q=1.5),
        # a batch of uneven scenes in one launch
        dict(name="batch of 6", kind="batch", scenes=6, scene_seed=7, iters=10),
        # a training pair's looks and network input (64x64x32, 32 looks)
        dict(name="data 64x64x32 L32", kind="data", nx=64, ny=64, nz=32, looks=32, radius=0.4, snr=10.0),
        # the BF16 CNN prior of the largest configuration
        dict(name="denoise bf16 256x256x128", kind="denoise", nx=256, ny=256, nz=128, layers=8, channels=48,
             dtype="bf16"),
        # the learned warm start at full size, and on a zero-padded grid
        dict(name="warm start 256x256x128", kind="warm_start", nx=256, ny=256, nz=128),
        dict(name="warm start 192x192x96", kind="warm_start", nx=192, ny=192, nz=96),
        # training: the warm start's mini-batch, and the prior network's patches
        dict(name="train 24x64x64x32", kind="train", batch=24, nx=64, ny=64, nz=32),
        dict(name="train 24x32x32x32", kind="train", batch=24, nx=32, ny=32, nz=32),
    ]


def _log_choice(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _scene_sizes(rng, cost):
    """Sizes of a scene with at most `cost` voxel-looks, spread over the logarithm of the range."""
    want = math.exp(rng.uniform(math.log(32 * 32 * 16 * 4), math.log(cost)))
    best = None
    for _ in range(40):
        nx, ny = rng.choice(AXES), rng.choice(AXES)
        ny = nx if rng.random() < 0.6 else ny
        s = dict(nx=nx, ny=ny, nz=rng.choice((16, 32, 64, 96, 128)), looks=rng.randint(2, 32))
        v = s["nx"] * s["ny"] * s["nz"] * s["looks"]
        if v <= cost and (best is None or abs(math.log(v / want)) < best[0]):
            best = (abs(math.log(v / want)), s)
    return best[1]


def draw(rng):
    kind = rng.choice(("reconstruct", "reconstruct_host", "iterate", "iterate", "step", "batch", "data", "denoise",
                       "warm_start", "train"))
    look = dict(radius=round(rng.uniform(0.3, 0.5), 3), snr=round(rng.uniform(1.5, 20.0), 2))
    if kind in ("reconstruct", "reconstruct_host"):
        it = rng.choice((5, 10, 20))
        return dict(kind=kind, iters=it, **_scene_sizes(rng, LARGEST // 8 // it), **look)
    if kind == "iterate":
        it = rng.choice((1, 2, 4))
        s = _scene_sizes(rng, LARGEST // it)
        if rng.random() < 0.4 and s["nx"] * s["ny"] * s["nz"] <= 1 << 20:
            return dict(kind=kind, iters=it, prior="cnn", layers=rng.randint(3, 5), channels=rng.choice((16, 32, 48)),
                        dtype="fp32", **s, **look)
        return dict(kind=kind, iters=it, prior="gauss", **s, **look)
    if kind == "step":
        q = rng.choice((1.0, 1.5, 2.0))
        return dict(kind=kind, q=q, **_scene_sizes(rng, LARGEST // 4), **dict(look, radius=round(look["radius"] / q, 3)))
    if kind == "batch":
        return dict(kind=kind, scenes=rng.randint(2, 6), scene_seed=rng.randrange(1000), iters=10)
    if kind == "data":
        return dict(kind=kind, **_scene_sizes(rng, LARGEST // 4), **look)
    if kind == "denoise":
        nx, ny, nz = rng.choice((128, 256)), 2 * _log_choice(rng, 8, 128), 2 * _log_choice(rng, 8, 64)
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, layers=rng.randint(3, 8), channels=rng.choice((16, 32, 48, 64)),
                    dtype="bf16")
    if kind == "warm_start":
        return dict(kind=kind, nx=rng.choice((32, 64, 96, 128, 192, 256)), ny=4 * _log_choice(rng, 8, 64),
                    nz=4 * _log_choice(rng, 4, 32))
    nx = rng.choice((16, 32, 64))
    return dict(kind=kind, batch=_log_choice(rng, 2, 24), nx=nx, ny=4 * _log_choice(rng, 4, 16),
                nz=4 * _log_choice(rng, 4, 8))


def _batch_scenes(case):
    """The scenes of a batch: sizes and looks of the batch configuration, none above a twelfth of the largest."""
    rng, out = random.Random(case["scene_seed"]), []
    while len(out) < case["scenes"]:
        n = rng.choice((64, 96, 128, 192, 256))
        s = dict(nx=n, ny=n, nz=rng.choice((32, 64, 128)), looks=rng.randint(4, 32),
                 radius=round(rng.uniform(0.3, 0.5), 3), snr=round(rng.uniform(5.0, 20.0), 2), iters=case["iters"])
        if s["nx"] * s["ny"] * s["nz"] * s["looks"] <= LARGEST // 12:
            out.append(s)
    return out


# ------------------------------------------------------------------------------ inputs

DEV = "cuda"


def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + stream)
    return g


def _freq(n):
    k = torch.arange(n, device=DEV, dtype=torch.float64)
    return torch.where(k <= (n - 1) // 2, k, k - n)


def _pupil(nx, ny, radius):
    fx, fy = 2 * _freq(nx) / nx, 2 * _freq(ny) / ny
    return ((fy[:, None] ** 2 + fx[None, :] ** 2) <= radius * radius + 1e-12).float()


def _window(nz, q=1.0):
    m, f = nz / q, _freq(nz)
    h = 0.5 * (1.0 + torch.cos(2.0 * math.pi * f / m))
    return torch.where(f.abs() <= m / 2.0, h, torch.zeros_like(h)).float()


def _scene(nx, ny, nz, gen):
    """One surface per (x, y) column at a smooth random depth, reflectance U[0.2, 1]."""
    white = torch.randn((ny, nx), generator=gen, device=DEV, dtype=torch.float64)
    s = max(nx, ny) / 8.0
    h = torch.exp(-2.0 * (math.pi * s) ** 2 * ((_freq(ny) / ny)[:, None] ** 2 + (_freq(nx) / nx)[None, :] ** 2))
    d = torch.fft.ifft2(torch.fft.fft2(white) * h).real
    d = (d - d.min()) / (d.max() - d.min()).clamp_min(1e-300)
    z = torch.floor((0.2 + 0.6 * d) * nz + 0.5).long().clamp_(0, nz - 1)
    refl = 0.2 + 0.8 * torch.rand((ny, nx), generator=gen, device=DEV, dtype=torch.float64)
    return torch.zeros((nz, ny, nx), device=DEV, dtype=torch.float64).scatter_(0, z[None], refl[None]).float()


def _cn(shape, gen):
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), generator=gen, device=DEV) * math.sqrt(0.5))


def _noise_var(r, pupil, window, snr):
    sp, sw = pupil.double().square().sum(), window.double().square().sum()
    supp = int((pupil != 0).sum()) * int((window != 0).sum())
    return float(np.float32(float(r.double().mean() * sp * sw) / supp / 10.0 ** (snr / 10.0)))


def _looks(s, seed):
    """r, y [L][nz][ny][nx] complex64, pupil, window, noise variance of a scene."""
    gen, q = _gen(seed, 1), s.get("q", 1.0)
    r = _scene(s["nx"], s["ny"], s["nz"], gen)
    pupil, window = _pupil(s["nx"], s["ny"], s["radius"]), _window(s["nz"], q)
    nv = _noise_var(r, pupil, window, s["snr"])
    a, root = window[:, None, None] * pupil[None], r.sqrt()
    y = torch.empty((s["looks"],) + tuple(r.shape), dtype=torch.complex64, device=DEV)
    for l in range(s["looks"]):
        y[l] = a * torch.fft.fftn(root * _cn(r.shape, gen), norm="ortho") + math.sqrt(nv) * _cn(r.shape, gen)
    return r, y, pupil, window, nv


def _params(s, nv, iters=0):
    return C.make_params(s["nx"], s["ny"], s["nz"], s["looks"], nv, PROX_VAR, max_iters=iters)


def _state(y, pupil, window):
    """mu, r, w of a reconstruction's start: mu_l = A^H y_l / alpha, r and w the speckle average."""
    a = window[:, None, None] * pupil[None]
    alpha = float(a.double().square().mean())
    mu = torch.empty_like(y)
    r0 = torch.zeros(y.shape[1:], dtype=torch.float32, device=DEV)
    for l in range(y.shape[0]):
        x = torch.fft.ifftn(a * y[l], norm="ortho")
        r0 += x.real.square() + x.imag.square()
        mu[l] = x / alpha
    r0 = (r0 / y.shape[0]).clamp_min_(1e-12 * float(r0.max()))
    r = r0[None].expand((y.shape[0] + 1,) + tuple(r0.shape)).contiguous()
    return mu, r, r.clone()


def _cnn_weights(case, seed):
    """He-normal 3x3x3 weights, the last layer scaled by 0.01, zero biases (as the configurations')."""
    return I.cnn_weights(case["layers"], case["channels"], seed)


def _unet_weights(case, seed):
    if case["kind"] == "train":
        return I.unet_params(CHANNELS, seed)
    path = os.path.join(os.path.dirname(os.path.abspath(C.__file__)), "weights", "unet_warmstart.npz")
    with np.load(path) as f:
        return np.asarray(f["params"], np.float32)


def _average_and_scene(nx, ny, nz, seed):
    """A speckle average of eight looks and its scene seen through the same aperture (the target)."""
    s = dict(nx=nx, ny=ny, nz=nz, looks=8, radius=0.4, snr=10.0)
    r, y, pupil, window, _ = _looks(s, seed)
    a = window[:, None, None] * pupil[None]
    r0 = torch.zeros_like(r)
    for l in range(8):
        x = torch.fft.ifftn(a * y[l], norm="ortho")
        r0 += (x.real.square() + x.imag.square()) / 8.0
    return r0.clamp_min_(1e-12 * float(r0.max())), r


def _prior(case, seed):
    if case.get("prior") == "cnn" or case["kind"] == "denoise":
        return C.Denoiser.cnn(*_cnn_weights(case, seed), dtype=case["dtype"])
    return C.Denoiser.gauss(SIGMA)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, kind=kind)
    if kind in ("reconstruct", "reconstruct_host", "iterate", "step"):
        _, y, pupil, window, nv = _looks(case, seed)
        p = _params(case, nv, case.get("iters", 0))
        st.update(p=p, y=y, pupil=pupil, window=window, den=_prior(case, seed))
        if kind == "reconstruct":
            st["ws"] = C.reconstruct_workspace(p, st["den"])
        elif kind == "reconstruct_host":
            host = {}
            for name in ("y", "pupil", "window"):
                host[name] = C.host_empty(st[name].shape, st[name].dtype)
                host[name].copy_(st[name])
                st[name] = host[name].numpy()
            out = C.host_empty((p.nz, p.ny, p.nx), torch.float32)
            st.update(host=host, out=out, r_out=out.numpy())
        else:
            st["mu"], st["r"], st["w"] = _state(y, pupil, window)
            st["wbar"] = torch.empty_like(st["r"][0])
            st["ce"] = torch.zeros(case.get("iters", 1), dtype=torch.float64, device=DEV)
            st["ws"] = C.iterate_workspace(p, st["den"])
    elif kind == "batch":
        scenes = []
        for i, s in enumerate(_batch_scenes(case)):
            r, y, pupil, window, nv = _looks(s, 100 * seed + i)
            scenes.append((_params(s, nv, s["iters"]), y, pupil, window, torch.empty_like(r)))
        st["batch"] = C.Batch(scenes, C.Denoiser.gauss(SIGMA))
        st["out"] = [s[4] for s in scenes]
    elif kind == "data":
        gen = _gen(seed, 1)
        r = _scene(case["nx"], case["ny"], case["nz"], gen)
        pupil, window = _pupil(case["nx"], case["ny"], case["radius"]), _window(case["nz"])
        p = _params(case, _noise_var(r, pupil, window, case["snr"]))
        shape = (case["looks"],) + tuple(r.shape)
        st.update(p=p, r=r, pupil=pupil, window=window, z=_cn(shape, gen), eta=_cn(shape, gen), ws=C.workspace(p))
    elif kind == "denoise":
        gen = _gen(seed, 1)
        r = _scene(case["nx"], case["ny"], case["nz"], gen)
        st["den"] = _prior(case, seed)
        # what the prior agent sees: a blurred scene with a noise floor
        st["x"] = 0.05 * r + 0.01 * torch.rand(r.shape, generator=gen, device=DEV)
        st["out"] = torch.empty_like(r)
        st["ws"] = torch.empty(st["den"].workspace_size(case["nx"], case["ny"], case["nz"]), dtype=torch.uint8,
                               device=DEV)
    elif kind == "warm_start":
        st["r0"], _ = _average_and_scene(case["nx"], case["ny"], case["nz"], seed)
        st["net"] = C.UNet(*CHANNELS, params=_unet_weights(case, seed))
        st["net"].workspace(1, case["nx"], case["ny"], case["nz"], False)
    else:
        pairs = [_average_and_scene(case["nx"], case["ny"], case["nz"], 100 * seed + b) for b in range(case["batch"])]
        m = [float(x.double().sum()) / (case["nx"] * case["ny"]) for x, _ in pairs]
        st["x"] = torch.stack([x / v for (x, _), v in zip(pairs, m)])
        st["t"] = torch.stack([t / v for (_, t), v in zip(pairs, m)])
        st["loss"] = torch.zeros((), dtype=torch.float64, device=DEV)
        st["net"] = C.UNet(*CHANNELS, params=_unet_weights(case, seed))
        st["net"].workspace(case["batch"], case["nx"], case["ny"], case["nz"], True)
    return st


# ------------------------------------------------------------------------------ one pass

K_FIRST = 10   # iterations in the middle of a run: the index the surrogate's interval depends on


def run(st):
    kind, case = st["kind"], st["case"]
    if kind == "reconstruct":
        res = C.reconstruct(st["p"], st["y"], st["pupil"], st["window"], st["den"], ws=st["ws"])
        return dict(r=res.r, ce=res.ce_hist.astype(np.float32), mu_res=res.mu_hist.astype(np.float32))
    if kind == "reconstruct_host":
        res = C.reconstruct_host(st["p"], st["y"], st["pupil"], st["window"], st["den"], r_out=st["r_out"])
        return dict(r=res.r, ce=res.ce_hist.astype(np.float32), mu_res=res.mu_hist.astype(np.float32))
    if kind == "iterate":
        C.iterate(st["p"], K_FIRST, case["iters"], st["y"], st["pupil"], st["window"], st["den"], st["mu"], st["r"],
                  st["w"], st["wbar"], ce_out=st["ce"], ws=st["ws"])
        return dict(mu=st["mu"], r=st["r"], w=st["w"], wbar=st["wbar"], ce=st["ce"].float())
    if kind == "step":
        L = case["looks"]
        C.forward_prox(st["p"], K_FIRST, st["y"], st["pupil"], st["window"], st["mu"], st["r"], st["w"], ws=st["ws"])
        C.denoise(st["den"], st["w"][L], st["r"][L])
        C.mace_step(st["p"], st["r"], st["w"], st["wbar"], st["ce"], ws=st["ws"])
        return dict(mu=st["mu"], r=st["r"], w=st["w"], wbar=st["wbar"], ce=st["ce"].float())
    if kind == "batch":
        st["batch"].launch()
        return st["out"]
    if kind == "data":
        y = C.simulate(st["p"], st["r"], st["z"], st["eta"], st["pupil"], st["window"])
        return dict(y=y, r0=C.speckle_average(st["p"], y, st["pupil"], st["window"], ws=st["ws"]))
    if kind == "denoise":
        C.denoise(st["den"], st["x"], st["out"], ws=st["ws"])
        return st["out"]
    if kind == "warm_start":
        return st["net"].warm_start(st["r0"])
    st["net"].backward(st["x"], st["t"], st["loss"])
    return dict(loss=st["loss"].float(), grads=st["net"].get("grads"))


# ------------------------------------------------------------------------------ what a pass cannot do without

def _support(s):
    """Share of the (ky, kx) plane inside the circular pupil."""
    return min(1.0, math.pi * s["radius"] ** 2 / 4.0)


def _iteration_work(s):
    """One iteration: mu, r and w read and written, the data read on the aperture's support; a
    transform of the whole volume and back."""
    n = s["nx"] * s["ny"] * s["nz"]
    v = n * s["looks"]
    return v * (32.0 + 8.0 * _support(s)) + 12.0 * n, v * (2 * 5 * math.log2(n) + 60.0) + 54.0 * n


def _cnn_flops(s):
    n, c = s["nx"] * s["ny"] * s["nz"], s["channels"]
    return 54.0 * n * (2 * c + (s["layers"] - 2) * c * c)


def _unet_flops():
    """Multiply-adds counted as two, per voxel of the full-size level."""
    c1, c2, c3 = CHANNELS
    return (54.0 * (c1 + c1 * c1 + 2 * c1 * c1 + c1 * c1) + 2 * c2 * c1 + 2 * c1 +
            (54.0 * (c1 * c2 + c2 * c2 + 2 * c2 * c2 + c2 * c2) + 2 * c3 * c2) / 8 + 54.0 * (c2 * c3 + c3 * c3) / 64)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        b = f = 0.0
        for s in _batch_scenes(case):
            n = s["nx"] * s["ny"] * s["nz"]
            ib, if_ = _iteration_work(s)
            b += s["iters"] * ib + 8.0 * n * s["looks"] * _support(s) + 4.0 * n
            f += s["iters"] * if_
        return dict(bytes=b, flops=f)
    n = case["nx"] * case["ny"] * case["nz"]
    if kind in ("reconstruct", "reconstruct_host", "iterate", "step"):
        b, f = _iteration_work(case)
        it = case.get("iters", 1)
        f += _cnn_flops(case) if case.get("prior") == "cnn" else 0.0
        extra = (8.0 * n * case["looks"] * _support(case) + 4.0 * n) if kind.startswith("reconstruct") else 0.0
        return dict(bytes=it * b + extra, flops=it * f)
    if kind == "data":   # speckle and noise read, y written, the average written; one transform each way
        v = n * case["looks"]
        return dict(bytes=24.0 * v + 8.0 * n, flops=v * (2 * 5 * math.log2(n) + 10.0))
    if kind == "denoise":
        return dict(bytes=8.0 * n, flops=_cnn_flops(case))
    if kind == "warm_start":
        return dict(bytes=8.0 * n, flops=n * _unet_flops())
    nb = n * case["batch"]
    return dict(bytes=8.0 * nb, flops=3.0 * nb * _unet_flops())


# ------------------------------------------------------------------------------ 64-bit results

def _gauss64(x):
    e = math.exp(-1.0 / (2.0 * SIGMA * SIGMA))
    g0, g1 = e / (1.0 + 2.0 * e), 1.0 / (1.0 + 2.0 * e)
    for ax in range(3):
        n = x.shape[ax]
        z = torch.zeros_like(x.narrow(ax, 0, 1))
        p = torch.cat([z, x, z], dim=ax)
        x = g0 * (p.narrow(ax, 0, n) + p.narrow(ax, 2, n)) + g1 * x
    return x


def _conv64(x, w, b):
    """3x3x3 convolution, zero padding: x [ci][nz][ny][nx], w [co][ci][3][3][3], all float64."""
    ci, nz, ny, nx = x.shape
    p = torch.nn.functional.pad(x, (1, 1, 1, 1, 1, 1))
    out = None
    for t in range(27):
        dz, dy, dx = t // 9, t // 3 % 3, t % 3
        part = w[:, :, dz, dy, dx].contiguous() @ p[:, dz:dz + nz, dy:dy + ny, dx:dx + nx].reshape(ci, -1)
        out = part if out is None else out + part
    return out.reshape(-1, nz, ny, nx) + b[:, None, None, None]


def _cnn64(x, case, seed):
    h = x[None]
    ws, bs = _cnn_weights(case, seed)
    for i, (w, b) in enumerate(zip(ws, bs)):
        h = _conv64(h, torch.from_numpy(w).to(DEV).double(), torch.from_numpy(b).to(DEV).double())
        h = h.clamp_min_(0.0) if i < len(ws) - 1 else h
    return x + h[0]


def _iterations64(case, seed, y, pupil, window, nv, mu, r, w, k_first, iters):
    """Iterations of Alg. 2 on float64 state (mu, r, w changed in place); (wbar, ce, mu_res)."""
    L = y.shape[0]
    s2 = float(np.float32(PROX_VAR))
    a = window.double()[:, None, None] * pupil.double()[None]
    alpha = float(a.square().mean())
    ups, ups_p = 0.5 / L, 0.5
    ce_all, res_all = [], []
    for k in range(k_first, k_first + iters):
        beta = 1.0 + 2.0 / math.log(k + 1.0)
        r_prior = _cnn64(w[L], case, seed) if case.get("prior") == "cnn" else _gauss64(w[L])
        wb = ups_p * w[L]
        for l in range(L):
            wb = wb + ups * w[l]
        xb, num, res = ups_p * (2.0 * r_prior - w[L]), float((r_prior - wb).square().sum()), 0.0
        for l in range(L):
            yl, rp = y[l].to(torch.complex128), r[l].clone()
            D = 1.0 / (rp + nv / alpha)
            d = torch.fft.ifftn(a * (yl - a * torch.fft.fftn(mu[l], norm="ortho")), norm="ortho") / nv - D * mu[l]
            d2 = d.real.square() + d.imag.square()
            s1, s3 = float(d2.sum()), float((D * d2).sum())
            ad = a * torch.fft.fftn(d, norm="ortho")
            s4 = float((a * yl).abs().square().sum())
            gamma = s1 / (float(ad.abs().square().sum()) / nv + s3)
            res += math.sqrt(s1) / (math.sqrt(s4) / nv) / L
            mu[l] += gamma * d
            K = nv * rp / (alpha * rp + nv) + mu[l].real.square() + mu[l].imag.square()
            drho = 1.0 / rp - K / rp ** 2 + (rp - w[l]) / s2
            xi = torch.where(drho > 0, rp / beta, beta * rp)
            q_r = 1.0 / rp - K / rp ** 2
            aq = (K / rp ** 2 - K / xi ** 2) / (xi - rp)
            rn = (w[l] - s2 * (q_r - aq * rp)) / (1.0 + s2 * aq)
            r[l] = torch.minimum(torch.maximum(rn, torch.minimum(rp, xi)), torch.maximum(rp, xi))
            xb = xb + ups * (2.0 * r[l] - w[l])
            num += float((r[l] - wb).square().sum())
        r[L] = r_prior
        ce_all.append(math.sqrt(num / ((L + 1) * float(wb.square().sum()))))
        res_all.append(res)
        w += xb[None] - r
    wbar = ups_p * w[L]
    for l in range(L):
        wbar = wbar + ups * w[l]
    return wbar, torch.tensor(ce_all, dtype=torch.float64), torch.tensor(res_all, dtype=torch.float64)


def _reconstruct64(case, seed, iters):
    _, y, pupil, window, nv = _looks(case, seed)
    a = window.double()[:, None, None] * pupil.double()[None]
    mu = torch.stack([torch.fft.ifftn(a * y[l], norm="ortho") for l in range(y.shape[0])])
    r0 = (mu.real.square() + mu.imag.square()).mean(0)
    r0 = r0.clamp_min(1e-12 * float(r0.max()))
    r = r0[None].repeat(y.shape[0] + 1, 1, 1, 1)
    return _iterations64(case, seed, y, pupil, window, nv, mu / float(a.square().mean()), r, r.clone(), 1, iters)


def _unet64(flat, x):
    """U-Net output [nz][ny][nx] for x [nz][ny][nx], parameters `flat` (float64, in order)."""
    c1, c2, c3 = CHANNELS
    spec = [(3, 1, c1), (3, c1, c1), (3, c1, c2), (3, c2, c2), (3, c2, c3), (3, c3, c3), (2, c3, c2), (3, 2 * c2, c2),
            (3, c2, c2), (2, c2, c1), (3, 2 * c1, c1), (3, c1, c1), (1, c1, 1)]
    layers, off = [], 0
    for k, ci, co in spec:
        shape = (ci, co, 2, 2, 2) if k == 2 else (co, ci, k, k, k)
        nw = ci * co * k ** 3
        layers.append((flat[off:off + nw].reshape(shape), flat[off + nw:off + nw + co]))
        off += nw + co

    def conv(i, t):
        return torch.relu(_conv64(t, *layers[i]))

    def pool(t):
        c, nz, ny, nx = t.shape
        return t.reshape(c, nz // 2, 2, ny // 2, 2, nx // 2, 2).amax(dim=(2, 4, 6))

    def up(i, t):
        (w, b), (c, nz, ny, nx) = layers[i], t.shape
        u = w.reshape(c, -1).t() @ t.reshape(c, -1)
        u = u.reshape(-1, 2, 2, 2, nz, ny, nx).permute(0, 4, 1, 5, 2, 6, 3).reshape(-1, 2 * nz, 2 * ny, 2 * nx)
        return u + b[:, None, None, None]

    s1 = conv(1, conv(0, x[None]))
    s2 = conv(3, conv(2, pool(s1)))
    d2 = conv(8, conv(7, torch.cat([up(6, conv(5, conv(4, pool(s2)))), s2])))
    d1 = conv(11, conv(10, torch.cat([up(9, d2), s1])))
    w, b = layers[12]
    return (w.reshape(1, -1) @ d1.reshape(c1, -1)).reshape(x.shape) + b


def exact(case, seed):
    kind = case["kind"]
    if kind in ("reconstruct", "reconstruct_host"):
        wbar, ce, res = _reconstruct64(case, seed, case["iters"])
        return dict(r=wbar, ce=ce, mu_res=res)
    if kind in ("iterate", "step"):
        _, y, pupil, window, nv = _looks(case, seed)
        mu, r, w = _state(y, pupil, window)
        mu, r, w = mu.to(torch.complex128), r.double(), w.double()
        wbar, ce, _ = _iterations64(case, seed, y, pupil, window, nv, mu, r, w, K_FIRST, case.get("iters", 1))
        return dict(mu=mu, r=r, w=w, wbar=wbar, ce=ce)
    if kind == "batch":
        return [_reconstruct64(s, 100 * seed + i, s["iters"])[0] for i, s in enumerate(_batch_scenes(case))]
    if kind == "data":
        st = prepare(case, seed)
        a = st["window"].double()[:, None, None] * st["pupil"].double()[None]
        sig, root = math.sqrt(st["p"].noise_var), st["r"].double().sqrt()
        y, r0 = torch.empty(st["z"].shape, dtype=torch.complex128, device=DEV), torch.zeros_like(root)
        for l in range(case["looks"]):
            y[l] = a * torch.fft.fftn(root * st["z"][l], norm="ortho") + sig * st["eta"][l].to(torch.complex128)
            r0 += torch.fft.ifftn(a * y[l], norm="ortho").abs().square() / case["looks"]
        return dict(y=y, r0=r0.clamp_min(1e-12 * float(r0.max())))
    if kind == "denoise":
        return _cnn64(prepare(case, seed)["x"].double(), case, seed)
    flat = torch.from_numpy(_unet_weights(case, seed)).to(DEV).double()
    if kind == "warm_start":
        r0 = _average_and_scene(case["nx"], case["ny"], case["nz"], seed)[0].double()
        m = float(r0.sum()) / (case["nx"] * case["ny"])
        with torch.no_grad():
            return m * _unet64(flat, r0 / m).clamp_min(1e-3)
    st = prepare(case, seed)
    flat.requires_grad_(True)
    loss, count = 0.0, st["x"].numel()
    for x, t in zip(st["x"], st["t"]):
        part = (_unet64(flat, x.double()) - t.double()).square().sum() / count
        part.backward()
        loss += float(part.detach())
    return dict(loss=torch.tensor(loss, dtype=torch.float64), grads=flat.grad)
