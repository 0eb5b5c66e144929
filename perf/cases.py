"""Timed cases of the smooth-and-clip library, through its Python binding.

A case is one call that a user of the library makes: S+C on a cube (`run`), on
a cube stored in 16 bits (`run_half`), on a batch of sub-cubes (`run_batch`),
one smoothed cube (`smooth`), the local noise normalisation (`noise_scale`),
the auto-flagger (`autoflag`) and the linker (`link`). Sizes run from the
64 x 64 x 128 test cube to the WALLABY-shaped 1200 x 1200 x 1024 one. Inputs
are synthetic H I cubes made on the GPU from a seed: beam-correlated Gaussian
noise with a channel ripple, mock galaxies, and NaN-blanked corners or borders.

`exact` repeats a case in float64 with plain torch, sharing no code with the
library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2106_15789_gb300 import Context
from paper_2106_15789_gb300 import sc

FWHM_TO_SIGMA = 1.0 / math.sqrt(8.0 * math.log(2.0))
DEV = "cuda:0"
REPLACEMENT = 2.0
MAX_SOURCES = 1 << 14

# (spatial FWHM px, spectral boxcar channels), spatial outer, spectral inner.
KERNEL_LISTS = {
    "12": [(float(f), w) for f in (0, 3, 6) for w in (0, 3, 7, 15)],
    "paper": [(float(f), w) for f in (0, 5, 10) for w in (0, 3, 7, 15)],
    "20": [(float(f), w) for f in (0, 3, 6, 10) for w in (0, 3, 7, 15, 31)],
}


def listed() -> list:
    run = dict(op="run", kernels="12", t=3.5, noise="mad", sampled=False, blank="border")
    return [
        # the test cube, also a cut-out around one source: latency and launches count
        dict(run, name="run-small", nx=64, ny=64, nz=128, n_gal=20, blank="corner"),
        # a sub-cube cut at odd places: rows that are no multiple of 16 bytes
        dict(run, name="run-ragged", nx=217, ny=331, nz=509, n_gal=60),
        # the cube and kernel list of the paper's speed test
        dict(run, name="run-paper", nx=360, ny=360, nz=1464, n_gal=400, kernels="paper", blank="none"),
        # a survey-sized cube: the headline workload
        dict(run, name="run-wallaby", nx=1200, ny=1200, nz=1024, n_gal=3000),
        # the Gaussian-fit noise mode, on a cube of ordinary size
        dict(run, name="run-gauss", nx=400, ny=360, nz=512, n_gal=150, noise="gauss"),
        # sampled spatial Gaussians and the standard deviation as noise
        dict(run, name="run-sampled-std", nx=256, ny=250, nz=600, n_gal=80, noise="std", sampled=True),
        # a sub-cube of a stream: FP16 storage, the 20-pair list
        dict(run, op="half", name="half-stream", nx=256, ny=312, nz=640, n_gal=100, kernels="20", t=4.0, bf16=False,
             blank="none"),
        # uneven sub-cubes of a survey as one graph-replayed batch
        dict(op="batch", name="batch-12", n=12, sizes=1, lo=128, hi=512, zlo=256, zhi=1024, kernels="12", t=3.5),
        # local noise normalisation of the paper's speed test: 31-voxel windows on 16-voxel cells
        dict(op="noise_scale", name="noise-scale", nx=360, ny=360, nz=1464, n_gal=400, blank="border", noise="mad",
             wx=31, wy=31, wz=31, gx=16, gy=16, gz=16),
        # flagging of channels and pixels before the source finding
        dict(op="autoflag", name="autoflag", nx=600, ny=600, nz=1024, n_gal=800, blank="border", noise="mad", k=4.0,
             channels=True, pixels=True),
        # detections from the mask of a large cube, with the paper's radii and sizes
        dict(op="link", name="link", nx=640, ny=640, nz=1024, n_gal=1000, r_xy=2, r_z=2, min_xy=8, min_z=5),
        # one smoothed cube, masked voxels replaced
        dict(op="smooth", name="smooth", nx=512, ny=512, nz=256, n_gal=150, blank="border", fwhm=6.0, w=7,
             sampled=False),
    ]


def _log_uniform(rng, lo: float, hi: float) -> float:
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _draw_dims(rng, lo: float, hi: float, max_nz: int = 1600) -> dict:
    """nx, ny, nz of a cube of log-uniform volume, axis ratios up to 3, half
    of them with whatever nx comes out and half with rows of 16-byte multiples."""
    v = _log_uniform(rng, lo, hi)
    a, b = _log_uniform(rng, 1.0 / 3.0, 3.0), _log_uniform(rng, 0.5, 4.0)
    side = (v / (a * b)) ** (1.0 / 3.0)
    nz = min(max_nz, max(16, int(side * b)))
    nxy = math.sqrt(v / nz)
    nx, ny = max(24, int(nxy * math.sqrt(a))), max(24, int(nxy / math.sqrt(a)))
    if rng.random() < 0.5:
        nx = (nx + 7) // 8 * 8
    n_gal = max(5, int(nx * ny * nz / 5e5))
    return dict(nx=nx, ny=ny, nz=nz, n_gal=min(n_gal, 1500))


def draw(rng) -> dict:
    op = rng.choice(["run", "run", "run", "run", "half", "batch", "noise_scale", "autoflag", "link", "smooth"])
    blank = rng.choice(["none", "corner", "border"])
    if op in ("run", "half"):
        c = dict(op=op, kernels=rng.choice(sorted(KERNEL_LISTS)), t=round(rng.uniform(3.2, 4.5), 2),
                 noise=rng.choice(["mad", "mad", "mad", "std", "gauss"]), sampled=rng.random() < 0.2, blank=blank,
                 **_draw_dims(rng, 3e5, 4e8))
        if op == "half":
            c["bf16"] = rng.random() < 0.5
        return c
    if op == "batch":
        return dict(op=op, n=rng.randint(2, 16), sizes=rng.randint(2, 1 << 20), lo=64, hi=384, zlo=128, zhi=768,
                    kernels=rng.choice(["12", "paper"]), t=round(rng.uniform(3.2, 4.5), 2))
    if op == "noise_scale":
        w = [2 * rng.randint(5, 17) + 1 for _ in range(3)]
        return dict(op=op, blank=blank, noise=rng.choice(["mad", "mad", "std", "gauss"]), wx=w[0], wy=w[1], wz=w[2],
                    gx=(w[0] + 1) // 2, gy=(w[1] + 1) // 2, gz=(w[2] + 1) // 2, **_draw_dims(rng, 1e6, 1e8))
    if op == "autoflag":
        kind = rng.choice(["both", "both", "channels", "pixels"])
        return dict(op=op, blank=blank, noise=rng.choice(["mad", "mad", "std", "gauss"]), k=round(rng.uniform(3, 6), 2),
                    channels=kind != "pixels", pixels=kind != "channels", **_draw_dims(rng, 1e6, 4e8, max_nz=1500))
    if op == "link":
        r = rng.randint(1, 3)
        return dict(op=op, r_xy=r, r_z=rng.randint(1, 3), min_xy=rng.randint(1, 8), min_z=rng.randint(1, 5),
                    **_draw_dims(rng, 5e5, 5e8))
    return dict(op="smooth", blank=blank, fwhm=rng.choice([0.0, 3.0, 5.0, 6.0, 10.0]), w=rng.choice([0, 3, 7, 15, 31]),
                sampled=rng.random() < 0.2, **_draw_dims(rng, 3e5, 4e8))


# ---- inputs ----------------------------------------------------------------


def _gauss_taps(fwhm: float) -> list:
    s = fwhm * FWHM_TO_SIGMA
    r = int(math.ceil(4.0 * s))
    g = [math.exp(-0.5 * (i / s) ** 2) for i in range(-r, r + 1)]
    return [v / sum(g) for v in g]


def _fir(x: torch.Tensor, taps: list, dim: int) -> torch.Tensor:
    """Zero-padded centred FIR along one axis, as a sum of shifted copies."""
    r, n = (len(taps) - 1) // 2, x.shape[dim]
    out = torch.zeros_like(x)
    for i, g in enumerate(taps):
        d = i - r
        if abs(d) < n:
            out.narrow(dim, max(-d, 0), n - abs(d)).add_(x.narrow(dim, max(d, 0), n - abs(d)), alpha=g)
    return out


def _cube(nx: int, ny: int, nz: int, n_gal: int, blank: str, seed: int) -> torch.Tensor:
    """A float32 cube [nz][ny][nx]: noise of a 5 px beam with unit RMS and a 10 %
    channel ripple, galaxies as 3-D Gaussians of peak S/N 2 to 50, blanked voxels."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    cube = torch.randn((nz, ny, nx), generator=gen, device=DEV)
    beam = _gauss_taps(5.0)
    cube = _fir(_fir(cube, beam, 2), beam, 1)
    ripple = 1.0 + 0.1 * torch.sin(2.0 * math.pi * torch.arange(nz, device=DEV) / 128.0)
    cube *= (ripple / sum(b * b for b in beam))[:, None, None]
    u = torch.rand((n_gal, 8), generator=torch.Generator().manual_seed(seed + 77), dtype=torch.float64).tolist()
    for r in u:
        snr = math.exp(math.log(2.0) + r[0] * math.log(25.0))
        maj, sz = (2.0 + 10.0 * r[1] * r[1]) * FWHM_TO_SIGMA, (5.0 + 35.0 * r[4]) * FWHM_TO_SIGMA
        mnr, pa = maj * (0.3 + 0.7 * r[2]), math.pi * r[3]
        x, y, z = r[5] * (nx - 1), r[6] * (ny - 1), r[7] * (nz - 1)
        rx, rz = math.ceil(3 * maj), math.ceil(3 * sz)
        x0, x1, y0, y1 = max(0, int(x) - rx), min(nx, int(x) + rx + 2), max(0, int(y) - rx), min(ny, int(y) + rx + 2)
        z0, z1 = max(0, int(z) - rz), min(nz, int(z) + rz + 2)
        xs = torch.arange(x0, x1, device=DEV)[None, :] - x
        ys = torch.arange(y0, y1, device=DEV)[:, None] - y
        a, b = math.cos(pa) * xs + math.sin(pa) * ys, math.cos(pa) * ys - math.sin(pa) * xs
        sky = torch.exp(-0.5 * ((a / maj) ** 2 + (b / mnr) ** 2))
        spec = torch.exp(-0.5 * ((torch.arange(z0, z1, device=DEV) - z) / sz) ** 2)
        cube[z0:z1, y0:y1, x0:x1] += snr * spec[:, None, None] * sky
    if blank == "corner":
        cube[:nz * 3 // 8, :ny * 3 // 8, :nx * 3 // 8] = float("nan")
    elif blank == "border":
        e = max(1, min(16, nx // 16, ny // 16))
        cube[:, :e] = float("nan")
        cube[:, -e:] = float("nan")
        cube[:, :, :e] = float("nan")
        cube[:, :, -e:] = float("nan")
    return cube


def _detections(cube: torch.Tensor) -> torch.Tensor:
    """A detection mask as S+C leaves one (noise peaks, sources on several
    scales), from plain threshold cuts on Gaussian- and boxcar-smoothed copies."""
    mask = torch.zeros(cube.shape, dtype=torch.uint8, device=cube.device)
    for fwhm in (0.0, 3.0, 6.0):
        xy = _fir(_fir(cube, _gauss_taps(fwhm), 2), _gauss_taps(fwhm), 1) if fwhm else cube
        for w in (1, 3, 7, 15):
            s = _fir(xy, [1.0 / w] * w, 0) if w > 1 else xy
            sample = s.reshape(-1)[:: max(1, s.numel() // 1_000_000)]
            mask |= s.abs() > 3.5 * 1.4826 * sample.abs().median()
    return mask


def _encode16(cube: torch.Tensor, bf16: bool):
    """16-bit storage with one float32 scale per channel: (bit patterns, scales)."""
    top = torch.nan_to_num(cube.abs(), nan=0.0).reshape(cube.shape[0], -1).amax(dim=1)
    scale = torch.where(top > 0, top / (256.0 if bf16 else 16384.0), torch.ones_like(top))
    half = (cube / scale[:, None, None]).to(torch.bfloat16 if bf16 else torch.float16)
    return half.view(torch.int16).contiguous(), scale.contiguous()


def _batch_shapes(case: dict) -> list:
    """(nx, ny, nz) of every sub-cube: log-uniform in the case's ranges."""
    g = torch.Generator().manual_seed(7919 * int(case["sizes"]))
    out = []
    for _ in range(int(case["n"])):
        r = torch.rand(3, generator=g, dtype=torch.float64).tolist()
        size = [int(round(lo * (hi / lo) ** u)) for u, lo, hi in
                zip(r, (case["lo"], case["lo"], case["zlo"]), (case["hi"], case["hi"], case["zhi"]))]
        out.append(tuple(size))
    return out


def _inputs(case: dict, seed: int):
    """The data that the call of a case reads."""
    op = case["op"]
    if op == "batch":
        return [_cube(nx, ny, nz, 20, "none", 1000 * seed + i) for i, (nx, ny, nz) in enumerate(_batch_shapes(case))]
    cube = _cube(case["nx"], case["ny"], case["nz"], case["n_gal"], case.get("blank", "none"), seed)
    if op == "half":
        return _encode16(cube, case["bf16"])
    if op == "link":
        return _detections(cube)
    if op == "smooth":
        return cube, (cube.abs() > 3.5).to(torch.uint8)
    if op == "autoflag":  # channels with interference, pixels with residual continuum
        gen = torch.Generator(device=DEV).manual_seed(seed + 5)
        nz, ny, nx = cube.shape
        cube *= torch.where(torch.rand(nz, generator=gen, device=DEV) < 0.01, 4.0, 1.0)[:, None, None]
        cube *= torch.where(torch.rand((ny, nx), generator=gen, device=DEV) < 0.002, 3.0, 1.0)[None]
    return cube


def prepare(case: dict, seed: int) -> dict:
    """Inputs and outputs in GPU memory and the context that a program keeps."""
    op, data = case["op"], _inputs(case, seed)
    state = dict(case=case, data=data)
    if op == "batch":
        state["ctx"] = Context(0, max(c.numel() for c in data))
        state["masks"] = [torch.empty(c.shape, dtype=torch.uint8, device=DEV) for c in data]
        return state
    shape = (case["nz"], case["ny"], case["nx"])
    state["ctx"] = Context(0, shape[0] * shape[1] * shape[2])
    if op == "link":
        state["table"] = np.zeros((MAX_SOURCES, 7), dtype=np.int32)
    kind = {"run": torch.uint8, "half": torch.uint8, "link": torch.int32}.get(op, torch.float32)
    state["out"] = torch.empty(shape, dtype=kind, device=DEV)
    return state


def run(state: dict) -> dict:
    case, data, ctx, out = state["case"], state["data"], state["ctx"], state.get("out")
    op = case["op"]
    flags = sc.SC_FLAG_SAMPLED_GAUSS if case.get("sampled") else 0
    if op == "run":
        mask, sigmas, sigma0 = ctx.run(data, KERNEL_LISTS[case["kernels"]], case["t"], case["noise"], REPLACEMENT,
                                       mask=out, flags=flags)
        return dict(mask=mask, sigmas=np.array(sigmas), sigma0=sigma0)
    if op == "half":
        mask, sigmas, sigma0 = ctx.run_half(data[0], case["bf16"], data[1], KERNEL_LISTS[case["kernels"]], case["t"],
                                            case["noise"], REPLACEMENT, mask=out, flags=flags)
        return dict(mask=mask, sigmas=np.array(sigmas), sigma0=sigma0)
    if op == "batch":
        masks, sigmas, sigma0s = ctx.run_batch(data, KERNEL_LISTS[case["kernels"]], case["t"], "mad", REPLACEMENT,
                                               masks=state["masks"], flags=sc.SC_FLAG_GRAPH)
        return dict(masks=masks, sigmas=np.array(sigmas), sigma0s=np.array(sigma0s))
    if op == "noise_scale":
        scaled, _ = ctx.noise_scale(data, (case["wx"], case["wy"], case["wz"]), (case["gx"], case["gy"], case["gz"]),
                                    case["noise"], out=out)
        return dict(scaled=scaled)
    if op == "autoflag":
        cube, chan, pix, chan_noise, pix_noise = ctx.autoflag(data, case["k"], case["channels"], case["pixels"],
                                                              case["noise"], out=out)
        return dict(cube=cube, chan=chan, pix=pix, chan_noise=chan_noise, pix_noise=pix_noise)
    if op == "link":
        labels, n, extents = ctx.link(data, case["r_xy"], case["r_z"], case["min_xy"], case["min_z"], labels=out,
                                      extents_cap=MAX_SOURCES)
        table = state["table"]  # the program's source table: one row per detection, zeros after the last
        table[: len(extents)] = extents
        table[len(extents):] = 0
        return dict(labels=labels, n=n, extents=table)
    cube, mask = data
    return dict(smoothed=ctx.smooth(cube, (case["fwhm"], case["w"]), mask=mask, replacement_value=2.0, out=out,
                                    flags=flags))


def work(case: dict) -> dict:
    """Bytes: the cube (or mask) read once, the result written once. Flops: a
    running-sum smoothing (two additions per boxcar pass) per kernel pair, or
    one comparison pass per order statistic."""
    op = case["op"]
    if op == "batch":
        n = sum(x * y * z for x, y, z in _batch_shapes(case))
    else:
        n = case["nx"] * case["ny"] * case["nz"]
    pairs = KERNEL_LISTS.get(case.get("kernels"), [])
    per_pair = sum((12 if f > 0 else 0) + (2 if w > 1 else 0) + 4 for f, w in pairs)
    per_voxel = {"run": 5, "batch": 5, "half": 3, "noise_scale": 8, "autoflag": 8, "link": 5, "smooth": 9}[op]
    flops = per_pair if pairs else {"smooth": 16, "link": 0}.get(op, 4)
    return {"bytes": per_voxel * n, "flops": flops * n}


def tolerance(case: dict):
    """Labels and extents are whole numbers. S is exact up to its rounding to
    float32 (measured against float64: 5e-8 in norm, 1.5e-7 for one value), and
    so are the noises of one measurement. In a run of pairs, a voxel within
    that rounding of a threshold may fall on either side of it; in the smallest
    cube one such voxel moved the later pairs' noises by 5e-6 (1e-5 for one)."""
    if case["op"] == "link":
        return "exact"
    if case["op"] in ("run", "half", "batch"):
        return {"rel": 2e-5, "max": 4e-5, "differ": 8e-6}
    return {"rel": 2e-7, "max": 7e-7, "differ": 3e-6}


# ---- the same in float64, plain torch ---------------------------------------


def _widths(fwhm: float) -> list:
    """Three odd boxcars whose cascade has a Gaussian's variance (Kovesi 2010)."""
    if fwhm <= 0:
        return []
    v = 12.0 * (fwhm * FWHM_TO_SIGMA) ** 2
    lo = int(math.sqrt(v / 3.0 + 1.0))
    lo -= 1 - lo % 2
    m = int(math.floor((v - 3 * lo * lo - 12 * lo - 9) / (-4.0 * lo - 4.0) + 0.5))
    m = min(max(m, 0), 3)
    return [lo] * m + [lo + 2] * (3 - m)


def _spatial_kernel(fwhm: float, sampled: bool) -> list:
    if sampled and fwhm > 0:
        s = fwhm * FWHM_TO_SIGMA
        h = int(math.floor(4.0 * s))
        taps = np.rint(1024.0 * np.exp(-np.arange(-h, h + 1) ** 2 / (2.0 * s * s)))
        return list(taps / taps.sum())
    k = np.ones(1)
    for w in _widths(fwhm):
        k = np.convolve(k, np.full(w, 1.0 / w))
    return list(k)


def _smooth64(c: torch.Tensor, mask: torch.Tensor, fwhm: float, w: int, value: float, sampled: bool) -> torch.Tensor:
    finite = torch.isfinite(c)
    x = torch.where(finite, c, 0.0)
    if value > 0:
        x = torch.where(mask & finite, torch.where(c >= 0, value, -value), x)
    k = _spatial_kernel(fwhm, sampled)
    if len(k) > 1:
        x = _fir(_fir(x, k, 2), k, 1)
    if w > 1:
        x = _fir(x, [1.0 / w] * w, 0)
    return torch.where(finite, x, math.nan)


def _medians(v: torch.Tensor, n: torch.Tensor) -> torch.Tensor:
    """Median of the first n (smallest) values of every row of v, other values +inf."""
    s = torch.sort(v, dim=1).values
    lo, hi = torch.clamp((n - 1) // 2, min=0), torch.clamp(n // 2, max=v.shape[1] - 1)
    return 0.5 * (s.gather(1, lo[:, None]) + s.gather(1, hi[:, None]))[:, 0]


def _noises64(v: torch.Tensor, mode: str) -> torch.Tensor:
    """Noise of the finite values of every row of v (float64); NaN for none."""
    ok = torch.isfinite(v)
    n = ok.sum(dim=1)
    if mode == "std":
        z = torch.where(ok, v, 0.0)
        mean = z.sum(dim=1) / n
        dev = torch.where(ok, v - mean[:, None], 0.0)
        sig = torch.sqrt((dev * dev).sum(dim=1) / torch.clamp(n - 1, min=1))
        return torch.where(n > 0, sig, math.nan)
    m = _medians(torch.where(ok, v, math.inf), n)
    sig = 1.4826 * _medians(torch.where(ok, (v - m[:, None]).abs(), math.inf), n)
    sig = torch.where(n > 0, sig, math.nan)
    if mode == "gauss":
        for i in torch.nonzero(sig > 0)[:, 0].tolist():
            sig[i] = _gauss64(v[i][ok[i]], float(sig[i]))
    return sig


def _gauss64(v: torch.Tensor, sigma_mad: float) -> float:
    """Width of the least-squares Gaussian through 256 bins over +-5 MAD noises."""
    k = np.float32(128.0 / (5.0 * sigma_mad))
    q = torch.floor(v.to(torch.float32) * float(k))
    q = q[(q >= -128) & (q < 128)].to(torch.int64) + 128
    h = torch.bincount(q, minlength=256).cpu().numpy().astype(np.float64)
    x2 = ((np.arange(256) + 0.5) / 128.0 - 1.0) ** 2

    def slope(tau):
        g = np.exp(-x2 / (2.0 * tau * tau))
        return np.sum(g * g) * np.sum(h * x2 * g) - np.sum(h * g) * np.sum(x2 * g * g)

    lo, hi = 0.05, 0.8
    if not (slope(lo) > 0 > slope(hi)):
        return sigma_mad
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if slope(mid) > 0 else (lo, mid)
    return 0.5 * (lo + hi) * 128.0 / float(k)


def _noise64(v: torch.Tensor, mode: str) -> float:
    return float(_noises64(v[torch.isfinite(v)][None, :], mode)[0])


def _run64(cube: torch.Tensor, kernels: list, t: float, mode: str, sampled: bool):
    c = cube.to(torch.float64)
    mask = torch.zeros(c.shape, dtype=torch.bool, device=c.device)
    sigma0 = _noise64(c, mode)
    sigmas = []
    for fwhm, w in kernels:
        s = _smooth64(c, mask, fwhm, w, REPLACEMENT * sigma0, sampled)
        sigmas.append(_noise64(s, mode))
        if sigmas[-1] > 0:
            mask |= s.abs() > t * sigmas[-1]
    return mask.to(torch.uint8), np.array(sigmas), sigma0


def _noise_scale64(cube: torch.Tensor, case: dict) -> torch.Tensor:
    """Every cell divided by the noise of the window around its centre voxel."""
    c = cube.to(torch.float64)
    cells = []
    for n, g, w in zip(c.shape, (case["gz"], case["gy"], case["gx"]), (case["wz"], case["wy"], case["wx"])):
        start = torch.arange(0, n, g, device=DEV)
        centre = start + (torch.clamp(start + g, max=n) - start - 1) // 2
        cells.append(centre[:, None] + torch.arange(-(w // 2), w // 2 + 1, device=DEV)[None, :])
    pad = torch.nn.functional.pad(c, [p for n in (2, 1, 0) for p in (20, 20)], value=math.nan)
    z, y, x = (i + 20 for i in cells)
    sig = torch.empty((z.shape[0], y.shape[0], x.shape[0]), dtype=torch.float64, device=DEV)
    for k in range(z.shape[0]):
        slab = pad[z[k]]
        for j in range(y.shape[0]):
            v = slab[:, y[j]][:, :, x]  # [wz][wy][cells x][wx]
            sig[k, j] = _noises64(v.permute(2, 0, 1, 3).reshape(x.shape[0], -1), case["noise"])
    nz, ny, nx = c.shape
    at = torch.meshgrid(torch.arange(nz, device=DEV) // case["gz"], torch.arange(ny, device=DEV) // case["gy"],
                        torch.arange(nx, device=DEV) // case["gx"], indexing="ij")
    s = sig[at]
    return torch.where((s > 0) & torch.isfinite(c), c / s, math.nan)


def _flags64(noise: torch.Tensor, k: float) -> torch.Tensor:
    v = noise.to(torch.float32).to(torch.float64).reshape(-1)
    good = v[torch.isfinite(v)].cpu().numpy()
    if not good.size:
        return torch.zeros(noise.shape, dtype=torch.bool, device=DEV)
    m = float(np.median(good))
    r = 1.4826 * float(np.median(np.abs(good - m)))
    return ((v - m).abs() > k * r).reshape(noise.shape)


def _autoflag64(cube: torch.Tensor, case: dict) -> dict:
    c = cube.to(torch.float64)
    nz, ny, nx = c.shape
    chan, pix = (torch.zeros(s, dtype=torch.bool, device=DEV) for s in ((nz,), (ny, nx)))
    cn, pn = None, None
    if case["channels"]:
        cn = torch.cat([_noises64(c[z:z + 32].reshape(-1, ny * nx), case["noise"]) for z in range(0, nz, 32)])
        chan = _flags64(cn, case["k"])
    if case["pixels"]:
        pn = torch.stack([_noises64(c[:, y].T.contiguous(), case["noise"]) for y in range(ny)])
        pix = _flags64(pn, case["k"])
    blanked = torch.where(chan[:, None, None] | pix[None] | ~torch.isfinite(c), math.nan, c)
    return dict(cube=blanked, chan=chan.cpu().numpy(), pix=pix.cpu().numpy(),
                chan_noise=None if cn is None else cn.cpu().numpy(),
                pix_noise=None if pn is None else pn.cpu().numpy())


def exact(case: dict, seed: int):
    op = case["op"]
    n = 0 if op == "batch" else case["nx"] * case["ny"] * case["nz"]
    if op == "link" or n > 4e8 or (case.get("noise") == "gauss" and op in ("noise_scale", "autoflag")):
        return None
    data = _inputs(case, seed)
    if op == "run":
        mask, sigmas, sigma0 = _run64(data, KERNEL_LISTS[case["kernels"]], case["t"], case["noise"], case["sampled"])
        return dict(mask=mask, sigmas=sigmas, sigma0=sigma0)
    if op == "half":
        kind = torch.bfloat16 if case["bf16"] else torch.float16
        cube = data[0].view(kind).to(torch.float32) * data[1][:, None, None]
        mask, sigmas, sigma0 = _run64(cube, KERNEL_LISTS[case["kernels"]], case["t"], case["noise"], case["sampled"])
        return dict(mask=mask, sigmas=sigmas, sigma0=sigma0)
    if op == "batch":
        got = [_run64(c, KERNEL_LISTS[case["kernels"]], case["t"], "mad", False) for c in data]
        return dict(masks=[g[0] for g in got], sigmas=np.stack([g[1] for g in got]), sigma0s=np.array([g[2] for g in got]))
    if op == "noise_scale":
        return dict(scaled=_noise_scale64(data, case))
    if op == "autoflag":
        return _autoflag64(data, case)
    cube, mask = data
    return dict(smoothed=_smooth64(cube.to(torch.float64), mask.bool(), case["fwhm"], case["w"], 2.0, case["sampled"]))
