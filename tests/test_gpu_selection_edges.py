"""Windows, planes and spectra at the sizes and values where their selections
change path, against the oracles (tolerances as in test_gpu_noise_scale.py and
test_gpu_flagger.py)."""
import numpy as np
import pytest
import torch

import oracle.flagger as FL
import oracle.noise_scale as NS
from paper_2106_15789_gb300 import Context, sc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = Context(0, 1 << 23)
    yield c
    c.close()


def _values(kind: str, shape, seed: int) -> np.ndarray:
    rng = np.random.default_rng(seed)
    x = rng.standard_normal(shape).astype(np.float32)
    if kind == "ties":  # more equal values in a step than are ranked directly
        x = np.round(x * 2).astype(np.float32)
    elif kind == "constant":
        x[:] = 3.25
    elif kind == "offset":  # the spread far below a power-of-two bin
        x = (x * np.float32(1e-3) + np.float32(100.0)).astype(np.float32)
    elif kind == "outliers":  # a range far wider than the bulk
        x[rng.random(shape) < 0.01] *= np.float32(1e6)
    elif kind == "nan":
        x[rng.random(shape) < 0.4] = np.nan
        x[rng.random(shape) < 0.01] = np.inf
        x[rng.random(shape) < 0.01] = -np.inf
    elif kind == "two":  # half zeros: the median between a tie and the rest
        x[rng.random(shape) < 0.5] = 0.0
    return x


KINDS = ["normal", "ties", "constant", "offset", "outliers", "nan", "two"]


# window sizes around the lane groups (4, 8, 16, 32 voxels), the turns of a
# plane's rows, windows copied whole (up to 20 voxels a thread) and sampled
# ones, rows longer than 32 voxels, and the largest window
@pytest.mark.parametrize("window", [(17, 19, 15), (31, 31, 31), (33, 17, 17), (31, 33, 9), (15, 35, 31), (5, 9, 121),
                                    (101, 21, 21), (1, 31, 601), (601, 31, 1)])
def test_window_shapes(ctx, window):
    w = [min(v, 650) for v in window]
    shape = (w[2] + 3, w[1] + 2, w[0] + 5)
    x = _values("normal", shape, sum(window))
    _, sig = ctx.noise_scale(torch.from_numpy(x).cuda(), window, (w[0], w[1], w[2]), "mad", want_sigma=True)
    np.testing.assert_allclose(sig, NS.noise_grid(x, window, (w[0], w[1], w[2])), rtol=1e-6, atol=0)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("window", [(11, 11, 11), (21, 23, 25), (31, 31, 31)])
def test_window_values(ctx, kind, window):
    x = _values(kind, (40, 37, 45), 5)
    _, sig = ctx.noise_scale(torch.from_numpy(x).cuda(), window, (16, 16, 16), "mad", want_sigma=True)
    np.testing.assert_allclose(sig, NS.noise_grid(x, window, (16, 16, 16)), rtol=1e-6, atol=0)


# planes at and above the size that takes the passes over the cube, with and
# without 16-byte loads, whole runs of 1,024 values and a remainder
@pytest.mark.parametrize("mode", ["mad", "gauss"])
@pytest.mark.parametrize("ny,nx", [(256, 128), (128, 256), (181, 181), (200, 180), (211, 200)])
def test_plane_sizes(ctx, ny, nx, mode):
    x = _values("normal", (5, ny, nx), ny)
    x[3] *= 4
    x[4, 17] = np.nan
    _check_noises(ctx, x, mode, pixels=False)


@pytest.mark.parametrize("kind", KINDS)
def test_plane_values(ctx, kind):
    x = _values(kind, (4, 190, 200), 7)
    x[2] = np.nan  # no finite voxel
    x[3, 1:] = np.nan  # few
    _check_noises(ctx, x, "mad", pixels=False)


# spectra around multiples of the 256 values read at a time and of the warp,
# tiles of 16 pixels and a remainder, the longest spectrum
@pytest.mark.parametrize("nz,nx", [(1, 3), (2, 16), (31, 17), (32, 15), (33, 33), (255, 16), (256, 5), (257, 16),
                                   (1024, 20), (1536, 16)])
@pytest.mark.parametrize("mode", ["mad", "std", "gauss"])
def test_spectrum_lengths(ctx, nz, nx, mode):
    _check_noises(ctx, _values("nan" if nz > 40 else "normal", (nz, 3, nx), nz), mode, channels=False)


@pytest.mark.parametrize("kind", KINDS)
def test_spectrum_values(ctx, kind):
    x = _values(kind, (300, 4, 19), 11)
    x[:, 0, 0] = np.nan
    x[5:, 0, 1] = np.nan
    x[:, 0, 2] = -7.0
    _check_noises(ctx, x, "mad", channels=False)


def _check_noises(ctx, x, mode, channels=True, pixels=True):
    _, _, _, cn, pn = ctx.autoflag(torch.from_numpy(x).cuda(), 1e9, channels, pixels, mode)
    for got, want in ((cn, FL.channel_noise(x, mode) if channels else None),
                      (pn, FL.pixel_noise(x, mode) if pixels else None)):
        if want is None:
            continue
        assert np.array_equal(np.isnan(got), np.isnan(want))
        ok = np.isfinite(want)
        # (a value whose bin the fit's histogram decides in float32 can move by
        # one bin with the noise's last bit: 4e-6 as in test_gpu_gauss.py)
        np.testing.assert_allclose(got[ok], want[ok], rtol=4e-6 if mode == "gauss" else 2.0**-22, atol=0)


# the spectral-only kernel's default form above 2^22 voxels: planes with and
# without 16-byte copies, widths of each form
@pytest.mark.parametrize("shape", [(70, 250, 250), (70, 251, 251)])
@pytest.mark.parametrize("w", [3, 7, 9, 15])
def test_spectral_default_form(ctx, shape, w):
    g = torch.Generator(device="cuda").manual_seed(w)
    c = torch.randn(shape, generator=g, device="cuda")
    c[:, 3, 5:9] = float("nan")
    m = (c.abs() > 3).to(torch.uint8)
    a = ctx.smooth(c, (0.0, w), mask=m, replacement_value=2.0)
    b = ctx.smooth(c, (0.0, w), mask=m, replacement_value=2.0, flags=sc.SC_FLAG_GENERIC)
    assert torch.equal(a.view(torch.int32), b.view(torch.int32))


# short cubes: chunks of a few planes
@pytest.mark.parametrize("nz", [1, 2, 4, 5, 7, 13, 33])
def test_short_chunks(ctx, nz):
    g = torch.Generator(device="cuda").manual_seed(nz)
    c = torch.randn((nz, 70, 72), generator=g, device="cuda")
    kernels = [(0.0, 0), (0.0, 3), (3.0, 0), (3.0, 3), (3.0, 15), (6.0, 0), (6.0, 7), (6.0, 31)]
    a = ctx.run(c, kernels, 3.0)
    b = ctx.run(c, kernels, 3.0, flags=sc.SC_FLAG_GENERIC)
    assert torch.equal(a[0], b[0]) and a[1] == b[1] and a[2] == b[2]


def test_planes_on_either_side_of_the_passes(ctx):
    """The same finite values in planes of the size that takes the passes over
    the cube and in smaller ones that a block streams: the same noise to the
    last bit (an even count, whose |x - m| is rounded from two middle values)."""
    nz, n = 200, 106 * 307  # below 2^15, with 400 blanked voxels above it
    x = np.random.default_rng(3).standard_normal((nz, n)).astype(np.float32)
    x += np.linspace(0, 30, nz, dtype=np.float32)[:, None]
    big = np.full((nz, 181 * 182), np.nan, dtype=np.float32)
    big[:, :n] = x
    noises = [ctx.autoflag(torch.from_numpy(a.reshape(shape)).cuda(), 1e9, True, False, "mad")[3]
              for a, shape in ((x, (nz, 106, 307)), (big, (nz, 181, 182)))]
    np.testing.assert_array_equal(noises[0], noises[1])
