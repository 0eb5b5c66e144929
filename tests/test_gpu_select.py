"""Median and MAD selection from the candidate lists (one thread-block cluster)
against numpy, at the sizes where its paths change: lists of one block and of
the whole cluster, arrays up to 2^21 values (full passes by the cluster) and
above (full passes by the grid)."""
import numpy as np
import pytest
import torch

from paper_2106_15789_gb300 import Context, sc

pytestmark = pytest.mark.gpu

ALL_MAX = 1 << 21  # kSelectAllMax
GRID_MIN = 1 << 25  # kSelectGridMin


def _data(kind: str, n: int) -> np.ndarray:
    rng = np.random.default_rng(n)
    x = rng.standard_normal(n).astype(np.float32)
    if kind == "zeros":  # blanked with zeros: the median's bin holds 3 % of the values
        x[rng.random(n) < 0.03] = 0.0
    elif kind == "ties":  # few distinct values, most order statistics tied
        x = np.round(x * 4).astype(np.float32)
    elif kind == "offset":  # the MAD far below the median, keys of either sign of s - m
        x = (x * np.float32(1e-3) + np.float32(7.0)).astype(np.float32)
    elif kind == "wide":  # magnitudes over many octaves, NaN and Inf among them
        x = (x * np.exp(rng.uniform(-60, 60, n))).astype(np.float32)
        x[rng.random(n) < 0.01] = np.nan
        x[rng.random(n) < 0.001] = np.inf
    return x


def _sigma(x: np.ndarray) -> float:
    v = x[np.isfinite(x)].astype(np.float64)

    def median(a):
        lo, hi = (a.size - 1) // 2, a.size // 2
        p = np.partition(a, [lo, hi])
        return 0.5 * (p[lo] + p[hi])

    keys = np.abs(v - median(v)).astype(np.float32).astype(np.float64)
    return float(np.float32(1.4826 * median(keys)))


@pytest.mark.parametrize("kind", ["normal", "zeros", "ties", "offset", "wide"])
@pytest.mark.parametrize("n", [1, 2, 3, 1023, 2048, 16384, 16385, 70000, 300001, ALL_MAX - 1, ALL_MAX, ALL_MAX + 1,
                               3000000])
def test_noise_selection(kind, n):
    x = _data(kind, n)
    if not np.isfinite(x).any():
        x[0] = 1.0
    d = torch.from_numpy(x).cuda()
    with Context(0, n) as ctx:
        got = ctx.noise(d)
        full = ctx.noise(d, flags=sc.SC_FLAG_NO_FAST_SELECT)
    want = _sigma(x)
    # the library's sigma is a float32; forming |s - m| in float64 first, as
    # numpy does here, can round differently by at most one unit of it
    assert abs(got - want) <= 2.0**-23 * abs(want), (got, want)
    assert got == full


@pytest.mark.parametrize("kind,n", [("normal", GRID_MIN), ("normal", GRID_MIN + 1), ("normal", GRID_MIN + 2),
                                    ("offset", GRID_MIN + 3), ("ties", GRID_MIN + 4), ("zeros", GRID_MIN + 5)])
def test_noise_selection_long_lists(kind, n):
    test_noise_selection(kind, n)


@pytest.mark.parametrize("shape", [(16, 300, 301), (40, 256, 260), (64, 256, 256)])  # below, above and at 2^21 + 2^21
def test_run_with_full_selection_passes(shape):
    """A cube with zero-filled voxels (a candidate set above capacity) gives
    the same run with and without the forced full passes."""
    g = torch.Generator(device="cuda").manual_seed(3)
    cube = torch.randn(shape, generator=g, device="cuda")
    cube[:, :40] = 0.0
    kernels = [(0.0, 0), (0.0, 3), (3.0, 0), (3.0, 3)]
    with Context(0, cube.numel()) as ctx:
        a = ctx.run(cube, kernels, 3.5)
        b = ctx.run(cube, kernels, 3.5, flags=sc.SC_FLAG_NO_FAST_SELECT)
    assert a[1] == b[1] and a[2] == b[2]
    assert torch.equal(a[0], b[0])


@pytest.mark.parametrize("n", [1, 2, 3, 255, 4097, 300001])
@pytest.mark.parametrize("kind", ["normal", "offset", "far", "outlier", "wide"])
def test_std(kind, n):
    """STD mode's sums in pairs of floats: shifts far from the mean, magnitudes
    at both ends of float32, unaligned data."""
    x = _data({"far": "normal", "outlier": "normal"}.get(kind, kind), n)
    if kind == "far":  # the spread below the width of the median's bin
        x = (np.float32(1.0e6) + x * np.float32(0.5)).astype(np.float32)
    elif kind == "outlier":
        x[n // 2] = 3.0e37
    if not np.isfinite(x).any():
        x[0] = 1.0
    d = torch.from_numpy(np.concatenate([x[:1], x])).cuda()[1:]  # rows start 4 bytes off a 16-byte boundary
    v = x[np.isfinite(x)].astype(np.float64)
    want = float(np.sqrt(((v - v.mean()) ** 2).sum() / (v.size - 1))) if v.size > 1 else 0.0
    with Context(0, n + 1) as ctx:
        got = ctx.noise(d, "std")
    # one float32 rounding of the result; the sums are good to 2^-47
    assert abs(got - want) <= 2.0**-24 * 1.01 * abs(want), (got, want)


@pytest.mark.parametrize("shapes", [[(40, 230, 230)] * 3, [(40, 230, 230), (9, 250, 251), (64, 256, 256)]])
def test_full_selection_passes_on_lanes(shapes):
    """Forced full passes of cubes side by side and of one cube alone give the
    listed selection's run."""
    g = torch.Generator(device="cuda").manual_seed(4)
    cubes = [torch.randn(s, generator=g, device="cuda") for s in shapes]
    kernels = [(0.0, 0), (3.0, 3)]
    with Context(0, max(c.numel() for c in cubes)) as ctx:
        masks, sig, sig0 = ctx.run_batch(cubes, kernels, 3.5, flags=sc.SC_FLAG_NO_FAST_SELECT)
        for i, c in enumerate(cubes):
            for flags in (0, sc.SC_FLAG_NO_FAST_SELECT):
                m, s, s0 = ctx.run(c, kernels, 3.5, flags=flags)
                assert list(s) == list(sig[i]) and s0 == sig0[i]
                assert torch.equal(m, masks[i])
