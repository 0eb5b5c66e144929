"""The flagger's channel noises in groups of channels: cubes whose scratch is
above its bound, and a device that is all but full, where the groups are smaller
or the channels are measured by a block each. The noises are those of the
channels measured a few at a time, to the last bit."""
import numpy as np
import pytest
import torch

from full_device import MB, FullDevice
from paper_2106_15789_gb300 import Context

pytestmark = pytest.mark.gpu

SHAPE = (140, 4096, 4096)  # 8.4 MB of scratch a channel: 127 channels are the most of a group


def _noises(ctx, cube, mode):
    ctx.stats(reset=True)
    return ctx.autoflag(cube, 1e9, True, False, mode, out=cube)[3]  # (nothing is flagged: the cube stays)


def _groups(ctx):
    """Groups of the last call, from its launches: five each (or one kernel for
    all channels: 0), then the statistics, the flags and the blanked cube."""
    n = ctx.stats()["launches"] - 3
    return n // 5 if n > 1 else 0


def _cube():
    g = torch.Generator(device="cuda").manual_seed(5)
    cube = torch.randn(SHAPE, generator=g, device="cuda")
    cube *= torch.linspace(0.5, 2.0, SHAPE[0], device="cuda")[:, None, None]
    cube[3, 17] = float("nan")
    cube[5] = float("nan")
    return cube


@pytest.mark.parametrize("mode", ["mad", "gauss"])
def test_groups_of_channels(mode):
    cube = _cube()
    with Context(0, 1 << 16) as ctx:
        want = np.concatenate([_noises(ctx, cube[z:z + 20], mode) for z in range(0, SHAPE[0], 20)])
    with Context(0, 1 << 16) as ctx:
        before = torch.cuda.mem_get_info()[0]
        np.testing.assert_array_equal(_noises(ctx, cube, mode), want)
        assert _groups(ctx) == 2
        assert before - torch.cuda.mem_get_info()[0] < (1024 + 96 + 8) * MB  # the scratch, 5 bytes a pixel, rounding


# memory for a few of the 70 channels of a group, and for none (the half plane
# that loads the kernels leaves 4 MB)
@pytest.mark.parametrize("left,few", [(30, True), (3, False)])
def test_groups_beside_a_full_device(left, few):
    cube = _cube()
    with Context(0, 1 << 16) as ctx:
        want = _noises(ctx, cube, "mad")
    with Context(0, 1 << 16) as ctx:
        _noises(ctx, cube[:1, :64, :64].contiguous(), "mad")  # (the kernels are loaded)
        _noises(ctx, cube[:1, :, :2048].contiguous(), "mad")
        _noises(ctx, cube[:1].contiguous(), "std")  # 5 bytes a pixel; no scratch
        torch.cuda.synchronize()
        with FullDevice(left * MB):
            first = _noises(ctx, cube, "mad")
            assert (_groups(ctx) > 2) if few else (_groups(ctx) == 0)
            second = _noises(ctx, cube, "mad")
    np.testing.assert_array_equal(first, want)
    np.testing.assert_array_equal(second, want)
