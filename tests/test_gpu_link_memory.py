"""The linker beside a device that is all but full: a call goes on with the
memory that its mask needs, and gives the labels of a call with room. A file of
its own, since it takes the device's memory for a moment."""
import numpy as np
import pytest
import torch

from full_device import MB, FullDevice
from paper_2106_15789_gb300 import Context

pytestmark = pytest.mark.gpu


def _boxes(shape, count, seed, gap):
    """A mask of boxes; gap: only every gap-th voxel of their rows is set."""
    rng = np.random.default_rng(seed)
    m = np.zeros(shape, dtype=np.uint8)
    for _ in range(count):
        z, y, x = (int(rng.integers(0, n - 24)) for n in shape)
        m[z:z + rng.integers(1, 20), y:y + rng.integers(1, 20), x:x + rng.integers(1, 24):gap] = 1
    return torch.from_numpy(m).cuda()


# few runs and detections (a few hundred KB); more than the first tight room
# has, and a detection per few voxels
@pytest.mark.parametrize("gap,r_xy,count", [(1, 2, 500), (2, 1, 3000), (3, 2, 3000)])
def test_link_beside_a_full_device(gap, r_xy, count):
    shape = (250, 500, 512)  # 64 M voxels: a context keeps 36 MB for them
    mask = _boxes(shape, count, gap, gap)
    labels = torch.empty(shape, dtype=torch.int32, device="cuda")
    with Context(0, 1 << 16) as ctx:
        want, n, ext = ctx.link(mask, r_xy, 1, min_xy=2)
    with Context(0, 1 << 16) as ctx:
        ctx.link(mask[:3], r_xy, 1)  # (the kernels are loaded)
        with FullDevice(24 * MB) as full:
            assert full.free < 32 * MB
            _, n1, ext1 = ctx.link(mask, r_xy, 1, min_xy=2, labels=labels)
        assert n1 == n and np.array_equal(ext1, ext) and torch.equal(labels, want)
        labels.fill_(-1)
        _, n2, ext2 = ctx.link(mask, r_xy, 1, min_xy=2, labels=labels)  # with room again
        assert n2 == n and np.array_equal(ext2, ext) and torch.equal(labels, want)


def test_room_of_a_dense_mask_is_given_up():
    """After a mask with many runs, a larger cube with few of them, where there
    is no memory for the larger cube and that many runs."""
    dense = torch.zeros((64, 256, 512), dtype=torch.uint8, device="cuda")
    dense[:, :, ::2] = 1  # 4 M runs: 34 MB
    shape = (250, 500, 512)
    mask = _boxes(shape, 300, 9, 1)
    labels = torch.empty(shape, dtype=torch.int32, device="cuda")
    with Context(0, 1 << 16) as ctx:
        want, n, ext = ctx.link(mask, 1, 1)
    with Context(0, 1 << 16) as ctx:
        assert ctx.link(dense, 2, 0)[1] == 64
        with FullDevice(8 * MB):  # with the 39 MB that the context holds: not for 34 + 20 + 9
            _, n1, ext1 = ctx.link(mask, 1, 1, labels=labels)
        assert n1 == n and np.array_equal(ext1, ext) and torch.equal(labels, want)
