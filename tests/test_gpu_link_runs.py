"""The linker's bits and runs where they can go wrong: masks off a 16-byte
boundary, chunks and words that rows straddle, more runs or detections than a
fresh context has room for (the call starts over), a second call in the room
of the first, values other than 1."""
import numpy as np
import pytest
import torch

import oracle.linker as LK
from paper_2106_15789_gb300 import Context

pytestmark = pytest.mark.gpu


def _check(ctx, mask_np, r_xy, r_z, offset=0, **filt):
    flat = torch.zeros(mask_np.size + 16, dtype=torch.uint8, device="cuda")
    mask = flat[offset:offset + mask_np.size].view(mask_np.shape)
    mask.copy_(torch.from_numpy(mask_np))
    lab, n, ext = ctx.link(mask, r_xy, r_z, **filt)
    ref, ext_ref = LK.link(mask_np, r_xy, r_z, **filt)
    np.testing.assert_array_equal(lab.cpu().numpy(), ref.astype(np.int32))
    np.testing.assert_array_equal(ext.astype(np.int64), ext_ref)
    assert n == int(ref.max())


# rows shorter and longer than a word, a word, and a chunk of 8,192 voxels
@pytest.mark.parametrize("shape", [(5, 40, 31), (5, 40, 32), (5, 40, 33), (600, 30, 1), (2, 3, 8191), (2, 3, 8192),
                                   (2, 3, 8193), (3, 2, 20000)])
@pytest.mark.parametrize("offset", [0, 1])
def test_shapes(shape, offset):
    rng = np.random.default_rng(sum(shape))
    m = (rng.random(shape) < 0.4).astype(np.uint8) * rng.integers(1, 256, shape, dtype=np.uint8)
    m[:, 0, : shape[2] // 2] = 128  # a long run across words
    with Context(0, 1 << 16) as ctx:
        _check(ctx, m, 2, 1, offset)


@pytest.mark.parametrize("r_xy,r_z,density", [(0, 0, 0.3), (1, 1, 0.3), (32, 3, 0.002)])
def test_room_grows_and_is_kept(r_xy, r_z, density):
    rng = np.random.default_rng(4)
    big = (rng.random((96, 128, 160)) < density).astype(np.uint8)
    with Context(0, 1 << 16) as ctx:
        _check(ctx, (rng.random((7, 9, 11)) < 0.3).astype(np.uint8), 1, 1)
        _check(ctx, big, r_xy, r_z)
        _check(ctx, big[:40], r_xy, r_z, min_xy=2, min_z=1)
        _check(ctx, np.zeros((4, 5, 6), np.uint8), 1, 1)


def test_restart_in_recycled_memory():
    """A context whose buffer holds another owner's bytes (all ones: totals of
    -1) and whose first mask needs more room than the first buffer has."""
    rng = np.random.default_rng(6)
    m = (rng.random((96, 128, 160)) < 0.3).astype(np.uint8)
    for _ in range(2):
        room = [torch.full((1 << 24,), -1, dtype=torch.int32, device="cuda") for _ in range(4)]
        torch.cuda.synchronize()
        del room
        torch.cuda.empty_cache()  # given back to the driver, for the context to take
        with Context(0, 1 << 16) as ctx:
            _check(ctx, m, 1, 1, min_xy=2)
