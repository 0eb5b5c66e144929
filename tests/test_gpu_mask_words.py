"""The working mask made from a caller's bytes: whole words by 16-byte loads
against the byte-wise reading of a mask off a 16-byte boundary."""
import pytest
import torch

from paper_2106_15789_gb300 import Context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 31), (1, 1, 32), (1, 1, 33), (3, 5, 64), (4, 33, 65), (7, 64, 64)])
@pytest.mark.parametrize("density", [0.02, 0.5, 1.0])
def test_mask_words(shape, density):
    n = shape[0] * shape[1] * shape[2]
    g = torch.Generator(device="cuda").manual_seed(n)
    cube = torch.randn(shape, generator=g, device="cuda")
    cube[torch.rand(shape, generator=g, device="cuda") < 0.1] = float("nan")
    cube[torch.rand(shape, generator=g, device="cuda") < 0.02] = float("inf")
    values = torch.tensor([1, 2, 128, 255], dtype=torch.uint8, device="cuda")
    mask = values[torch.randint(0, 4, shape, generator=g, device="cuda")]
    mask = mask * (torch.rand(shape, generator=g, device="cuda") < density)
    room = torch.zeros(n + 16, dtype=torch.uint8, device="cuda")
    off = 1 + (-room.data_ptr()) % 16
    shifted = room[off : off + n].view(shape)
    shifted.copy_(mask)
    # a replaced voxel: finite and set, whatever its byte
    want = torch.where((mask != 0) & torch.isfinite(cube), torch.copysign(torch.tensor(2.5, device="cuda"), cube), cube)
    with Context(0, n) as ctx:
        a = ctx.smooth(cube, (3.0, 3), mask=mask, replacement_value=2.5)
        b = ctx.smooth(cube, (3.0, 3), mask=shifted, replacement_value=2.5)
        c = ctx.smooth(want, (3.0, 3))
    assert torch.equal(a.view(torch.int32), b.view(torch.int32))
    ok = torch.isfinite(c)
    assert torch.equal(ok, torch.isfinite(a))
    # the two calls may quantise with different scales: an ulp of |S| < 4
    # (2.4e-7) and the scales' quanta, far below it
    assert float((a[ok] - c[ok]).abs().max() if ok.any() else 0.0) <= 1e-6
