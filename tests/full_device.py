"""A device whose memory is all but taken, for tests of calls beside one."""
import torch

MB = 1 << 20


class FullDevice:
    """Holds all of the device's free memory but `left` bytes."""

    def __init__(self, left):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.held = []
        for unit in (1 << 30, 64 * MB, 2 * MB):
            while True:
                free = torch.cuda.mem_get_info()[0]
                if free - left < unit:
                    break
                try:
                    self.held.append(torch.empty((free - left) // unit * unit, dtype=torch.uint8, device="cuda"))
                except torch.OutOfMemoryError:
                    break
        self.free = torch.cuda.mem_get_info()[0]

    def __enter__(self):
        return self

    def __exit__(self, *a):
        self.held.clear()
        torch.cuda.empty_cache()
