"""The raw cube's histogram window of cubes that are blank but for a few voxels:
the sample it is placed by goes on until it has found some. The library's own
launcher is called through a small program linked to it."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2106_15789_gb300 import Context, build, sc

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
BELOW = 20  # octaves of the window under the median's

PROGRAM = r"""
#include "sc_internal.h"
using namespace sc;
// Exponent field of the window's lowest bin; -1 on an error.
extern "C" int window_base(const float* x, long long n) {
  DevState* st = nullptr;
  int e = -1;
  if (cudaMalloc(&st, sizeof(DevState)) == cudaSuccess && cudaMemset(st, 0, sizeof(DevState)) == cudaSuccess &&
      launch_window_from_sample(x, nullptr, n, n, st, 0) == cudaSuccess)
    if (cudaMemcpy(&e, reinterpret_cast<char*>(st) + offsetof(DevState, win) + offsetof(BinCfg, e_base), 4,
                   cudaMemcpyDeviceToHost) != cudaSuccess)
      e = -1;
  cudaFree(st);
  return e;
}
"""


@pytest.fixture(scope="module")
def window_base(tmp_path_factory):
    d = tmp_path_factory.mktemp("window")
    (d / "window.cu").write_text(PROGRAM)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I",
                    os.path.join(ROOT, "include"), "-I", build.CSRC, str(d / "window.cu"), sc.LIB_PATH, "-Xlinker",
                    f"-rpath={os.path.dirname(sc.LIB_PATH)}", "-o", str(d / "libwindow.so")], check=True)
    f = ctypes.CDLL(str(d / "libwindow.so")).window_base
    f.argtypes = [ctypes.c_void_p, ctypes.c_longlong]
    with Context(0, 1 << 10):  # raises the kernels' shared-memory limits
        yield f


# every voxel finite, and one in 8,000 (one expected in the first sample, eight
# in all of them); cubes smaller than a sample, a little larger, and large
@pytest.mark.parametrize("n,finite", [(1, 1), (5000, 3), (8192, 1), (9000, 400), (1 << 20, 1 << 20), (1 << 24, 2097),
                                      (100_000_003, 12_500)])
@pytest.mark.parametrize("seed", range(6))
def test_window_finds_the_finite_voxels(window_base, n, finite, seed):
    rng = np.random.default_rng(seed)
    x = torch.full((n,), float("nan"), device="cuda")
    at = torch.from_numpy(np.sort(rng.choice(n, finite, replace=False)) if n < 1 << 22 else rng.integers(0, n, finite))
    scale = 2.0 ** rng.integers(-40, 40)
    x[at.cuda()] = (torch.from_numpy(rng.uniform(1.0, 2.0, finite).astype(np.float32)) * scale).cuda()
    e = 127 + int(np.log2(scale)) - BELOW
    # the upper edge of the median's bin: its own octave or the next
    assert window_base(x.data_ptr(), n) in (e, e + 1)
