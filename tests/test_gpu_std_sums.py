"""STD mode's sums, before the noise is rounded to float32, against exact
integer sums: as good as float64 sums about the mean. The library's own
launchers are called through a small program linked to it."""
import ctypes
import math
import os
import subprocess
from fractions import Fraction

import pytest
import torch

from paper_2106_15789_gb300 import build, sc

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "sc_internal.h"
using namespace sc;
// sigma of x[0 .. n) before its rounding to float32; -1 on an error.
extern "C" double std_noise(const float* x, long long n, int sms) {
  DevState* st = nullptr;
  unsigned long long* hist = nullptr;
  double d = -1.0;
  Lists L{};
  if (cudaMalloc(&st, sizeof(DevState)) == cudaSuccess && cudaMalloc(&hist, 8 * kNumBins) == cudaSuccess &&
      cudaMemset(st, 0, sizeof(DevState)) == cudaSuccess && cudaMemset(hist, 0, 8 * kNumBins) == cudaSuccess &&
      launch_hist(x, n, st, hist, 0, 0, sms, 0) == cudaSuccess &&
      launch_plan(st, hist, 0, x, n, L, 1.0f, 0, 1, 0u, 0) == cudaSuccess &&
      launch_std(x, n, st, SC_MAX_KERNELS, sms, 0) == cudaSuccess)
    if (cudaMemcpy(&d, reinterpret_cast<char*>(st) + offsetof(DevState, sigma_cur_d), 8, cudaMemcpyDeviceToHost) !=
        cudaSuccess)
      d = -1.0;
  cudaFree(st);
  cudaFree(hist);
  return d;
}
"""


@pytest.fixture(scope="module")
def std_noise(tmp_path_factory):
    d = tmp_path_factory.mktemp("std")
    (d / "std.cu").write_text(PROGRAM)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I",
                    os.path.join(ROOT, "include"), "-I", build.CSRC, str(d / "std.cu"), sc.LIB_PATH, "-Xlinker",
                    f"-rpath={os.path.dirname(sc.LIB_PATH)}", "-o", str(d / "libstd.so")], check=True)
    f = ctypes.CDLL(str(d / "libstd.so")).std_noise
    f.restype = ctypes.c_double
    f.argtypes = [ctypes.c_void_p, ctypes.c_longlong, ctypes.c_int]
    with sc_context():  # raises the kernels' shared-memory limits
        yield f


def sc_context():
    from paper_2106_15789_gb300 import Context

    return Context(0, 1 << 10)


BITS = 20  # the values are multiples of 2^-20 below 8: 24-bit integers


@pytest.mark.parametrize("kind,mean,sd", [("noise", 0.0, 1.0), ("tail", 0.0, 0.05), ("mean", 5.0, 0.7),
                                          ("offset", 7.3, 0.03), ("far", 7.77, 0.001)])
@pytest.mark.parametrize("n", [1000, 300001, 1 << 21, 38_400_000, 1 << 27])
def test_std_sums(std_noise, kind, mean, sd, n):
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randn(n, generator=g, device="cuda") * sd + mean
    if kind == "tail":
        x[::997] *= 100
    i = (x.double() * 2**BITS).round_().clamp_(-(2**23) + 1, 2**23 - 1).to(torch.int64)
    x = (i.double() / 2**BITS).float()
    s1, lo = int(i.sum()), i & 0xFFF
    i >>= 12
    s2 = (int((i * i).sum()) << 24) + (int((i * lo).sum()) << 13) + int((lo * lo).sum())
    var = Fraction(n * s2 - s1 * s1, n * (n - 1) << 2 * BITS)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    got = Fraction(std_noise(x.data_ptr(), n, sms))
    assert got > 0
    # up to 6 blocks an SM add their float64 sums in any order: 2^-53 sqrt(912)
    # of S2, half of that in sigma, and four times as much as the bound (two
    # passes of float64 sums give 2^-50 here, sums in pairs of floats 2^-44)
    assert abs(float((got * got - var) / var)) / 2 <= 2.0**-47, math.log2(abs(float((got * got - var) / var)) / 2)
