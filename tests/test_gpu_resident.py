"""Measurements beside a kernel of the program that keeps a whole SM: they go on
with the other SMs, and do not wait for its end. The kernel ends by itself
after the time it is given."""
import ctypes
import subprocess

import pytest
import torch

from paper_2106_15789_gb300 import Context, build, sc

pytestmark = pytest.mark.gpu

SOURCE = r"""
// One block that keeps its SM's shared memory for ns nanoseconds (less than 2^30).
__global__ void __launch_bounds__(1024) k_keep(unsigned long long ns) {
  extern __shared__ unsigned char room[];
  unsigned long long t0, t = 0;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  if (threadIdx.x == 0) room[0] = 1;
  for (int i = 0; i < (1 << 24) && t < ns; ++i) {
    __nanosleep(1000);
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    t -= t0;
  }
}
extern "C" int keep(unsigned long long ns, int smem, void* stream) {
  if (cudaFuncSetAttribute(k_keep, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return 1;
  k_keep<<<1, 1024, smem, (cudaStream_t)stream>>>(ns & ((1ull << 30) - 1));
  return cudaGetLastError() != cudaSuccess;
}
"""

KEEP_NS, SMEM = 500_000_000, 220 << 10  # 0.5 s; an SM has 227 KB for one block


@pytest.fixture(scope="module")
def keep(tmp_path_factory):
    d = tmp_path_factory.mktemp("keep")
    (d / "keep.cu").write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, "-shared", "-Xcompiler", "-fPIC", str(d / "keep.cu"), "-o",
                    str(d / "libkeep.so")], check=True)
    f = ctypes.CDLL(str(d / "libkeep.so")).keep
    f.argtypes = [ctypes.c_ulonglong, ctypes.c_int, ctypes.c_void_p]
    return f


# arrays of more than 2^21 values, whose selection has its full passes behind
# it; forced, the passes do their work
@pytest.mark.parametrize("call", ["run", "noise", "noise_forced", "static"])
def test_does_not_wait_for_a_resident_kernel(keep, call):
    g = torch.Generator(device="cuda").manual_seed(1)
    cube = torch.randn((40, 256, 260), generator=g, device="cuda")
    side = torch.cuda.Stream()
    with Context(0, cube.numel()) as ctx:

        def measure():
            if call == "run":
                return ctx.run(cube, [(0.0, 0), (3.0, 3), (3.0, 7)], 3.5)[1]
            if call == "static":
                return sc.sc_noise_static(cube)
            return ctx.noise(cube, flags=sc.SC_FLAG_NO_FAST_SELECT if call == "noise_forced" else 0)

        assert keep(1000, SMEM, ctypes.c_void_p(side.cuda_stream)) == 0  # (both are loaded)
        want = measure()
        torch.cuda.synchronize()
        done = torch.cuda.Event()
        assert keep(KEEP_NS, SMEM, ctypes.c_void_p(side.cuda_stream)) == 0
        done.record(side)
        got = measure()  # returns with the noises, on the host
        still = not done.query()
        torch.cuda.synchronize()
    assert still, "the measurement waited for the resident kernel"
    assert got == want
