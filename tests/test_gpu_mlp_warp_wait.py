"""A bounded wait of the network kernels' epilogue warps gives every lane the
same answer: half a warp sees another role's failure and gives up, the other
half sees the barrier complete a moment later (nothing waits without end)."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PROBE = r"""
#include "dm_mlp_fused.cu"
namespace dm { void set_error(const std::string &) {} }
using namespace dm;
// warp 0 waits, its lower half with `failed` set; warp 1 arrives 50 ms later
__global__ void k_probe(int failed, int *out) {
  __shared__ uint64_t bar;
  __shared__ int flags[2];
  if (threadIdx.x == 0) {
    tc::mbar_init(&bar, 1);
    flags[0] = failed;
    flags[1] = 0;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    out[threadIdx.x] = wait_warp(&bar, 0, &flags[threadIdx.x / 16]);
  } else if (threadIdx.x == 32) {
    for (int k = 0; k < 50; ++k) __nanosleep(1000000);
    arrive(&bar);
  }
}
extern "C" int probe(int failed, int *out) {
  int *d = nullptr;
  if (cudaMalloc(&d, 32 * sizeof(int)) != cudaSuccess) return 1;
  k_probe<<<1, 64>>>(failed, d);
  const cudaError_t e = cudaMemcpy(out, d, 32 * sizeof(int), cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)e;
}
"""


def test_every_lane_gets_one_answer(tmp_path):
    from paper_2311_18126_gb300 import build as b
    (tmp_path / "probe.cu").write_text(PROBE)
    so = str(tmp_path / "libprobe.so")
    subprocess.run([b._nvcc(), *b.ARCH, *b.NVCC_FLAGS, "-shared", "-I", b.CSRC, "-o", so, str(tmp_path / "probe.cu"),
                    "-lcudart"], check=True)
    L = ctypes.CDLL(so)
    out = np.full(32, -1, np.int32)
    for failed in (0, 1):
        assert L.probe(failed, out.ctypes.data_as(ctypes.c_void_p)) == 0
        assert np.array_equal(out, np.full(32, 1 - failed)), out
