"""A wait between the blocks of a contact system's factorisation that runs out
is told apart from a zero pivot.  dm_contact.cu is built with two small
launchers: one block meets a second one that is never launched (a bounded
wait: it gives up after a second or so and returns), and the substitution is
given each reason to stop."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

PROBE = r"""
#include "dm_contact.cu"
namespace dm {
void set_error(const std::string &) {}
__global__ void k_probe_meeting(int32_t *bar, int32_t *bad, int32_t *met) {
  int target = 0;
  lu_arrive(bar, 2, target);
  *met = lu_wait(bar, bad, 2, target, false);
}
}  // namespace dm
using namespace dm;
// ints on the device: [0] meeting counter, [1] reason, [2] met; returns the reason
extern "C" int probe_meeting(int *met) {
  int32_t *d = nullptr, h[3] = {0, 0, -1};
  if (cudaMalloc(&d, sizeof(h)) != cudaSuccess) return -1;
  cudaMemcpy(d, h, sizeof(h), cudaMemcpyHostToDevice);
  k_probe_meeting<<<1, 32>>>(d, d + 1, d + 2);
  const cudaError_t e = cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost);
  cudaFree(d);
  *met = h[2];
  return e == cudaSuccess ? h[1] : -1;
}
// the status a system gets whose factorisation stopped for `reason`
extern "C" int probe_status(int reason) {
  // [0] contact system -> system, [1] go, [2] reason, [3] status, [4] active, [5..8] counters
  int32_t *d = nullptr, h[9] = {0, 1, reason, 0, 1, 0, 0, 1 << 30, 0};
  if (cudaMalloc(&d, sizeof(h)) != cudaSuccess) return -1;
  cudaMemcpy(d, h, sizeof(h), cudaMemcpyHostToDevice);
  ContactArgs a{};
  SolveArgs v{};
  a.contact_sys = d, a.cgo = d + 1, a.cbad = d + 2;
  v.sys_status = d + 3, v.sys_active = d + 4, v.ctrl = d + 5;
  k_cc_subst<<<1, 32 * kSubstWarps>>>(a, v);
  const cudaError_t e = cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e == cudaSuccess && h[4] == 0 && h[6] == 1 && h[7] == 0 ? h[3] : -1;
}
"""
DM_ERR_DEGENERATE, DM_ERR_CUDA = 4, 6


def test_timeout_is_not_a_zero_pivot(tmp_path):
    from paper_2311_18126_gb300 import build as b
    (tmp_path / "probe.cu").write_text(PROBE)
    so = str(tmp_path / "libprobe.so")
    subprocess.run([b._nvcc(), *b.ARCH, *b.NVCC_FLAGS, "-shared", "-I", b.CSRC, "-o", so, str(tmp_path / "probe.cu"),
                    "-lcudart"], check=True)
    L = ctypes.CDLL(so)
    met = ctypes.c_int(-1)
    reason = L.probe_meeting(ctypes.byref(met))
    assert met.value == 0 and reason > 0
    assert L.probe_status(reason) == DM_ERR_CUDA
    zero_pivot = 1
    assert reason != zero_pivot and L.probe_status(zero_pivot) == DM_ERR_DEGENERATE
