"""Launch shapes of the contact systems' factorisation (CPU): dm_contact.cu's
host code with stand-ins for the CUDA calls that report the device's attributes
and launch.  Several blocks of a system wait for one another, so more than one
needs a cooperative launch; without those, and under MPS, there is one."""
import ctypes
import os
import subprocess

import pytest

PROBE = r"""
#include <cuda_runtime.h>
namespace probe {
int coop, mps, grid[2][3], cooperative, launches;
cudaError_t device(int *d) { return *d = 0, cudaSuccess; }
cudaError_t attribute(int *v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrCooperativeLaunch ? coop : a == cudaDevAttrMpsEnabled ? mps : 0;
  return cudaSuccess;
}
template <class... T>
cudaError_t launch(const cudaLaunchConfig_t *c, T...) {
  int *g = grid[launches & 1];
  g[0] = c->gridDim.x, g[1] = c->gridDim.y, g[2] = c->gridDim.z;
  if (launches++ == 0)
    cooperative = c->numAttrs == 1 && c->attrs[0].id == cudaLaunchAttributeCooperative && c->attrs[0].val.cooperative;
  return cudaSuccess;
}
}  // namespace probe
#define cudaGetDevice probe::device
#define cudaDeviceGetAttribute probe::attribute
#define cudaLaunchKernelEx probe::launch
#include "dm_contact.cu"
namespace dm { void set_error(const std::string &) {} }
// blocks of the factorisation per system, negative where the launch is cooperative
extern "C" int probe_blocks(int coop, int mps, int systems, int tiles, int sms) {
  probe::coop = coop, probe::mps = mps, probe::launches = 0;
  dm::ContactArgs a{};
  dm::SolveArgs v{};
  a.n_contact = systems, a.max_tiles = tiles;
  (void)dm::lu_solve(a, v, sms, nullptr);
  if (probe::launches != 2 || probe::grid[0][0] != systems) return 0;
  return probe::cooperative ? -probe::grid[0][1] : probe::grid[0][1];
}
"""


@pytest.fixture(scope="module")
def blocks(tmp_path_factory):
    from paper_2311_18126_gb300 import build as b
    d = tmp_path_factory.mktemp("launch")
    (d / "probe.cu").write_text(PROBE)
    so = str(d / "libprobe.so")
    subprocess.run([b._nvcc(), *b.ARCH, "-O0", "-Xptxas", "-O0", "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler",
                    "-fPIC", "-shared", "-I", b.CSRC, "-o", so, str(d / "probe.cu"), "-lcudart"], check=True)
    return ctypes.CDLL(so).probe_blocks


@pytest.mark.parametrize("coop,mps,systems,tiles,want", [
    (1, 0, 1, 63, -152), (1, 0, 4, 38, -38), (1, 0, 1, 2, -16), (1, 0, 76, 8, -2),
    (1, 0, 77, 8, 1), (1, 0, 70000, 1, 1),                  # more systems than half the SMs
    (0, 0, 1, 63, 1), (1, 1, 1, 63, 1), (0, 1, 4, 38, 1),   # no cooperative launches to be had
])
def test_blocks_per_system(blocks, coop, mps, systems, tiles, want):
    assert blocks(coop, mps, systems, tiles, 152) == want
