"""The reciprocal and the square root that kernels form from integer and FP32
pieces (dm_kernels.cuh), against exact arithmetic."""
import ctypes
import subprocess
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PROBE = r"""
#include "dm_kernels.cuh"
__global__ void k_probe(int op, int n, const double *x, double *y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = op == 0 ? dm::rcp_any(x[i]) : dm::sqrt_any(x[i]);
}
extern "C" int probe(int op, int n, const double *x, double *y) {
  double *d = nullptr;
  if (cudaMalloc(&d, 2 * sizeof(double) * n) != cudaSuccess) return 1;
  cudaMemcpy(d, x, sizeof(double) * n, cudaMemcpyHostToDevice);
  k_probe<<<(n + 255) / 256, 256>>>(op, n, d, d + n);
  const cudaError_t e = cudaMemcpy(y, d + n, sizeof(double) * n, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)e;
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_2311_18126_gb300 import build as b
    d = tmp_path_factory.mktemp("arithmetic")
    (d / "probe.cu").write_text(PROBE)
    so = str(d / "libprobe.so")
    subprocess.run([b._nvcc(), *b.ARCH, *b.NVCC_FLAGS, "-shared", "-I", b.CSRC, "-o", so, str(d / "probe.cu"),
                    "-lcudart"], check=True)
    L = ctypes.CDLL(so)

    def run(op, x):
        x = np.ascontiguousarray(x, np.float64)
        y = np.empty_like(x)
        P = ctypes.POINTER(ctypes.c_double)
        assert L.probe(op, x.size, x.ctypes.data_as(P), y.ctypes.data_as(P)) == 0
        return y
    return run


def test_reciprocal(probe):
    rng = np.random.default_rng(1)
    d = np.concatenate([2.0 ** rng.uniform(-1021, 1021, 20000), rng.uniform(1, 2, 20000), -rng.uniform(1, 2, 2000),
                        2.0 ** np.arange(-1021, 1022), np.nextafter(2.0 ** np.arange(-1021, 1022), 0)])
    r = probe(0, d)
    # e^3 = 2^-66 of the series and half a unit in the last place
    bound = Fraction(101, 100) / 2 ** 53
    assert all(abs(Fraction(float(a)) * Fraction(float(b)) - 1) <= bound for a, b in zip(d, r))
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324])
    with np.errstate(divide="ignore", over="ignore"):
        np.testing.assert_array_equal(probe(0, special), 1.0 / special)


def test_square_root(probe):
    rng = np.random.default_rng(2)
    x = np.concatenate([2.0 ** rng.uniform(-110, 110, 1 << 21), rng.uniform(1, 4, 1 << 21),
                        np.arange(1, 1 << 12, dtype=np.float64) ** 2])
    got, want = probe(1, x), np.sqrt(x)  # (numpy's is correctly rounded)
    off = np.abs(got.view(np.int64) - want.view(np.int64))
    # off by a unit only within 2^-19 of one of a tie: two in 2^19 of all numbers
    assert off.max() <= 1 and (off > 0).mean() <= 2 * 2.0 ** -18
    assert np.array_equal(got[-4095:], want[-4095:])  # exact roots
    special = np.array([0.0, np.inf, np.nan, 5e-324, 1e-310, 1e300])
    np.testing.assert_array_equal(probe(1, special), np.sqrt(special))
