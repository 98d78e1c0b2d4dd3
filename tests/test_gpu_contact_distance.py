"""The contact pairs' distance with its first and second derivatives in closed
form (dm_contact.cu) against the oracle's rule differentiated by autograd:
crossing, clamped and nearly parallel segments."""
import ctypes
import subprocess

import numpy as np
import pytest
import torch

from oracle.contact import segment_distance

pytestmark = pytest.mark.gpu

PROBE = r"""
#include "dm_contact.cu"
namespace dm { void set_error(const std::string &) {} }
// per pair: D, its 12 first and 78 second derivatives (packed upper triangle)
__global__ void k_probe(const double *x, double *y) {
  dm::HLane ln;
  ln.load(threadIdx.x);
  const dm::Distance q = dm::pair_distance(x + 12 * blockIdx.x, ln);
  double *o = y + 91 * blockIdx.x;
  if (threadIdx.x == 0) o[0] = q.D;
  if (threadIdx.x < 12) o[1 + threadIdx.x] = q.Dx;
  for (int k = 0; k < dm::kHP; ++k)
    if (ln.on[k]) o[13 + threadIdx.x + 32 * k] = q.h[k];
}
extern "C" int probe(int n, const double *x, double *y) {
  double *d = nullptr;
  if (cudaMalloc(&d, 103 * sizeof(double) * n) != cudaSuccess) return 1;
  cudaMemcpy(d, x, 12 * sizeof(double) * n, cudaMemcpyHostToDevice);
  k_probe<<<n, 32>>>(d, d + 12 * n);
  const cudaError_t e = cudaMemcpy(y, d + 12 * n, 91 * sizeof(double) * n, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)e;
}
"""


def _pairs(kind, rng, n=24):
    """Edge b from a point beside edge a (of length 1 along a random direction)."""
    out = []
    for _ in range(n):
        u, v = rng.standard_normal((2, 3))
        u /= np.linalg.norm(u)
        v -= (v @ u) * u
        v /= np.linalg.norm(v)
        w = np.cross(u, v)
        # the angle to edge a: |a x b|^2 < 1e-12 |a|^2 |b|^2 counts as parallel.
        # Nearly parallel edges lie in one plane, so that the closest point of
        # edge a is a distance of 1e-7 off its first node on one side or the other
        # (exactly parallel ones are on the rule's kink there)
        angle = rng.uniform(0.4, 1.5) if kind == "crossing" else rng.choice([-1.0, 1.0]) * rng.uniform(3e-7, 9e-7)
        b = rng.uniform(0.5, 2.0) * (np.cos(angle) * u + np.sin(angle) * v) * rng.choice([-1.0, 1.0])
        p = rng.standard_normal(3)
        at = rng.uniform(-0.6, 1.6)  # beyond the ends: clamped
        q = p + at * u + rng.uniform(0.2, 0.9) * (w if kind == "crossing" else v) - rng.uniform(0.1, 0.9) * b
        out.append(np.concatenate([p, p + u, q, q + b]))
    return np.array(out)


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_2311_18126_gb300 import build as b
    d = tmp_path_factory.mktemp("distance")
    (d / "probe.cu").write_text(PROBE)
    so = str(d / "libprobe.so")
    subprocess.run([b._nvcc(), *b.ARCH, *b.NVCC_FLAGS, "-shared", "-I", b.CSRC, "-o", so, str(d / "probe.cu"),
                    "-lcudart"], check=True)
    return ctypes.CDLL(so).probe


@pytest.mark.parametrize("kind", ["crossing", "nearly parallel"])
def test_distance_derivatives(probe, kind):
    x = np.ascontiguousarray(_pairs(kind, np.random.default_rng(7)))
    y = np.empty((len(x), 91))
    P = ctypes.POINTER(ctypes.c_double)
    assert probe(len(x), x.ctypes.data_as(P), y.ctypes.data_as(P)) == 0
    iu = np.triu_indices(12)
    distance = lambda z: segment_distance(z[0:3], z[3:6], z[6:9], z[9:12])[0]
    for xi, yi in zip(x, y):
        z = torch.tensor(xi, requires_grad=True)
        D = distance(z)
        g = torch.autograd.grad(D, z)[0].numpy()
        H = torch.autograd.functional.hessian(distance, torch.tensor(xi)).numpy()
        # some hundred roundings of terms of this size (lengths are of order one)
        assert abs(yi[0] - D.item()) <= 1e-14 * D.item()
        assert np.abs(yi[1:13] - g).max() <= 1e-12
        assert np.abs(yi[13:] - H[iu]).max() <= 1e-11 * np.abs(H).max()
