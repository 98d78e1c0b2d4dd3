"""A training step whose kernels report a failure (a bounded wait that ran out)
leaves the network as it was, and does not hide an earlier asynchronous
failure.  dm_mlp.cu is built against stand-ins for the kernels' launchers,
which set the error word or fill the partial gradients: nothing waits."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

FAKE = r"""
#include "dm_internal.h"
#include "dm_mlp.cuh"
namespace dm {
int fail_train = 0, fail_forward = 0;
void set_error(const std::string &) {}
MlpTrainShape mlp_train_shape(int M) { return {1, 1, 1}; }
cudaError_t launch_gemm_bf16(int, int, int, const void *, const void *, const float *, void *, int, int, int *,
                             cudaStream_t) { return cudaSuccess; }
cudaError_t launch_mlp_fused(int, const void *, const void *const *, const float *const *, float *, int *err,
                             cudaStream_t st) {
  return fail_forward ? cudaMemsetAsync(err, 1, sizeof(int), st) : cudaSuccess;
}
cudaError_t launch_mlp_train(int, const void *, const float *, int, const void *const *, const void *const *,
                             const float *const *, void *const *, void *const *, void *, double *, float *part,
                             float *gb4, int *err, cudaStream_t st) {
  // 0x3c3c3c3c is the float 0.0115; a failed launch leaves other numbers behind
  cudaMemsetAsync(part, fail_train ? 0x41 : 0x3c, mlp_part_offset(4, 1, 1) * sizeof(float), st);
  cudaMemsetAsync(gb4, fail_train ? 0x41 : 0x3c, 4 * 64 * sizeof(float), st);
  return fail_train ? cudaMemsetAsync(err, 1, sizeof(int), st) : cudaSuccess;
}
}  // namespace dm
extern "C" void fake_fail(int train, int forward) { dm::fail_train = train, dm::fail_forward = forward; }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2311_18126_gb300 import build as b
    d = tmp_path_factory.mktemp("mlp")
    (d / "fake.cu").write_text(FAKE)
    so = str(d / "libmlp.so")
    subprocess.run([b._nvcc(), *b.ARCH, "-O1", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", b.CSRC, "-o", so,
                    os.path.join(b.CSRC, "dm_mlp.cu"), str(d / "fake.cu"), "-lcudart"], check=True)
    L = ctypes.CDLL(so)
    L.dm_mlp_num_params.restype = ctypes.c_int64
    for f in ("dm_mlp_get_params", "dm_mlp_check", "dm_mlp_destroy"):
        getattr(L, f).argtypes = [ctypes.c_void_p] * (2 if "params" in f else 1)
    L.dm_mlp_create.argtypes = [ctypes.c_int32, ctypes.c_int32, ctypes.c_uint64, ctypes.c_void_p, ctypes.c_void_p]
    L.dm_mlp_forward_async.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int32]
    L.dm_mlp_train_step.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int32, ctypes.c_float, ctypes.c_void_p,
                                                             ctypes.c_void_p]
    return L


def _net(lib):
    m = ctypes.c_void_p()
    assert lib.dm_mlp_create(40, 4, 1, None, ctypes.byref(m)) == 0
    return m


def _params(lib, m):
    p = np.empty(lib.dm_mlp_num_params(), np.float32)
    assert lib.dm_mlp_get_params(m, p.ctypes.data) == 0
    return p


def test_failed_step_changes_nothing(lib):
    import torch
    X = torch.zeros((128, 64), dtype=torch.bfloat16, device="cuda")
    Y = torch.zeros((128, 64), dtype=torch.float32, device="cuda")
    step = lambda m: lib.dm_mlp_train_step(m, X.data_ptr(), Y.data_ptr(), 128, 1e-2, None, None)
    a, b = _net(lib), _net(lib)
    for m in (a, b):
        lib.fake_fail(0, 0)
        assert step(m) == 0
        before = _params(lib, m)
        if m is a:
            lib.fake_fail(1, 0)
            for _ in range(3):
                assert step(m) != 0
            assert np.array_equal(_params(lib, m), before)
            lib.fake_fail(0, 0)
        assert step(m) == 0  # Adam's moments and step count are those of the second step
    assert np.array_equal(_params(lib, a), _params(lib, b))
    assert not np.array_equal(_params(lib, a), before)
    for m in (a, b):
        lib.dm_mlp_destroy(m)


def test_earlier_asynchronous_failure_is_still_reported(lib):
    import torch
    X = torch.zeros((128, 64), dtype=torch.bfloat16, device="cuda")
    Y = torch.zeros((128, 64), dtype=torch.float32, device="cuda")
    m = _net(lib)
    lib.fake_fail(0, 1)
    assert lib.dm_mlp_forward_async(m, X.data_ptr(), Y.data_ptr(), 128) == 0
    lib.fake_fail(0, 0)
    assert lib.dm_mlp_train_step(m, X.data_ptr(), Y.data_ptr(), 128, 1e-2, None, None) == 0
    assert lib.dm_mlp_check(m) != 0
    assert lib.dm_mlp_check(m) == 0
    lib.dm_mlp_destroy(m)
