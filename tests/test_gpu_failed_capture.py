"""A Newton round whose capture is invalidated returns an error, and the process
goes on: a copy of the library whose end of capture first does what a failed
launch does to it (here a synchronisation of the capturing stream, which CUDA
refuses), run in a process of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

PROBE = r"""
#include <cuda_runtime.h>
#include <cstdlib>
static cudaError_t probe_end(cudaStream_t st, cudaGraph_t *g) {
  if (getenv("SPOIL_CAPTURE")) (void)cudaStreamSynchronize(st);
  return cudaStreamEndCapture(st, g);
}
#define cudaStreamEndCapture probe_end
#include "dm_api.cu"
"""

RUN = r"""
import os, sys
sys.path[:0] = [%(root)r, %(tests)r]
import numpy as np
import workloads
from paper_2311_18126_gb300 import dismech
dismech.load_library(%(so)r)
for desc, params in (workloads.cantilever(N=12), workloads.coil(N=60, pitch_factor=2.05)[:2]):
    s = dismech.System(desc, params)
    q0 = s.get_state()[0].copy()
    os.environ["SPOIL_CAPTURE"] = "1"
    for _ in range(2):
        try:
            s.step(1)
        except dismech.DismechError:
            continue
        sys.exit("the step did not fail")
    assert np.array_equal(s.get_state()[0], q0)
    del os.environ["SPOIL_CAPTURE"]
    s.step(1)  # captured anew
    t = dismech.System(desc, params)
    t.step(1)
    assert np.abs(s.get_state()[0] - t.get_state()[0]).max() < 1e-12
    s.close()
    t.close()
print("done")
"""


def test_step_returns_an_error(tmp_path):
    from paper_2311_18126_gb300 import build as b
    b.build()
    (tmp_path / "probe.cu").write_text(PROBE)
    so, obj = str(tmp_path / "libprobe.so"), str(tmp_path / "probe.o")
    subprocess.run([b._nvcc(), *b.ARCH, *b.NVCC_FLAGS, "-I", b.CSRC, "-c", "-o", obj, str(tmp_path / "probe.cu")],
                   check=True)
    rest = [os.path.join(b.BUILD, os.path.basename(s) + ".o") for s in b.sources()
            if os.path.basename(s) != "dm_api.cu"]
    subprocess.run([b._nvcc(), *b.ARCH, "-shared", "-o", so, obj, *rest, "-lcudart"], check=True)
    tests = os.path.dirname(os.path.abspath(__file__))
    r = subprocess.run([sys.executable, "-c", RUN % dict(root=os.path.dirname(tests), tests=tests, so=so)],
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "done" in r.stdout, (r.returncode, r.stdout, r.stderr[-2000:])
