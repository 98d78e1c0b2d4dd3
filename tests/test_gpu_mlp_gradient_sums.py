"""Sums over the batch in the network's gradients: a network whose hidden
activations are all 1 and whose output weights are 1, so that every hidden
bias's and every weight's gradient of the last two layers is the plain sum of
the output gradients (bfloat16 numbers of one sign, known exactly)."""
import numpy as np
import pytest

from oracle import mlp as ref

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("draw", ["half normal", "lognormal"])
@pytest.mark.parametrize("M", [128, 512, 640, 3456, 16384, 131072, 524288])
def test_sums_of_one_sign(M, draw):
    import torch
    from paper_2311_18126_gb300 import MLP, ensure_built
    ensure_built()
    off = np.concatenate([[0], np.cumsum([fo * fi + fo for fi, fo in zip(ref.DIN, ref.DOUT)])])
    net = MLP(64, 1, seed=1)
    p = np.zeros(net.n_params, np.float32)
    for l in range(3):
        p[off[l + 1] - 256:off[l + 1]] = 1.0
    p[off[3]:off[3] + 256] = 1.0
    net.set_params(p)
    z = np.random.default_rng(M).standard_normal(M)
    y = (256.0 - (np.abs(z) if draw == "half normal" else np.exp(1.5 * z))).astype(np.float32)
    g = torch.empty(net.n_params, dtype=torch.float32, device="cuda")
    X = torch.zeros((M, 64), dtype=torch.bfloat16, device="cuda")
    net.train_step(X, torch.from_numpy(y[:, None].copy()).cuda(), 0.0, g)
    g = g.cpu().numpy().astype(np.float64)
    # the output is 256 exactly; its gradient as the kernel rounds it
    dy = (np.float32(2.0) * (np.float32(256.0) - y) / np.float32(M)).astype(np.float32)
    want = torch.from_numpy(dy).to(torch.bfloat16).double().sum().item()
    # a chain of 32 tensor-core accumulations (512 rows) may lose a unit in the
    # last place (2^-23) of its running sum, half the chain's on average, at
    # each; its chains per share (at least 12 of the batch) and the shares are
    # FP32 sums, rounded to nearest (2^-24)
    tol = 16 * 2.0 ** -23 + 0.5 * (M / 512 / 12 + 25) * 2.0 ** -24
    parts = {"hidden bias": g[off[3] - 256:off[3]], "hidden weights": g[off[2]:off[3] - 256],
             "output weights": g[off[3]:off[3] + 256]}
    for name, got in parts.items():
        err = np.abs(got / want - 1.0).max()
        assert err <= tol, (name, err, tol)
