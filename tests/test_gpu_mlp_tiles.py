"""The inference kernel's two tiles in flight: batches of one tile, of fewer and
more tiles than multiprocessors, with odd and even counts per CTA.  A row's
result does not depend on its tile's place, so a batch is compared bit for bit
with its tiles computed one at a time; and the weight blocks' order with the
reference."""
import numpy as np
import pytest

from oracle import mlp as ref

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tiles", [1, 2, 3, 151, 153, 304, 305, 457])
def test_batches_match_single_tiles(tiles):
    import torch
    from paper_2311_18126_gb300 import MLP, ensure_built
    ensure_built()
    net = MLP(40, 4, seed=3)
    gen = torch.Generator().manual_seed(tiles)
    base = torch.randn((128 * min(tiles, 5), 64), generator=gen).to(torch.bfloat16).cuda()
    base[:, 40:] = 0
    reps = -(-tiles // 5) if tiles > 5 else 1
    X = base.repeat(reps, 1)[:128 * tiles].contiguous()
    out = torch.full((128 * tiles, 64), float("nan"), dtype=torch.float32, device="cuda")
    net.forward(X, out)
    one = torch.empty((128, 64), dtype=torch.float32, device="cuda")
    single = []
    for k in range(base.shape[0] // 128):
        net.forward(base[128 * k:128 * (k + 1)].contiguous(), one)
        single.append(one.clone())
    want = torch.cat(single).repeat(reps, 1)[:128 * tiles]
    assert torch.equal(out, want)
    r = ref.forward(net.get_params().astype(np.float64), base.float().cpu().numpy().astype(np.float64),
                    rounding=True)[-1]
    # an operand may round to the neighbouring bfloat16 (2^-8), layer by layer
    np.testing.assert_allclose(torch.cat(single).cpu().numpy(), r, rtol=2 ** -7, atol=2 ** -7 * np.abs(r).max())


def test_special_values_stay_in_their_rows():
    """A NaN or infinite input spoils its own row only; ReLU maps NaN to 0 (the
    larger of a number and NaN is the number)."""
    import torch
    from paper_2311_18126_gb300 import MLP, ensure_built
    ensure_built()
    net = MLP(40, 4, seed=4)
    X = torch.randn((384, 64), generator=torch.Generator().manual_seed(1)).to(torch.bfloat16).cuda()
    X[:, 40:] = 0
    out, bad = (torch.empty((384, 64), dtype=torch.float32, device="cuda") for _ in range(2))
    net.forward(X, out)
    Y = X.clone()
    Y[5, 3], Y[200, 0] = float("nan"), float("inf")
    net.forward(Y, bad)
    same = torch.ones(384, dtype=torch.bool, device="cuda")
    same[5] = same[200] = False
    assert torch.equal(out[same], bad[same])
    assert torch.isfinite(bad[5]).all()  # every first-layer sum is NaN, its ReLU 0
