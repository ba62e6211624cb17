"""The extended features where a piece's group lists can go wrong: pieces of
one tile and of many, fewer than five groups or entries, the five largest in
one lane-tile, in one lane over many tiles, and tied over all tiles, negative
and masked rows, both types, against the oracle.  The oracle reads the same
logits, so both types have the fp32 tolerance: a sum's terms are within 2^-22 (ex2
and its argument) and added as fp32 pairs, q and the probabilities end in an expf
of two units: 6e-7 in all, 4e-6 allowed."""
import numpy as np
import pytest
import torch

from paper_2608_14787_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,gamma,V", [(1, 1, 3), (1, 4, 40), (2, 5, 2047), (3, 9, 20483), (1, 3, 262144), (40, 9, 9001)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_features(sdd, orc, B, gamma, V, dtype):
    q = 8 if dtype == torch.bfloat16 else 4
    g = torch.Generator(device="cuda")
    g.manual_seed(V)
    z = torch.zeros(B, gamma, -(-V // q) * q, dtype=dtype, device="cuda")[..., :V]
    z.copy_(torch.randn(B, gamma, V, generator=g, device="cuda") * 2 - 9)
    flat = [(b, j) for b in range(B) for j in range(gamma)]
    tile = 256 * q
    for i, (b, j) in enumerate(flat):
        kind = i % 6
        r = z[b, j]
        if kind == 0:                               # all in one vector
            r[: min(V, q)] = torch.linspace(3, 4, q, device="cuda")[: min(V, q)].to(dtype)
        elif kind == 1:                             # one lane, one entry per tile
            at = torch.arange(0, V, tile, device="cuda") + min(5, V - 1)
            at = at[at < V]
            r[at] = (2 + torch.arange(len(at), device="cuda") * 0.0625).to(dtype)
        elif kind == 2:                             # tied everywhere
            r[:] = -3.0
        elif kind == 3:                             # four finite entries
            keep = r[: min(V, 4)].clone()
            r[:] = -float("inf")
            r[V - len(keep):] = keep
        elif kind == 4:                             # the row's end
            r[V - min(V, 5):] = torch.linspace(1, 2, 5, device="cuda")[: min(V, 5)].to(dtype)
    x = torch.randint(0, V, (B, gamma), generator=g, device="cuda", dtype=torch.int32)
    conf = sdd.confidence(z, x, features=True)
    margin, top5 = orc.row_features(synth.bf16_bits(z))
    rtol = 4e-6
    np.testing.assert_allclose(conf.top5.cpu().numpy(), top5, rtol=rtol)
    p1 = conf.maxprob.cpu().numpy()
    assert np.all(np.abs(conf.margin.cpu().numpy() - margin) <= rtol * p1)
