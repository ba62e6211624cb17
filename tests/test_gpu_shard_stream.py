"""The sharded records (sdd_shard_partials) against fp64 on the slice, where the
streaming form can go wrong: rows that do and do not divide over the clusters,
rows crossing a cluster's middle, ragged slices, and the candidate lists under
ties (few levels, constant rows), masked rows, candidates bunched in one lane
or at the slice's ends, up to the largest k; both types, odd slice starts."""
import numpy as np
import pytest
import torch

import paper_2608_14787_gb300 as sdd
from paper_2608_14787_gb300 import vocab_shard

pytestmark = pytest.mark.gpu

REC = np.dtype([("m", "f4"), ("r", "f4"), ("t2", "f4"), ("sh", "f4"), ("sl", "f4"), ("amax", "i4"), ("g", "f4"),
                ("info", "i4"), ("cz", "f4", 16), ("cv", "i4", 16)])


def _logits(kind, B, P, V, dtype, gen):
    z = torch.randn(B, P, V, generator=gen, device="cuda") * 2
    if kind == "levels":
        z = (z * 2).round() / 2
    elif kind == "constant":
        z[:, ::2] = -1.5
    elif kind == "masked":
        keep = torch.rand(B, P, V, generator=gen, device="cuda") < 12 / V
        z = torch.where(keep, z, torch.full_like(z, -float("inf")))
        z[..., V // 2] = 0.25
    elif kind == "lane":
        at = torch.arange(3, V, 2048 if dtype == torch.bfloat16 else 1024, device="cuda")
        z[..., at] += 16
    elif kind == "ends":
        z[..., :9] += 16
        z[..., -9:] += 16
    return z.to(dtype)


@pytest.mark.parametrize("B,gamma,w,k", [(1, 32, 9000, 10), (16, 32, 8195, 16), (4, 9, 20001, 3), (7, 32, 4400, 1),
                                         (9, 17, 16384, 10), (2, 32, 30000, 0), (16, 32, 3000, 10),
                                         (5, 8, 9001, 5), (1, 1, 70000, 16)])
@pytest.mark.parametrize("kind", ["plain", "levels", "constant", "masked", "lane", "ends"])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_records(B, gamma, w, k, kind, dtype):
    if kind != "plain" and B * w > 40000:
        B = max(1, 76 // (2 * gamma + 1))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(B * 1000 + w + k)
    v0, V = 24, w + 100
    zd, zt = _logits(kind, B, gamma, w, dtype, gen), _logits(kind, B, gamma + 1, w, dtype, gen)
    x = torch.randint(0, V, (B, gamma), generator=gen, device="cuda", dtype=torch.int32)
    x[0, 0] = V
    r = vocab_shard.ShardRound(B, gamma, V, v0, v0 + w, dtype=dtype, ks=(k,) if k else ())
    sl = [vocab_shard.slice_logits(z, 0, w) for z in (zd, zt)]
    r.set_inputs(*sl, x)
    rec = np.frombuffer(r.partials().cpu().numpy().tobytes(), REC)
    assert int(r.status.item()) & ~sdd.DEV_BAD_TOKEN == 0
    z = torch.cat([zd.reshape(-1, w), zt.reshape(-1, w)]).double().cpu().numpy()
    z = np.maximum(z, -(2.0 ** 23))
    nd = B * gamma
    m = z.max(1)
    np.testing.assert_array_equal(rec["m"], m)
    np.testing.assert_array_equal(rec["amax"], v0 + z.argmax(1))
    ref = rec["r"].astype(np.float64)[:, None]
    e = np.exp2(z * np.log2(np.e) - ref)
    np.testing.assert_allclose(rec["sh"].astype(np.float64) + rec["sl"], e.sum(1), rtol=1e-6)   # ex2: 2^-22
    t2 = (e * (z - m[:, None]) * np.log2(np.e))[:nd].sum(1)
    scale = (e * np.abs(z - m[:, None]))[:nd].sum(1) + 1e-30
    assert np.all(np.abs(rec["t2"][:nd] - t2) <= 1e-5 * scale)                                   # fp32 sums
    xs = x.cpu().numpy()
    tok = np.concatenate([xs.reshape(-1), np.concatenate([xs, np.full((B, 1), -7, np.int32)], 1).reshape(-1)])
    has = tok != -7
    out = has & ((tok < 0) | (tok >= V))
    inside = has & ~out & (tok >= v0) & (tok < v0 + w)
    np.testing.assert_array_equal((rec["info"] & 1) != 0, inside)
    np.testing.assert_array_equal((rec["info"] & 2) != 0, out)
    rows = np.nonzero(inside)[0]
    np.testing.assert_array_equal(rec["g"][rows], z[rows, tok[rows] - v0].astype(np.float32))
    nc = (rec["info"] >> 8) & 0xFF
    assert np.all(nc[:nd] == 0) and np.all(nc[nd:] == min(k, w))
    if k:
        order = np.argsort(-z[nd:], axis=1, kind="stable")[:, :k]
        np.testing.assert_array_equal(rec["cv"][nd:, :k], v0 + order)
        np.testing.assert_array_equal(rec["cz"][nd:, :k], np.take_along_axis(z[nd:], order, 1).astype(np.float32))
