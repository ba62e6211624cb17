"""Streaming warps whose ranges touch more than 32 rows (their rows' facts are
held one row per lane and reloaded): short rows in large batches, the ranges
starting and ending inside rows, tokens out of range and masked rows among
them, against the oracle (the tolerance as in the extended features' tests)."""
import numpy as np
import pytest
import torch

from paper_2608_14787_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,gamma,V", [(700, 64, 8), (1400, 33, 24), (620, 64, 5)])
def test_many_rows_per_warp(sdd, orc, B, gamma, V):
    g = torch.Generator(device="cuda")
    g.manual_seed(B)
    stride = -(-V // 8) * 8
    mk = lambda n: torch.randn(B, n, stride, generator=g, device="cuda").to(torch.bfloat16)[..., :V]   # noqa: E731
    z_d, z_t = mk(gamma), mk(gamma + 1)
    z_d[3, 1] = -float("inf")
    x = torch.randint(0, V, (B, gamma), generator=g, device="cuda", dtype=torch.int32)
    x[5, 2], x[6, 0] = V, -1
    rnd = sdd.BlockRound(B, gamma, V, ks=(2,), K_min=0, greedy=True)
    rnd.set_inputs(z_d, z_t, x)
    rnd.run()
    st = orc.row_stats(synth.bf16_bits(z_d), tokens=x.cpu().numpy())
    ok = np.ones((B, gamma), bool)
    ok[3, 1] = ok[5, 2] = ok[6, 0] = False
    np.testing.assert_allclose(rnd.q.cpu().numpy()[ok], st.q[ok], rtol=4e-6)
    assert np.isnan(rnd.q.cpu().numpy()[~ok]).all()
    np.testing.assert_array_equal(rnd.argmax.cpu().numpy()[ok], st.argmax[ok])
    zt, xs = synth.bf16_bits(z_t), x.cpu().numpy()
    for b in list(range(0, B, 37)) + [4, 7, B - 1]:
        if b in (3, 5, 6):
            continue
        facts = orc.target_facts(zt[b], xs[b])
        L, tok, _ = orc.verify_topk(facts, xs[b], 2)
        assert int(rnd.L_topk[0, b]) == L and np.array_equal(rnd.tokens_topk[0, b].cpu().numpy(), tok)
    assert int(rnd.status.item()) == sdd.DEV_NONFINITE | sdd.DEV_BAD_TOKEN
