"""The pipelined call at the sizes where its form changes (a decide team of 128
threads up to 200 MiB of logits and from 480 MiB to 1 GiB, of 64 between, two
kernels above, and above 480 MiB where the draws would outlast the pass): chains whose rounds lie on both sides of each line, each
round's outputs against the same round unpipelined (decisions equal; statistics
within the rounding that another cut of the rows can make)."""
import pytest
import torch

import paper_2608_14787_gb300 as sdd
from paper_2608_14787_gb300 import synth

pytestmark = pytest.mark.gpu
WHOLE = ("argmax", "K", "D_out", "L_strict", "tokens_strict", "n_strict", "commit_tokens", "commit_n", "L_topk", "tokens_topk")


@pytest.mark.parametrize("sizes", [(10, 11, 10), (25, 26, 25), (54, 55, 3, 54)])
def test_sizes(sizes):
    gamma, V = 32, 151936       # 19.75 MB a block: 200 MiB lie between 10 and 11, 480 MiB between 25 and 26, 1 GiB at 54
    pairs = []
    for i, B in enumerate(sizes):
        blk = synth.make_block("c3", device="cuda", B=B, round_=20 + i)
        two = []
        for _ in range(2):
            r = sdd.BlockRound(B, gamma, V, ks=(2,))
            r.set_inputs(blk.z_d, blk.z_t, blk.x, seed=i, round_=i)
            two.append(r)
        pairs.append((two, blk))
    prev = None
    for two, _ in pairs:
        sdd.block_pipelined(two[0], prev)
        prev = two[0]
    sdd.block_pipelined(None, prev)
    for (a, b), _ in pairs:
        b.run()
        for n in WHOLE:
            assert torch.equal(getattr(a, n), getattr(b, n)), n
        for n in ("q", "maxprob", "entropy"):
            torch.testing.assert_close(getattr(a, n), getattr(b, n), rtol=2e-6, atol=1e-7)
        assert int(a.status.item()) == 0


@pytest.mark.parametrize("B,gamma", [(128, 4), (64, 8)])
def test_many_blocks_of_few_positions(B, gamma):
    """Rounds whose draws would outlast the streaming pass beside them (whole and half fp32 draw rows to a team: 3.4 and
    1.3 times the two kernels' time) take at most a fifth longer than the two kernels, and decide the same; a small
    round follows."""
    V = 151936
    blks = [synth.make_block("c3", device="cuda", B=b, gamma=gamma, dtype=torch.float32, round_=i)
            for i, b in enumerate((B, B, 3))]
    rnds = []
    for i, blk in enumerate(blks):
        r = sdd.BlockRound(blk.x.shape[0], gamma, V, dtype=torch.float32, ks=(2,))
        r.set_inputs(blk.z_d, blk.z_t, blk.x, seed=i, round_=i)
        rnds.append(r)
    prev = None
    for r in rnds:
        sdd.block_pipelined(r, prev)
        prev = r
    sdd.block_pipelined(None, prev)
    got = [{n: getattr(r, n).clone() for n in WHOLE} for r in rnds]
    for r, g in zip(rnds, got):
        r.run()
        assert all(torch.equal(getattr(r, n), g[n]) for n in WHOLE) and int(r.status.item()) == 0
    state = [0]

    def piped():
        state[0] ^= 1
        sdd.block_pipelined(rnds[state[0]], rnds[1 - state[0]])

    def us(fn, n=10):
        ts = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda._sleep(1000000)
            a.record()
            for _ in range(n):
                fn()
            b.record()
            torch.cuda.synchronize()
            ts.append(a.elapsed_time(b) * 1e3 / n)
        return min(ts)
    sdd.block_pipelined(rnds[0], None)
    two = us(lambda: rnds[0].run())
    rnds[0].run()
    sdd.block_pipelined(rnds[0], None)
    assert us(piped) <= 1.2 * two
