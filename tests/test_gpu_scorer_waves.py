"""The scorers where their launch changes shape: batches just inside and past
one CTA per SM (36 tiles of 128 rows as clusters of four on 152 SMs, 76 as
clusters of two) and of several waves with a ragged last tile, and K whose slices of 64 do not divide by four (and under
four of them), against fp64.  One layer: fp32 sums of K products in four
chains are off by 2e-7 at the most (K = 3,520); 1e-6 allowed.  Deep: as derived
in the scorer's own test (bf16 activations)."""
import pytest
import torch

from paper_2608_14787_gb300 import synth

pytestmark = pytest.mark.gpu


def _gelu(z):
    return 0.5 * z * (1 + torch.erf(z / 2 ** 0.5))


@pytest.mark.parametrize("M,K", [(36 * 128, 512), (36 * 128 + 1, 512), (38 * 128, 512), (38 * 128 + 1, 512), (76 * 128 - 5, 448), (20001, 320), (700, 192),
                                 (20001, 64), (300, 3520)])
def test_mlp(sdd, M, K):
    W1, b1, w2, b2 = synth.make_mlp(device="cuda", hidden=K)
    h = synth.make_hidden(M, device="cuda", seed=3, hidden=K)
    status = sdd.new_status()
    s = sdd.survival_mlp(h, W1, b1, w2, float(b2), status=status)
    again = sdd.survival_mlp(h, W1, b1, w2, float(b2), status=status)
    want = torch.sigmoid(_gelu(h.double() @ W1.double().T + b1.double()) @ w2.double() + b2.double())
    assert int(status.item()) == 0 and torch.equal(s, again)
    torch.testing.assert_close(s.double(), want, rtol=0, atol=1e-6)


@pytest.mark.parametrize("K", [512, 2048, 3584])
@pytest.mark.parametrize("M", [64 * 128, 12000, 152 * 128, 20001])
def test_mlp_error_does_not_grow_with_the_batch(sdd, M, K):
    """However a batch's tiles are run, a tile's K is summed in chains as short as a small batch's (four).  One CTA a
    tile (and the tiles left over) add the same sums in the same order as 2,048 rows at a time do; two CTAs a tile add
    them pairwise, so there the errors against fp64 are compared, which differ by their last rounding (a single chain's
    is four times as large at K = 3,584).  Under eight slices of K: test_mlp_short_k."""
    W1, b1, w2, b2 = synth.make_mlp(device="cuda", hidden=K)
    h = synth.make_hidden(M, device="cuda", seed=3, hidden=K)
    s = sdd.survival_mlp(h, W1, b1, w2, float(b2))
    small = torch.cat([sdd.survival_mlp(c, W1, b1, w2, float(b2)) for c in h.split(2048)])
    if M > 76 * 128:
        assert torch.equal(s, small)
    else:
        want = torch.sigmoid(_gelu(h.double() @ W1.double().T + b1.double()) @ w2.double() + b2.double())
        assert float((s - want).norm()) <= 1.1 * float((small - want).norm())


@pytest.mark.parametrize("K,bound", [(192, 5.5e-8), (256, 5.1e-8), (320, 6.3e-8), (384, 6.0e-8), (448, 6.8e-8)])
def test_mlp_short_k(sdd, K, bound):
    """Three to seven slices in one or two chains: the error against fp64 (2-norm) that a CTA with the whole of K, or two
    splits of it, always had (5.1e-8 at 192, 4.8e-8 at 256, 6.4e-8 at 448), and a twentieth."""
    W1, b1, w2, b2 = synth.make_mlp(device="cuda", hidden=K)
    h = synth.make_hidden(152 * 128, device="cuda", seed=3, hidden=K)
    want = torch.sigmoid(_gelu(h.double() @ W1.double().T + b1.double()) @ w2.double() + b2.double())
    s = sdd.survival_mlp(h, W1, b1, w2, float(b2))
    assert float((s - want).norm() / want.norm()) <= bound


@pytest.mark.parametrize("M,Kh", [(36 * 128, 256), (37 * 128, 256), (38 * 128, 256), (38 * 128 + 1, 256), (12345, 192), (20001, 64), (20001, 704)])
def test_deep(sdd, M, Kh):
    w = synth.make_scorer_deep(device="cuda", hidden=Kh)
    W1, b1, W2, b2, W3, b3, w4, b4 = w
    h = synth.make_hidden(M, device="cuda", seed=5, hidden=Kh)
    f = synth.make_features(M, device="cuda")
    status = sdd.new_status()
    s = sdd.scorer_deep(h, f, *w, status=status)
    again = sdd.scorer_deep(h, f, *w, status=status)
    u = torch.cat([h, f], 1).double()
    for W, b in ((W1, b1), (W2, b2), (W3, b3)):
        u = _gelu(u @ W.double().T + b.double())
    want = torch.sigmoid(u @ w4.double() + b4)
    assert int(status.item()) == 0 and torch.equal(s, again)
    torch.testing.assert_close(s.double(), want, rtol=0, atol=3e-4)


@pytest.mark.parametrize("Kh", [256, 704, 3584])
@pytest.mark.parametrize("M", [64 * 128, 12000, 152 * 128, 20001])
def test_deep_rows_do_not_depend_on_the_batch(sdd, M, Kh):
    """One CTA a tile and the split form sum alike: activations of the first layer and scores of a batch are those of
    its rows 2,048 at a time, except between 36 and 76 tiles, where two splits add the chains pairwise."""
    w = synth.make_scorer_deep(device="cuda", hidden=Kh)
    h, f = synth.make_hidden(M, device="cuda", seed=5, hidden=Kh), synth.make_features(M, device="cuda")
    act = [torch.empty(n, 256, dtype=torch.bfloat16, device="cuda") for n in (M, M)]
    s = sdd.scorer_deep(h, f, *w, act=act[0])
    small = torch.cat([sdd.scorer_deep(h[i:i + 2048], f[i:i + 2048], *w, act=act[1][i:i + 2048])
                       for i in range(0, M, 2048)])
    if M > 76 * 128:
        assert torch.equal(act[0], act[1]) and torch.equal(s, small)
    else:
        assert float((act[0] != act[1]).float().mean()) < 1e-3
        torch.testing.assert_close(s, small, rtol=0, atol=1e-4)   # a bf16 step of a few activations


@pytest.mark.parametrize("M", [38 * 128 + 1, 152 * 128 + 1, 157 * 128])
def test_hidden_states_written_just_before(sdd, M):
    """Every launch of a call (whole waves of tiles, then the tiles left over) sees what the stream wrote just ahead."""
    K = 256
    W1, b1, w2, b2 = synth.make_mlp(device="cuda", hidden=K)
    w = synth.make_scorer_deep(device="cuda", hidden=K)
    f = synth.make_features(M, device="cuda")
    src = [synth.make_hidden(M, device="cuda", seed=s, hidden=K) for s in (3, 4)]
    want = [(sdd.survival_mlp(h, W1, b1, w2, float(b2)), sdd.scorer_deep(h, f, *w)) for h in src]
    h = torch.zeros_like(src[0])
    torch.cuda.synchronize()
    got = []
    for i in (0, 1, 0):
        h.copy_(src[i])
        s = sdd.survival_mlp(h, W1, b1, w2, float(b2))
        h.copy_(src[1 - i])
        got.append((s, i, 0))
        got.append((sdd.scorer_deep(h, f, *w), 1 - i, 1))
    for s, i, k in got:
        assert torch.equal(s, want[i][k])


@pytest.mark.parametrize("M", [128, 38 * 128 + 1, 152 * 128 + 1])
def test_weights_written_just_before(sdd, M):
    """Every layer's launch sees weights and biases that the stream wrote just ahead of the call."""
    K = 256
    h, f = synth.make_hidden(M, device="cuda", seed=3, hidden=K), synth.make_features(M, device="cuda")
    src = [synth.make_scorer_deep(device="cuda", hidden=K, seed=s) for s in (1, 2)]
    want = [sdd.scorer_deep(h, f, *w) for w in src]
    w = [t.clone() if torch.is_tensor(t) else t for t in src[0]]
    torch.cuda.synchronize()
    got = []
    for i in (1, 0, 1):
        for dst, new in zip(w, src[i]):
            if torch.is_tensor(dst):
                dst.copy_(new)
        w[-1] = src[i][-1]
        got.append((sdd.scorer_deep(h, f, *w), i))
    for s, i in got:
        assert torch.equal(s, want[i])


def _us(fn, n=20):
    for _ in range(3):
        fn()
    ts = []
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda._sleep(1000000)
        a.record()
        for _ in range(n):
            fn()
        b.record()
        torch.cuda.synchronize()
        ts.append(a.elapsed_time(b) * 1e3 / n)
    return min(ts)


@pytest.mark.parametrize("K", [256, 448])
def test_split_tiles_fit_one_wave(sdd, K):
    """38 tiles of a short K (clusters of four that do not all fit at once took 1.6 times as long as 39 tiles, which run
    as clusters of two)."""
    W1, b1, w2, b2 = synth.make_mlp(device="cuda", hidden=K)
    b2, us = float(b2), []
    for tiles in (38, 39):
        h = synth.make_hidden(tiles * 128, device="cuda", hidden=K)
        ws, out = sdd.scorer_workspace(tiles * 128, "cuda"), torch.empty(tiles * 128, device="cuda")
        us.append(_us(lambda: sdd.survival_mlp(h, W1, b1, w2, b2, workspace=ws, out=out)))
    assert us[0] <= 1.2 * us[1], us
