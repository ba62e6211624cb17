"""The diagnostics at the edges of their kernels' tiles: logs around a warp, the
builder's and the prefix kernel's CTA, the parallel shuffle's limit, the largest
log and those whose builder needs about 48 KiB of shared memory, and the
metrics' tiles of sorted positives (1,024 of a cluster CTA's eighth of the
log), against the oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _log(B, gamma, seed):
    rng = np.random.default_rng(seed)
    z = rng.normal(size=(B, 1)) + 0.6 * rng.normal(size=(B, gamma)) + 1.5
    q = (np.round(64 / (1 + np.exp(-z))) / 64).astype(np.float32)      # 1/64 steps: ties
    L = (rng.random((B, gamma)) < q).cumprod(1).sum(1).astype(np.int32)
    return q, L


@pytest.mark.parametrize("B", [1, 2, 31, 32, 33, 255, 256, 257, 1025, 3376, 3377, 3413, 3449, 3450, 4095, 4096, 4097,
                               11323, 11324, 11450, 11564, 11565, 50000])
@pytest.mark.parametrize("signal", [0, 2])
def test_permutation_sizes(sdd, orc, B, signal):
    q, L = _log(B, 7, B)
    got = sdd.permutation_diagnostic(torch.from_numpy(q).cuda(), torch.from_numpy(L).cuda(), signal=signal,
                                     eta_b=0.70, eta_c=0.75, n_rep=3, seed=B)
    want = orc.permutation_diagnostic(q.astype(np.float64), L, signal, 0.70, 0.75, 3, B)
    np.testing.assert_array_equal(got.cpu().numpy(), want)


@pytest.mark.parametrize("B,gamma", [(1, 1), (7, 3), (33, 5), (2049, 4), (8193, 3), (9001, 2)])
@pytest.mark.parametrize("cond", [False, True])
def test_metrics_sizes(sdd, orc, B, gamma, cond):
    q, L = _log(B, gamma, B)
    got = sdd.position_metrics(torch.from_numpy(q).cuda(), torch.from_numpy(L).cuda(), conditional=cond)
    want = orc.position_metrics(q.astype(np.float64), L, cond)
    # fp64 sums of B terms in another order: below 2^-52 sqrt(B) of the sum of magnitudes, far inside 1e-12
    for g, w in zip(got[:3], want[:3]):
        np.testing.assert_allclose(g.cpu().numpy(), w, rtol=1e-12, atol=1e-15, equal_nan=True)
    for g, w in zip(got[3:], want[3:]):
        np.testing.assert_array_equal(g.cpu().numpy(), w)


@pytest.mark.parametrize("share", [0.02, 0.5, 0.98])
@pytest.mark.parametrize("B", [9, 257, 520, 2048, 8200, 16500])
def test_metrics_pairs(sdd, B, share):
    """The pair counts over any floats -- ties, signed zeros, infinities, NaN (in
    no pair) -- with few to nearly all blocks positive (the sorted tiles' powers
    of two), against counts by numpy's own sort."""
    rng = np.random.default_rng(B)
    q = rng.choice(np.array([0.0, -0.0, 0.25, 0.5, 0.5000001, 1.0, np.inf, -np.inf, np.nan], np.float32), size=(B, 2))
    q[:, 1] = np.where(rng.random(B) < 0.8, rng.random(B).astype(np.float32), q[:, 1])
    L = np.where(rng.random(B) < share, 2, 0).astype(np.int32)
    got = sdd.position_metrics(torch.from_numpy(q).cuda(), torch.from_numpy(L).cuda(), conditional=False)
    P, N = int((L > 0).sum()), int((L == 0).sum())
    for j in range(2):
        x = q[:, j]
        pos, neg = np.sort(x[(L > 0) & ~np.isnan(x)]), x[(L == 0) & ~np.isnan(x)]
        lt, le = np.searchsorted(pos, neg, "left"), np.searchsorted(pos, neg, "right")
        gt, eq = int((len(pos) - le).sum()), int((le - lt).sum())
        want = (gt + 0.5 * eq) / (float(P) * N) if P and N else float("nan")
        np.testing.assert_array_equal(got[2][j].item(), want)      # integers and one fp64 division
        assert got[3][j].item() == P and got[4][j].item() == N
