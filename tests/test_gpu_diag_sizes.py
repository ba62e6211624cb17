"""The diagnostics at the edges of their kernels' tiles: logs around a warp, the
builder's and the prefix kernel's CTA, the parallel shuffle's limit, and the
metrics' tiles of positives (1,024 of a cluster CTA's eighth of the log) and
negatives (4,096), against the oracle."""
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


@pytest.mark.parametrize("B", [1, 2, 31, 32, 33, 255, 256, 257, 1025, 4095, 4096, 4097])
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
