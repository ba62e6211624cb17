"""The pipelined pass's unequal warp shares (share_start, share_warp, set_shares of
csrc/internal.h, compiled for the host): every unit belongs to one warp and the
warps' shares follow the pattern, and the cost cut by units gives every warp a
non-empty range whose vectors it owns, at the workload's shapes."""
import numpy as np
import pytest

import index_shim

SLOW, FAST, WARPS = 12, 13, 14
CTA = 3 * (2 * SLOW + 2 * FAST) + 2 * SLOW


def test_units():
    L, W = index_shim.lib(), 152 * WARPS
    s = [L.shim_share_start(w) for w in range(W + 1)]
    assert s[0] == 0 and s[W] == 152 * CTA
    for w in range(W):
        assert s[w + 1] - s[w] == (FAST if (w % WARPS) & 3 >= 2 else SLOW)
        assert all(L.shim_share_warp(u) == w for u in range(s[w], s[w + 1]))


@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("B,gamma,RV", [(16, 32, 18992), (24, 32, 18992), (8, 64, 12001), (64, 8, 9001)])
def test_ranges(kind, B, gamma, RV):
    s, row, vec, _, facts = index_shim.cut(kind, B, gamma, gamma + 1, RV)
    W, T = len(s) - 1, B * (2 * gamma + 1) * RV
    assert facts["whole"] == 0 and facts["units"] == (152 * CTA if kind == 1 else 0)
    assert facts["C"] * max(facts["units"], W) < 2 ** 53 and s[0] == 0 and s[W] == T
    assert np.all(s[1:] > s[:-1])
    assert np.array_equal(row * RV + vec, s) and np.all((vec >= 0) & (vec < RV))
    rng = np.random.default_rng(B)
    v = np.unique(np.concatenate([rng.integers(0, T, 3000), s[:-1], s[1:] - 1]))
    _, _, _, own, _ = index_shim.cut(kind, B, gamma, gamma + 1, RV, owners=v)
    assert np.all((s[own] <= v) & (v < s[own + 1]))
    if kind == 1:   # a warp's range costs its share
        cost = np.diff(s).reshape(-1, WARPS).sum(0).astype(float)
        fast = [w for w in range(WARPS) if w & 3 >= 2]
        slow = [w for w in range(WARPS) if w & 3 < 2]
        assert abs(cost[fast].mean() / cost[slow].mean() - FAST / SLOW) < 0.02
