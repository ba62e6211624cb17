"""The pipelined pass's unequal warp shares (share_start, share_warp of
csrc/internal.h): every unit belongs to one warp and the warps' shares follow
the pattern, and the cost cut by units gives every warp a non-empty range whose
vectors it owns, at the workload's shapes."""
import numpy as np
import pytest

from test_index_math import _weighted

SLOW, FAST, WARPS = 12, 13, 14
FOUR = 2 * SLOW + 2 * FAST
CTA = 3 * FOUR + 2 * SLOW


def share_start(w):
    cta, i = divmod(w, WARPS)
    return cta * CTA + (i >> 2) * FOUR + (i & 3) * SLOW + (FAST - SLOW if (i & 3) == 3 else 0)


def share_warp(u):
    cta, o = divmod(u, CTA)
    four, x = divmod(o, FOUR)
    return cta * WARPS + 4 * four + (x >= SLOW) + (x >= 2 * SLOW) + (x >= 2 * SLOW + FAST)


def test_units():
    W = 152 * WARPS
    s = [share_start(w) for w in range(W + 1)]
    assert s[W] == 152 * CTA
    for w in range(W):
        assert s[w + 1] - s[w] == (FAST if (w % WARPS) & 3 >= 2 else SLOW)
        assert all(share_warp(u) == w for u in range(s[w], s[w + 1]))


@pytest.mark.parametrize("B,gamma,RV", [(16, 32, 18992), (24, 32, 18992), (8, 64, 12001), (64, 8, 9001)])
def test_ranges(B, gamma, RV):
    rows0, rows1 = B * gamma, B * (gamma + 1)
    U, W = 152 * CTA, 152 * WARPS
    R = 400 * 21 if 18 * RV + 400 * 21 >= 16 * (400 * 21 + 42) else 0
    T, start, owner, _, C = _weighted(rows0 * RV, rows1 * RV, U, 21, 18, RV, R)
    s = [start(share_start(w)) for w in range(W + 1)]
    assert C * U < 2 ** 53 and s[0] == 0 and s[W] == T
    assert all(s[w + 1] > s[w] for w in range(W))
    rng = np.random.default_rng(B)
    for v in set(rng.integers(0, T, 3000).tolist()) | set(s[:-1]) | {x - 1 for x in s[1:]}:
        w = share_warp(owner(int(v)))
        assert s[w] <= v < s[w + 1]
