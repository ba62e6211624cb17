"""The cut of a call's rows into whole pieces (scan_warps of csrc/internal.h):
with as many warps as rows times k and equal costs, every warp's range is a
non-empty piece of one row, the pieces of a row belong to k consecutive warps,
and the owner of every vector agrees with the ranges."""
import pytest

from test_index_math import _weighted


def _whole_pieces(W_max, T, rows, least=8, most=16):
    k = min(W_max // rows, most)
    return k if k >= least and 2 * rows * k <= T else 0


@pytest.mark.parametrize("rows0,rows1,RV", [(8, 9, 8000), (32, 33, 18992), (1, 2, 16), (1, 2, 40), (152, 152, 313),
                                            (150, 153, 17), (100, 0, 251), (0, 66, 999)])
def test_whole_pieces(rows0, rows1, RV):
    rows = rows0 + rows1
    T = rows * RV
    k = _whole_pieces(152 * 16, T, rows)
    if k == 0:
        pytest.skip("outside the rule")
    assert 8 <= k <= 16
    W = rows * k
    T, start, owner, _, C = _weighted(rows0 * RV, rows1 * RV, W, 1, 1, RV, 0)
    s = [start(w) for w in range(W + 1)]
    assert s[0] == 0 and s[W] == T
    for w in range(W):
        assert s[w] < s[w + 1]
        r = w // k
        assert r * RV <= s[w] and s[w + 1] <= (r + 1) * RV
    for r in range(rows):
        assert owner(r * RV) == r * k and owner((r + 1) * RV - 1) == (r + 1) * k - 1


def test_rule_edges():
    # 304 rows are the last with eight pieces on 152 SMs; short rows keep two vectors a piece
    assert _whole_pieces(2432, 304 * 1000, 304) == 8 and _whole_pieces(2432, 305 * 1000, 305) == 0
    assert _whole_pieces(2432, 17 * 31, 17) == 0 and _whole_pieces(2432, 17 * 32, 17) == 16
