"""The cut of a call's rows into whole pieces (whole_pieces, scan_warps,
part_start, part_owner of csrc/internal.h, compiled for the host): with as many
warps as rows times k and equal costs, every warp's range is a non-empty piece
of one row, the pieces of a row belong to k consecutive warps, and the owner of
every vector agrees with the ranges."""
import numpy as np
import pytest

import index_shim


@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("nb,npos0,npos1,RV", [(1, 8, 9, 8000), (1, 32, 33, 18992), (1, 1, 2, 16), (1, 1, 2, 40),
                                               (152, 1, 1, 313), (50, 3, 3, 17), (100, 1, 0, 251), (3, 11, 11, 999)])
def test_whole_pieces(kind, nb, npos0, npos1, RV):
    rows = nb * (npos0 + npos1)
    warps = 152 * (16, 14, 12)[kind]
    rule = index_shim.lib().shim_whole_pieces(warps, rows * RV, rows, 8 if kind else 16)
    s, row, vec, _, facts = index_shim.cut(kind, nb, npos0, npos1, RV)
    k = facts["whole"]
    assert k == rule or (rule == 0 and 2 * k == RV)   # (rows of 16 to 31 vectors, two to a warp, come out whole too)
    if k == 0:
        assert kind > 0 and warps // rows < 8   # (every listed shape is whole on sixteen warps a CTA)
        return
    assert 8 <= k <= 16 and len(s) - 1 == rows * k and s[0] == 0 and s[-1] == rows * RV
    assert np.all(s[1:] > s[:-1])
    w = np.arange(rows * k)
    assert np.array_equal(row[:-1], w // k) and np.all(s[1:] <= (w // k + 1) * RV)
    assert np.array_equal(row * RV + vec, s)
    v = np.arange(rows * RV) if rows * RV < 200000 else np.unique(np.concatenate([s[:-1], s[1:] - 1]))
    _, _, _, own, _ = index_shim.cut(kind, nb, npos0, npos1, RV, owners=v)
    assert np.all((s[own] <= v) & (v < s[own + 1]))


def test_rule_edges():
    # 304 rows are the last with eight pieces on 152 SMs; short rows keep two vectors a piece
    f = index_shim.lib().shim_whole_pieces
    assert f(2432, 304 * 1000, 304, 16) == 8 and f(2432, 305 * 1000, 305, 16) == 0
    assert f(2432, 17 * 31, 17, 16) == 0 and f(2432, 17 * 32, 17, 16) == 16
