"""The streaming sharded pass's index arithmetic (slice_row .. slice_slots of
csrc/internal.h, compiled for the host): the clusters' rows cover all rows,
every piece's slot is its own and inside the CTA's slots, and the merge reads
exactly the slots that the pieces of a row were written to."""
import pytest

import index_shim

CW = 32


@pytest.mark.parametrize("B,gamma,RV", [(16, 32, 9497), (1, 32, 6250), (7, 32, 550), (64, 64, 512), (5, 7, 1000),
                                        (2, 128, 4097), (76, 1, 700), (128, 64, 1251), (5, 8, 4001), (1, 1, 600), (3, 2, 18992)])
def test_slots(B, gamma, RV, G=76):
    L = index_shim.lib()
    nd, rows = B * gamma, B * (2 * gamma + 1)
    slots = L.shim_slice_slots(rows, G)
    cut = [L.shim_slice_row(nd, rows, c, G) for c in range(G + 1)]
    assert cut[0] == 0 and cut[G] == rows
    for ra, rb in zip(cut, cut[1:]):
        assert ra <= rb
        Tc = (rb - ra) * RV
        n0 = L.shim_slice_half(Tc, RV)
        written = {}
        for gw in range(CW):
            v, v1 = L.shim_slice_start(Tc, gw), L.shim_slice_start(Tc, gw + 1)
            while v < v1:
                l = v // RV
                e = min(v1, (l + 1) * RV)
                own, at = int(l >= n0), L.shim_slice_slot(l, n0, gw)
                assert 0 <= at < slots and (own, at) not in written
                written[(own, at)] = (l, v, e)
                v = e
        for l in range(rb - ra):
            own, f = int(l >= n0), l * RV
            fw, lw = L.shim_slice_owner(Tc, f), L.shim_slice_owner(Tc, f + RV - 1)
            pieces = [written.pop((own, L.shim_slice_slot(l, n0, w))) for w in range(fw, lw + 1)]
            assert len(pieces) <= CW and all(q[0] == l for q in pieces)
            assert pieces[0][1] == f and pieces[-1][2] == f + RV
            assert all(a[2] == b[1] for a, b in zip(pieces, pieces[1:]))
        assert not written
