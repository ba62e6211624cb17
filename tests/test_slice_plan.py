"""The streaming sharded pass's index arithmetic (shard_stream_kernel of
csrc/shard.cu) on the CPU: the clusters' rows cover all rows, every piece's
slot is its own and inside the CTA's slots, and the merge reads exactly the
slots that the pieces of a row were written to."""
import pytest

CW, WARPS = 32, 16


def _row(nd, rows, c, G):
    cd, ct = nd * 10, nd * 10 + (rows - nd) * 9
    x = ct * c // G
    return -(-x // 10) if x <= cd else nd + -(-(x - cd) // 9)


def _plan(rows, G, RV):
    most = -(-rows // G)
    if RV < 512:
        return 0
    return (most * 10 // 9 + 2) // 2 + 2 + 2 * WARPS


@pytest.mark.parametrize("B,gamma,RV", [(16, 32, 9497), (1, 32, 6250), (7, 32, 550), (64, 64, 512), (5, 7, 1000),
                                        (2, 128, 4097), (76, 1, 700), (128, 64, 1251), (5, 8, 4001), (1, 1, 600), (3, 2, 18992)])
def test_slots(B, gamma, RV, G=76):
    nd, rows = B * gamma, B * (2 * gamma + 1)
    slots = _plan(rows, G, RV)
    if not slots:
        pytest.skip("one CTA per row")
    assert _row(nd, rows, 0, G) == 0 and _row(nd, rows, G, G) == rows
    for c in range(G):
        ra, rb = _row(nd, rows, c, G), _row(nd, rows, c + 1, G)
        assert ra <= rb
        Tc = (rb - ra) * RV
        n0 = -(-(Tc * WARPS // CW) // RV)
        written = {}
        for gw in range(CW):
            v, v1 = Tc * gw // CW, Tc * (gw + 1) // CW
            while v < v1:
                l = v // RV
                e = min(v1, (l + 1) * RV)
                own = 1 if l >= n0 else 0
                at = (l - n0) + (gw - WARPS) if own else l + gw
                assert 0 <= at < slots and (own, at) not in written
                written[(own, at)] = (l, v, e)
                v = e
        for l in range(rb - ra):
            own = 1 if l >= n0 else 0
            f = l * RV
            fw, lw = ((f + 1) * CW - 1) // Tc, ((f + RV) * CW - 1) // Tc
            at = [(l - n0) - WARPS + w if own else l + w for w in range(fw, lw + 1)]
            pieces = [written.pop((own, a)) for a in at]
            assert len(at) <= 32 and all(q[0] == l for q in pieces)
            assert pieces[0][1] == f and pieces[-1][2] == f + RV
            assert all(a[2] == b[1] for a, b in zip(pieces, pieces[1:]))
        assert not written
