// index_shim.cu -- the kernels' index arithmetic (csrc/internal.h) behind a C interface, for the CPU tests.
#include "../paper_2608_14787_gb300/csrc/internal.h"

using namespace sdd;

extern "C" {

// A launch over nb blocks of npos0 drafter rows and npos1 target rows (0: one group) of RV vectors on `ctas` CTAs: kind 0
// the streaming kernel's cut, 1 the pipelined pass's beside the narrow decide team, 2 beside the wide one.  Fills start
// [W + 1], row and vec (the row that holds each start and the vector in it); returns W (0: `start` holds under W + 1).
int64_t shim_cut(int kind, int nb, int npos0, int npos1, int RV, int ctas, int64_t cap, int64_t *start, int64_t *row,
                 int32_t *vec, int64_t nv, const int64_t *v, int64_t *owner, int64_t *facts) {
    ScanParams p{};
    p.n_groups = npos1 > 0 ? 2 : 1;
    for (int g = 0; g < 2; ++g) {
        p.grp[g].kind = g;
        p.grp[g].nb = nb;
        p.grp[g].npos = g ? npos1 : npos0;
    }
    p.RV = RV;
    p.rows0 = static_cast<int64_t>(nb) * npos0;
    p.rows = p.rows0 + static_cast<int64_t>(nb) * npos1;
    p.T = p.rows * RV;
    p.ctas = ctas;
    const int wpc = kWarpsPerCta - (kind == 0 ? 0 : (kind == 1 ? kPipeTeam : kPipeTeamWide) / 32);
    if (kind == 0) {
        p.W = scan_warps(static_cast<int64_t>(ctas) * wpc, p.T, p.rows);
        set_divisors(p);
    } else {
        p.W = scan_warps(static_cast<int64_t>(ctas) * wpc, p.T, p.rows, kPipePieces);
        set_divisors(p, kPipeCostDrafter, kPipeCostTarget);
        if (wpc == kShareWarps && p.W == ctas * wpc && p.whole == 0) set_shares(p);
    }
    const PartView pv{nb, p.rows0, p.rows, p.T, p.T0, p.C, p.W};
    if (cap < p.W + 1) return 0;
    for (int64_t w = 0; w <= p.W; ++w) start[w] = part_start<true>(p, pv, w, row[w], vec[w]);
    for (int64_t i = 0; i < nv; ++i) owner[i] = part_owner(p, pv, v[i]);
    facts[0] = p.whole;
    facts[1] = p.units;
    facts[2] = p.C;
    return p.W;
}

int64_t shim_whole_pieces(int64_t W_max, int64_t T, int64_t rows, int64_t most) { return whole_pieces(W_max, T, rows, most); }
int64_t shim_share_start(int64_t w) { return share_start(w); }
int64_t shim_share_warp(int64_t u) { return share_warp(u); }

int shim_slice_row(int nd, int rows, int c, int G) { return slice_row(nd, rows, c, G); }
int64_t shim_slice_start(int64_t Tc, int w) { return slice_start(Tc, w); }
int shim_slice_owner(int64_t Tc, int64_t v) { return slice_owner(Tc, v); }
int shim_slice_half(int64_t Tc, int RV) { return slice_half(Tc, RV); }
int shim_slice_slot(int l, int n0, int w) { return slice_slot(l, n0, w); }
int shim_slice_slots(int64_t rows, int clusters) { return slice_slots(rows, clusters); }
}
