// scan.cuh -- the streaming pass of the path: one read of every drafter and
// target logit, producing per-row partial softmax statistics.
//
// What it computes (per row of logits z over the vocabulary):
//   M = max z, S = sum exp(z - M), T2 = sum exp(z - M) (z - M) log2(e),
//   the lowest index attaining M, and for target rows the saturated rank of
//   the drafted token x: #{v : z(v) > z(x)} + #{v < x : z(v) = z(x)}.
// From these follow the quantities of Sec. 4.2 (raw confidence q = p_draft(x_j),
// LSE, maxprob, entropy) and the target facts that the acceptance rules of
// Sec. 3.1 and App. A.6 read.
//
// How: the rows of the call are laid end to end as one sequence of 16-byte
// vectors, split into contiguous ranges of equal cost, one per warp (a drafter
// vector weighs 10, a target vector 9: the drafter rows' entropy accumulator
// costs more; no per-tile scheduling).  Each warp streams its range through a
// private ring of two 4 KiB shared-memory tiles filled by 1D bulk copies
// (cp.async.bulk + mbarrier), keeps an online-softmax state per lane (packed
// f32x2 arithmetic, exp-sums as double-floats), reduces it across the warp at
// the end of each row piece and publishes a 32-byte partial.  The feature
// instantiation also publishes each drafter row piece's five largest entries
// (group_update / group_top5 below).
// The decide kernel (decide.cu) merges each row's partials and finalises the
// rows; keeping that out of the streaming work keeps it free of register
// spills.  Included by scan.cu (the streaming kernel) and pipe.cu (the
// pipelined round).
#pragma once

#include "internal.h"

namespace sdd {

namespace {

struct Cursor {
    int64_t v;     // absolute vector index
    int64_t r;     // row
    int32_t k;     // vector offset inside the row
};

__device__ __forceinline__ void row_locate(const ScanParams &p, const PartView &pv, int64_t r, int &gi, int64_t &lr,
                                           int &j, int &b, bool &b_ok) {
    gi = (r >= pv.rows0) ? 1 : 0;
    lr = gi ? r - pv.rows0 : r;
    const ScanGroup &G = p.grp[gi];
    const int64_t i = fast_div(lr, p.divNpos[gi]);
    j = static_cast<int>(lr - i * G.npos);
    b = G.bidx ? __ldg(G.bidx + i) : static_cast<int>(i);
    b_ok = (b >= 0 && b < p.B);
    if (!b_ok) b = 0;  // keep every address inside the tensor; the row is flagged at the end
}

__device__ __forceinline__ const char *row_base(const ScanParams &p, const PartView &pv, int64_t r) {
    int gi, j, b;
    int64_t lr;
    bool ok;
    row_locate(p, pv, r, gi, lr, j, b, ok);
    const ScanGroup &G = p.grp[gi];
    return G.base + (static_cast<int64_t>(b) * G.npos + j) * G.stride_bytes;
}


// A tile that is not full, or that ends a row whose length is not a whole
// number of vectors, is completed in shared memory with -inf entries so that
// the hot loop can read every vector of the tile unconditionally.
template <int DT>
__device__ __noinline__ void pad_tile(uint4 *tile, int n, int lane, bool row_end, int tail) {
    const uint4 ninf = (DT == SDD_BF16) ? make_uint4(kNegInfPairBf16, kNegInfPairBf16, kNegInfPairBf16, kNegInfPairBf16)
                                        : make_uint4(0xFF800000u, 0xFF800000u, 0xFF800000u, 0xFF800000u);
    for (int idx = n + lane; idx < kTileVec; idx += 32) tile[idx] = ninf;
    if (row_end && tail && lane == ((n - 1) & 31)) {
        uint4 w = tile[n - 1];
        mask_tail<DT>(w, tail);
        tile[n - 1] = w;
    }
    __syncwarp();
}

// Entries of the lane's vectors in a (full, padded) tile that rank before the
// drafted token tok: value above g, or equal to g at a lower index.
template <int DT>
__device__ __noinline__ int count_before(const uint4 *tile, int n, int k0, int lane, float g, int tok) {
    constexpr int EPV = (DT == SDD_BF16) ? 8 : 4;
    if (DT == SDD_BF16 && g > clamp_floor()) {
        // Packed compares, two entries per instruction (g is a bf16 value above
        // the clamp value, so clamping cannot change a comparison, and padded
        // entries are -inf).  Entries equal to g rank before the token only at a
        // lower index: counted one by one, in the rare tiles that hold any.
        const uint32_t gb = __float_as_uint(g) >> 16, g2 = gb | (gb << 16);
        int cnt = 0;
        uint32_t eq = 0;
#pragma unroll
        for (int i = 0; i < kVPL; ++i) {
            const uint4 w = tile[lane + 32 * i];
            const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                cnt += __popc(bf16x2_gt(u[q], g2) & 0x00010001u);
                eq |= bf16x2_eq(u[q], g2);
            }
        }
        if (eq) {
#pragma unroll 1
            for (int i = 0; i < kVPL; ++i) {
                const uint4 w = tile[lane + 32 * i];
#pragma unroll
                for (int e = 0; e < EPV; ++e)
                    cnt += (vec_elem<DT>(w, e) == g && (k0 + lane + 32 * i) * EPV + e < tok) ? 1 : 0;
            }
        }
        return cnt;
    }
    int cnt = 0;
#pragma unroll 1
    for (int i = 0; i < kVPL; ++i) {
        const int idx = lane + 32 * i;
        if (idx >= n) break;
        const uint4 w = clamp_vec<DT>(tile[idx]);
#pragma unroll
        for (int e = 0; e < EPV; ++e) {
            const float z = vec_elem<DT>(w, e);
            const int v = (k0 + idx) * EPV + e;
            cnt += (z > g || (z == g && v < tok)) ? 1 : 0;
        }
    }
    return cnt;
}

// Process one full tile: the lane's vectors are lane, lane+32, ... of the tile.
// Sums are relative to the integer reference st.r (log2 units), so a new
// maximum rescales by an exact power of two.  A new maximum only records the
// tile (st.amax = k0); the exact index is resolved once at the end of the piece.
// Pairs of entries go through the packed f32x2 pipe: y = z log2(e) - r,
// s += 2^y and, for drafter rows (ENT), t2 += 2^y (z - m) log2(e), m the
// lane's maximum (so the dominant term of a peaked row adds 0).  Drafter entries are
// clamped first (so a masked entry adds 0 * finite to t2); target rows need no
// clamp (2^-inf = 0 and the maximum starts at the clamp value).  The lane's
// exp-sum is an fp32 pair (s_hi, s_lo) updated by TwoSum once per tile.
// Returns the lane's tile maximum (clamp value included).
template <int DT, bool ENT>
__device__ __forceinline__ float process_tile(const uint4 *tile, int k0, int lane, SoftState &st, float &s_hi,
                                              float &s_lo) {
    // pass 1: the tile maximum (clamp value included)
    float cm;
    if (DT == SDD_BF16) {
        uint32_t mx = kClampPairBf16;
#pragma unroll
        for (int i = 0; i < kVPL; ++i) {
            const uint4 w = tile[lane + 32 * i];
            const uint32_t vm = bf16x2_max_nan(bf16x2_max_nan(w.x, w.y), bf16x2_max_nan(w.z, w.w));
            mx = bf16x2_max_nan(mx, vm);
        }
        cm = fmax_nan(bf16_lo(mx), bf16_hi(mx));
    } else {
        cm = clamp_floor();
#pragma unroll
        for (int i = 0; i < kVPL; ++i) {
            const uint4 w = tile[lane + 32 * i];
            const float vm = fmax_nan(fmax_nan(__uint_as_float(w.x), __uint_as_float(w.y)),
                                      fmax_nan(__uint_as_float(w.z), __uint_as_float(w.w)));
            cm = fmax_nan(cm, vm);
        }
    }
    if (cm > st.m) {
        st.amax = k0;
        // the entropy accumulator is kept against the lane's maximum: a new
        // maximum shifts it by (m_old - m_new) log2(e) per unit of the sum
        if (ENT) st.t2 = fmaf((st.m - cm) * kLog2e, s_hi + s_lo, st.t2);
        st.m = cm;
        const float rn = ceilf(cm * kLog2e);
        if (rn > st.r) {
            const float k = st.r - rn;
            const float sc = pow2f_int(k);   // exact power of two (0 below the normal range)
            if (ENT) st.t2 *= sc;
            s_hi *= sc;
            s_lo *= sc;
            st.r = rn;
        }
    }
    // pass 2: the exp-sums, the vectors re-read from shared memory two at a
    // time; unrolled, so the reads of later steps issue ahead of the
    // arithmetic of earlier ones
    const float nr = -st.r;
    const f2_t L2 = f2_pack(kLog2e, kLog2e), NR = f2_pack(nr, nr);
    // the lane maximum's own y (the same fma as an entry's): y - DM is an
    // entry's (z - m) log2(e), exactly 0 for the maximum itself
    const float dm = fmaf(st.m, kLog2e, nr);
    const f2_t DM = f2_pack(dm, dm);
    f2_t sa = f2_pack(0.f, 0.f), sb = sa, ta = sa, tb = sa;
    constexpr int PAIRS = (DT == SDD_BF16) ? 4 : 2;   // entry pairs per 16-byte vector
#pragma unroll
    for (int i = 0; i < kVPL; i += 2) {
        uint4 w[2];
        w[0] = tile[lane + 32 * i];
        w[1] = tile[lane + 32 * (i + 1)];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (ENT) w[h] = clamp_vec<DT>(w[h]);
            const uint32_t *u = reinterpret_cast<const uint32_t *>(&w[h]);
#pragma unroll
            for (int q = 0; q < PAIRS; ++q) {
                const f2_t z = (DT == SDD_BF16) ? f2_pack(bf16_lo(u[q]), bf16_hi(u[q]))
                                                : f2_pack(__uint_as_float(u[2 * q]), __uint_as_float(u[2 * q + 1]));
                const f2_t y = f2_fma(z, L2, NR);
                float y0, y1;
                f2_unpack(y, y0, y1);
                const f2_t e = f2_pack(ex2(y0), ex2(y1));
                if (q & 1) {
                    sb = f2_add(sb, e);
                    if (ENT) tb = f2_fma(e, f2_sub(y, DM), tb);
                } else {
                    sa = f2_add(sa, e);
                    if (ENT) ta = f2_fma(e, f2_sub(y, DM), ta);
                }
            }
        }
    }
    float s0, s1;
    f2_unpack(f2_add(sa, sb), s0, s1);
    if (ENT) {
        // A tile dominated by one term (the others sum to < 1/16 of it: the
        // lane holding the peak of a peaked row) loses those others' low bits
        // next to it, and they make the row's entropy.  Such a lane's terms
        // are re-summed by the whole warp -- the maximum counted apart, the
        // others summed among themselves -- from shared memory (rare: about
        // one lane-tile per peaked row).
        const float ecm = ex2(fmaf(cm, kLog2e, nr));
        unsigned dom = __ballot_sync(0xFFFFFFFFu, s0 + s1 < 1.0625f * ecm && cm > clamp_floor());
        while (dom) {
            const int src = __ffs(dom) - 1;
            dom &= dom - 1;
            // src's tile maximum and reference (every lane has its own)
            const float cms = __shfl_sync(0xFFFFFFFFu, cm, src);
            const float nrs = __shfl_sync(0xFFFFFFFFu, nr, src);
            // src's 8 vectors, 8 bf16 (or 4 fp32) entries each: lane l takes
            // entries l and l + 32 of them
            constexpr int EN = kVPL * 2 * PAIRS;   // entries of one lane-tile
            float small = 0.f, nmax = 0.f;
#pragma unroll
            for (int t = lane; t < EN; t += 32) {
                const int i = t / (2 * PAIRS), k = t % (2 * PAIRS);
                const uint4 w = clamp_vec<DT>(tile[src + 32 * i]);
                const int wi = (DT == SDD_BF16) ? (k >> 1) : k;   // (word picked by selects, not by index)
                const uint32_t uw = (wi < 2) ? ((wi == 0) ? w.x : w.y) : ((wi == 2) ? w.z : w.w);
                const float z = (DT == SDD_BF16) ? ((k & 1) ? bf16_hi(uw) : bf16_lo(uw)) : __uint_as_float(uw);
                if (z == cms)
                    nmax += 1.f;
                else
                    small += ex2(fmaf(z, kLog2e, nrs));
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                small += __shfl_xor_sync(0xFFFFFFFFu, small, off);
                nmax += __shfl_xor_sync(0xFFFFFFFFu, nmax, off);
            }
            if (lane == src) {
                s0 = nmax * ecm;   // (nmax <= 64: exact)
                s1 = small;
            }
        }
    }
    float e1, e2, h;
    two_sum(s_hi, s0, h, e1);
    two_sum(h, s1, s_hi, e2);
    s_lo += e1 + e2;
    if (ENT) {
        float t0, t1;
        f2_unpack(f2_add(ta, tb), t0, t1);
        st.t2 += t0 + t1;
    }
    return cm;
}

// Extended features (drafter rows): the five largest clamped entries of a
// piece, with multiplicity.  A group is one lane's kVPL vectors of one tile.
// The five largest entries lie in the five groups with the largest maxima:
// every other group's maximum is at most the fifth largest group maximum,
// which those five groups' maxima reach, so an entry outside them can only
// tie the fifth largest entry.  While the piece streams, each lane keeps its
// five largest tile maxima (order-preserving integer keys) with the tiles'
// numbers; at the piece's end the warp merges the lanes' lists (five integer
// max reductions), re-reads the five groups (40 vectors, in halves over the
// lanes) from global memory and takes their five largest entries.
__device__ __forceinline__ uint32_t fkey(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float fkey_inv(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}

// The lane's list: ck descending, 0 = empty.  bf16 logits (exact in the upper
// half of a key): the key's upper half and, below it, the tile's number in the
// piece -- 16 bits, as a piece is at most a sixteenth of a row of 2 GiB, or a
// full grid's share of the device's memory (under 2^16 tiles of 4 KiB) -- so
// that an insertion is five pairs of integer max and min and takes no branch
// (~14 instructions a tile; with the tile numbers in registers of their own
// the update took 81, as nearly every tile has a lane that inserts).  fp32:
// the keys in ck, the tiles' numbers in ct.
template <int DT, int N>
__device__ __forceinline__ void group_update(float cm, uint32_t tile, uint32_t (&ck)[N], uint32_t (&ct)[N]) {
    if (DT == SDD_BF16) {
        uint32_t key = (fkey(cm) & 0xFFFF0000u) | (tile & 0xFFFFu);
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const uint32_t lo = min(ck[j], key);
            ck[j] = max(ck[j], key);
            key = lo;
        }
        return;
    }
    uint32_t key = fkey(cm);
    if (key <= ck[N - 1]) return;
#pragma unroll
    for (int j = 0; j < N; ++j)
        if (key > ck[j]) {
            const uint32_t tk = ck[j], tt = ct[j];
            ck[j] = key;
            ct[j] = tile;
            key = tk;
            tile = tt;
        }
}

// The five largest clamped entries (descending; -inf where the piece has
// fewer) of the piece [kb, ke) of row rowp, warp-uniform, from the lanes'
// group lists.
template <int DT>
__device__ __forceinline__ void group_top5(const char *rowp, int kb, int ke, int V, int lane, uint32_t (&ck)[5],
                                           uint32_t (&ct)[5], float (&t)[5]) {
    constexpr int EPV = (DT == SDD_BF16) ? 8 : 4;
    // (the rounds are rolled loops shifting their results in: this code runs
    // once per piece, and its instructions are fetched while L2 is busy)
    int gv[5];   // the five groups' first vectors (-1: none)
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        gv[k] = -1;
        t[k] = -INFINITY;
    }
#pragma unroll 1
    for (int k = 0; k < 5; ++k) {
        const uint32_t m = __reduce_max_sync(0xFFFFFFFFu, ck[0]);   // 0: every list is empty
        const int owner = __ffs(__ballot_sync(0xFFFFFFFFu, ck[0] == m)) - 1;
        const uint32_t tile = (DT == SDD_BF16) ? (m & 0xFFFFu) : __shfl_sync(0xFFFFFFFFu, ct[0], owner);
#pragma unroll
        for (int j = 0; j < 4; ++j) gv[j] = gv[j + 1];
        gv[4] = (m != 0u) ? kb + static_cast<int>(tile) * kTileVec + owner : -1;
        if (lane == owner) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                ck[j] = ck[j + 1];
                if (DT != SDD_BF16) ct[j] = ct[j + 1];
            }
            ck[4] = 0u;
        }
    }
    // half-vector u (0..79) of the groups: group u / 16, half u % 2 of its
    // (u % 16) / 2-th vector; lane q takes u = q, q + 32 and q + 64
    constexpr int HPV = EPV / 2;   // entries of a half-vector
    int vec[3];
    uint2 w[3];
#pragma unroll
    for (int h = 0; h < 3; ++h) {
        const int u = lane + 32 * h, g = u >> 4;
        int first = -1;
#pragma unroll
        for (int k = 0; k < 5; ++k)
            if (g == k) first = gv[k];
        const int v = first + 32 * ((u & 15) >> 1);
        vec[h] = (first >= 0 && v < ke) ? v : -1;
        w[h] = (vec[h] >= 0) ? __ldg(reinterpret_cast<const uint2 *>(rowp) + 2 * vec[h] + (u & 1)) : make_uint2(0, 0);
    }
    float e[3 * HPV];
#pragma unroll
    for (int h = 0; h < 3; ++h) {
        const uint4 c = clamp_vec<DT>(make_uint4(w[h].x, w[h].y, 0, 0));
        const int first = vec[h] * EPV + ((lane & 1) ? HPV : 0);   // (u and the lane have the same parity)
#pragma unroll
        for (int j = 0; j < HPV; ++j)
            e[h * HPV + j] = (vec[h] >= 0 && first + j < V) ? vec_elem<DT>(c, j) : -INFINITY;
    }
#pragma unroll 1
    for (int k = 0; k < 5; ++k) {   // five rounds: the warp's largest remaining entry
        float lm = e[0];
#pragma unroll
        for (int j = 1; j < 3 * HPV; ++j) lm = fmaxf(lm, e[j]);
        const uint32_t m = __reduce_max_sync(0xFFFFFFFFu, fkey(lm));
#pragma unroll
        for (int j = 0; j < 4; ++j) t[j] = t[j + 1];
        t[4] = fkey_inv(m);
        const int owner = __ffs(__ballot_sync(0xFFFFFFFFu, fkey(lm) == m)) - 1;
        if (lane == owner) {
            bool done = false;
#pragma unroll
            for (int j = 0; j < 3 * HPV; ++j)
                if (!done && e[j] == lm) {
                    e[j] = -INFINITY;
                    done = true;
                }
        }
    }
}

// What a warp needs of a row that its range touches, held one row per lane
// (RowWindow: rows first .. first + 31): computed for all the rows at once,
// with their token loads in flight together, when the warp starts.  The first
// tile of a full grid used to land 5.4 us after the kernel's wait (the range's
// ends, the rows and two dependent token loads one after another, ahead of the
// first tile's wait): with the two ends on two lanes, the rows on lanes and
// the token logits fetched behind the first copies 3.6 us.  Together with the
// piece's end below (2.4 -> 0.8 us) a 16-block streaming pass takes 51.1
// instead of 55.1 us (6.18 TB/s), one block 10.1 instead of 12.6 us.
struct RowWindow {
    int64_t first;
    const char *base;   // the row's logits
    int32_t tok;        // its drafted token (-1: none or out of range)
    float g;            // the token's clamped logit (NaN if none)
    uint32_t flags;     // kRowDrafter, kRowBadTok
};
constexpr uint32_t kRowDrafter = 1, kRowBadTok = 2;
// The kinds of rows in a call (scan_warp).  With one kind known, the streaming
// loop keeps one form of process_tile (119-121 registers for drafter rows
// instead of 124-128): GB300, confidence of 16 x 32 rows 32.7 -> 31.2 us, with
// the extended features 38.2 -> 35.7; of 128 x 32 187 -> 181 and 207 -> 188.
constexpr int kRowsMixed = 0, kRowsDrafter = 1, kRowsTarget = 2;

// Rows first + lane up to `last`; the token logits are loaded by window_logits.
__device__ __forceinline__ void window_rows(const ScanParams &p, const PartView &pv, int64_t first, int64_t last,
                                            int lane, RowWindow &w) {
    w.first = first;
    w.base = nullptr;
    w.tok = -1;
    w.flags = 0;
    const int64_t r = first + lane;
    if (r <= last) {
        int gi, j, b;
        int64_t lr;
        bool ok;
        row_locate(p, pv, r, gi, lr, j, b, ok);
        const ScanGroup &G = p.grp[gi];
        w.base = G.base + (static_cast<int64_t>(b) * G.npos + j) * G.stride_bytes;
        w.flags = (G.kind == 0) ? kRowDrafter : 0u;
        if (j < p.gamma) {
            w.tok = __ldg(p.tokens + static_cast<int64_t>(b) * p.gamma + j);
            w.flags |= kRowBadTok;   // (until window_logits has seen it)
        }
    }
}
template <int DT>
__device__ __forceinline__ void window_logits(const ScanParams &p, RowWindow &w) {
    w.g = __int_as_float(0x7FC00000);
    if ((w.flags & kRowBadTok) && w.tok >= 0 && w.tok < p.V) {
        w.flags &= ~kRowBadTok;
        w.g = fmax_nan(logit_at<DT>(w.base, w.tok), clamp_floor());
    } else {
        w.tok = -1;
    }
}
__device__ __forceinline__ const char *shfl_ptr(const char *ptr, int src) {
    return reinterpret_cast<const char *>(
        __shfl_sync(0xFFFFFFFFu, reinterpret_cast<unsigned long long>(ptr), src));
}

// The streaming work of streaming warp w of the CTA, once the work ahead of it
// in the stream has completed.  smem is the CTA's ring area,
// ring_bytes(STAGES, n_rings): one ring of STAGES tiles per streaming warp,
// then their barriers; this warp's is ring w.  FEAT: also the five largest logits of
// every drafter row piece (extended features); without it the code is
// unchanged.  KIND: the call's rows are all of one kind (the other kind's code
// is left out).  SHARES: the warps may have unequal shares (the pipelined round).
template <int DT, bool FEAT, int KIND = kRowsMixed, int STAGES = kStages, bool SHARES = false>
__device__ __forceinline__ void scan_warp(const ScanParams &p, unsigned char *smem, int w, int n_rings) {
    constexpr int kStages = STAGES;
    static_assert(!FEAT || KIND == kRowsDrafter, "the extended features are of drafter rows");
    const int lane = threadIdx.x & 31;
    const PartView pv = part_view(p);
    // the call's warps spread evenly over the CTAs (a call too small for every
    // warp, or a device block count, leaves warps of each CTA without work)
    const int wpc = p.nb_dev ? (pv.W + gridDim.x - 1) / gridDim.x : p.spread;
    const int64_t gw = static_cast<int64_t>(blockIdx.x) * wpc + w;
    if (w >= wpc || gw >= pv.W) return;
    // The sampling draw's arrival counters of this call's blocks start at zero
    // (the decide kernel behind this one reads them only after this grid has
    // completed), so the workspace needs no zero fill and calls of any shape
    // that fits it may follow one another.
    if (gw == 0 && p.dec.enabled && p.dec.res_count != nullptr)
        for (int i = lane; i < pv.nb; i += 32) p.dec.res_count[i] = 0u;
    constexpr int EPV = (DT == SDD_BF16) ? 8 : 4;
    const int tail = p.V % EPV;  // valid entries of the last vector of a row (0 = full)

    unsigned char *ring = smem + w * (kStages * kTileBytes);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + n_rings * kStages * kTileBytes) + w * kStages;
    if (lane == 0) {
#pragma unroll
        for (int s = 0; s < kStages; ++s) mbar_init(&bars[s], 1);
        fence_mbar_init();
    }
    __syncwarp();

    // the range's two ends by two lanes at once, then the rows it touches
    int64_t rs;
    int32_t ks;
    const int64_t vs = part_start<SHARES>(p, pv, gw + (lane & 1), rs, ks);
    const int64_t v0 = __shfl_sync(0xFFFFFFFFu, vs, 0), v1 = __shfl_sync(0xFFFFFFFFu, vs, 1);
    Cursor pc{v0, __shfl_sync(0xFFFFFFFFu, rs, 0), __shfl_sync(0xFFFFFFFFu, ks, 0)};
    const int64_t r_last = __shfl_sync(0xFFFFFFFFu, rs, 1) - (__shfl_sync(0xFFFFFFFFu, ks, 1) == 0 ? 1 : 0);
    Cursor cc = pc;
    RowWindow win;
    window_rows(p, pv, pc.r, r_last, lane, win);
    const char *prow = shfl_ptr(win.base, 0);
    const uint64_t pol = l2_evict_first_policy();   // the logits are read once
    uint32_t pending = 0;  // slots with a copy in flight
    uint32_t phase = 0;    // parity bit per slot
    bool drop = p.drop_copy != 0 && gw == 0;   // test hook: this warp's first copy is never issued

    auto issue = [&](int slot) {
        const int n = static_cast<int>(min(static_cast<int64_t>(min(kTileVec, p.RV - pc.k)), v1 - pc.v));
        if (drop) {
            // nothing will ever complete this slot's barrier: the consumer's
            // bounded wait runs out (no copy is in flight for the drain)
            drop = false;
        } else {
            if (lane == 0) {
            // the slot's previous contents were consumed into registers before the
            // warp reached this point (__syncwarp), so the copy may overwrite it
                mbar_arrive_expect_tx(&bars[slot], static_cast<uint32_t>(n) * 16u);
                bulk_g2s(ring + slot * kTileBytes, prow + static_cast<int64_t>(pc.k) * 16,
                         static_cast<uint32_t>(n) * 16u, &bars[slot], pol);
            }
            pending |= 1u << slot;
        }
        pc.v += n;
        pc.k += n;
        if (pc.k == p.RV && pc.v < v1) {
            pc.k = 0;
            pc.r += 1;
            prow = (pc.r - win.first < 32) ? shfl_ptr(win.base, static_cast<int>(pc.r - win.first))
                                           : row_base(p, pv, pc.r);
        }
    };
    for (int s = 0; s < kStages && pc.v < v1; ++s) issue(s);

    window_logits<DT>(p, win);   // (behind the first copies)

    SoftState st = soft_identity();
    uint32_t ck[5];        // FEAT: the lane's five largest tile maxima of the piece (keys) ...
    uint32_t ct[5];        // ... fp32: their tiles' numbers in the piece (drafter rows)
    int kb = 0;            // FEAT: the piece's first vector in the row
    uint32_t ftile = 0u;   // FEAT: the tile's number in the piece
    float s_hi = 0.f, s_lo = 0.f;   // the lane's exp-sum as an fp32 pair
    bool in_piece = false, fresh = false;   // fresh: the piece's token has not been fetched yet
    bool ent = false;      // warp-uniform: drafter row (entropy accumulator, clamped entries)
    int tok = -1;          // drafted token of the current row (-1: none or out of range)
    bool tok_bad = false;  // the row has a drafted token outside [0, V)
    float g = 0.f;         // its clamped logit (NaN if none)
    bool rank_on = false;  // warp-uniform: target row whose token's rank is still below kcap
    int wrank = 0;         // warp-uniform running rank count
    const char *crow = nullptr;
    int slot = 0;
    bool timed_out = false;
    while (cc.v < v1) {
        const int n = static_cast<int>(min(static_cast<int64_t>(min(kTileVec, p.RV - cc.k)), v1 - cc.v));
        if (!in_piece) {
            st = soft_identity();
            if (FEAT) {
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    ck[k] = 0u;
                    ct[k] = 0u;
                }
                kb = cc.k;
                ftile = 0u;
            }
            s_hi = 0.f;
            s_lo = 0.f;
            if (cc.r - win.first >= 32) {   // (a range of more than 32 rows)
                window_rows(p, pv, cc.r, r_last, lane, win);
                window_logits<DT>(p, win);
            }
            const int at = static_cast<int>(cc.r - win.first);
            crow = shfl_ptr(win.base, at);
            ent = (KIND == kRowsMixed) ? (__shfl_sync(0xFFFFFFFFu, win.flags, at) & kRowDrafter) != 0
                                       : KIND == kRowsDrafter;
            rank_on = false;
            wrank = 0;
            fresh = true;
            in_piece = true;
        }
        // warp-uniform outcome: a phase that one lane saw complete is complete for all
        if (!__any_sync(0xFFFFFFFFu, mbar_wait_bounded(&bars[slot], (phase >> slot) & 1u, p.wait_polls))) {
            timed_out = true;
            break;
        }
        uint4 *tile = reinterpret_cast<uint4 *>(ring + slot * kTileBytes);
        const bool row_end = (cc.k + n == p.RV);
        if (n < kTileVec || (row_end && tail)) pad_tile<DT>(tile, n, lane, row_end, tail);
        const float cm = (KIND == kRowsDrafter || (KIND == kRowsMixed && ent))
                             ? process_tile<DT, true>(tile, cc.k, lane, st, s_hi, s_lo)
                             : process_tile<DT, false>(tile, cc.k, lane, st, s_hi, s_lo);
        if (FEAT) group_update<DT>(cm, ftile++, ck, ct);
        if (fresh) {
            // the token's logit is first needed here: its load had the first
            // tile's copy and arithmetic to arrive
            const int at = static_cast<int>(cc.r - win.first);
            tok = __shfl_sync(0xFFFFFFFFu, win.tok, at);
            g = __shfl_sync(0xFFFFFFFFu, win.g, at);
            tok_bad = (__shfl_sync(0xFFFFFFFFu, win.flags, at) & kRowBadTok) != 0;
            rank_on = KIND != kRowsDrafter && !ent && tok >= 0;
            fresh = false;
        }
        if (KIND != kRowsDrafter && rank_on) {
            const bool want = cm >= g;
            if (__any_sync(0xFFFFFFFFu, want)) {
                int c = want ? count_before<DT>(tile, n, cc.k, lane, g, tok) : 0;
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, off);
                wrank += c;
                if (wrank >= p.kcap) rank_on = false;
            }
        }
        __syncwarp();
        phase ^= 1u << slot;
        pending &= ~(1u << slot);
        if (n < kTileVec || (row_end && tail)) fence_proxy_async_smem();  // generic writes of pad_tile
        if (pc.v < v1) issue(slot);
        slot = (slot + 1 == kStages) ? 0 : slot + 1;
        cc.v += n;
        cc.k += n;
        if (row_end || cc.v == v1) {
            // end of this warp's piece of row cc.r: its maximum M, the first
            // index that attains it, and the lanes' sums against M.  The lanes
            // that hold M re-read their vectors of its tile while the sums
            // are added.
            const float M = fkey_inv(__reduce_max_sync(0xFFFFFFFFu, fkey(st.m)));
            const bool holds = st.m == M && st.amax != INT32_MAX;
            const int va = (holds ? st.amax : 0) + lane;
            uint4 aw[kVPL];
#pragma unroll
            for (int i = 0; i < kVPL; ++i) {
                const int vec = va + 32 * i;
                aw[i] = (holds && vec < p.RV) ? __ldg(reinterpret_cast<const uint4 *>(crow) + vec)
                                              : make_uint4(0, 0, 0, 0);
            }
            float top[5];
            if (FEAT) group_top5<DT>(crow, kb, cc.k, p.V, lane, ck, ct, top);   // (cc.k: the piece's end)
            // every reference is a power of two below M's, so the rescaling is
            // exact; each step adds two lanes' double-floats the same way on
            // both, so all lanes agree
            const float rM = ceilf(M * kLog2e);
            const float sc = pow2f_int(st.r - rM);
            float t2 = sc * fmaf((st.m - M) * kLog2e, s_hi + s_lo, st.t2);
            float sh = s_hi * sc, sl = s_lo * sc;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                float h, e;
                two_sum(sh, __shfl_xor_sync(0xFFFFFFFFu, sh, off), h, e);
                fast_two_sum(h, e + (sl + __shfl_xor_sync(0xFFFFFFFFu, sl, off)), sh, sl);
                t2 += __shfl_xor_sync(0xFFFFFFFFu, t2, off);
            }
            int idx = INT32_MAX;
#pragma unroll
            for (int i = kVPL - 1; i >= 0; --i) {
                const int vec = va + 32 * i;
                const uint4 c = clamp_vec<DT>(aw[i]);
#pragma unroll
                for (int e = EPV - 1; e >= 0; --e)
                    if (vec * EPV + e < p.V && vec_elem<DT>(c, e) == M) idx = vec * EPV + e;
            }
            idx = __reduce_min_sync(0xFFFFFFFFu, holds ? idx : INT32_MAX);
            if (FEAT && lane == 0) {
                FeatPartial fp;
#pragma unroll
                for (int k = 0; k < 5; ++k) fp.top[k] = top[k];
                fp.pad[0] = fp.pad[1] = fp.pad[2] = 0.f;
                p.feat[cc.r + gw] = fp;
            }
            if (lane == 0) {
                Partial pt;
                pt.m = M;
                pt.r = rM;
                pt.t2 = t2;
                pt.sh = sh;
                pt.sl = sl;
                pt.amax = idx;
                pt.rank = tok_bad ? -1 : wrank;
                pt.g = g;
                p.partials[cc.r + gw] = pt;
            }
            in_piece = false;
            if (row_end) {
                cc.k = 0;
                cc.r += 1;
            }
        }
    }
    if (timed_out) {
        if (lane == 0) status_or(p.status, SDD_DEV_TIMEOUT);
        // let every copy still in flight land before the CTA's shared memory
        // goes away (the full limit, whatever the ring waits were given)
        for (int s = 0; s < kStages; ++s)
            if (pending & (1u << s)) (void)mbar_wait_bounded(&bars[s], (phase >> s) & 1u, kWaitPolls);
    }
}

}  // namespace

}  // namespace sdd
