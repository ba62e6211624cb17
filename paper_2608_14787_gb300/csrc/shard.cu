// shard.cu -- the per-slice half of the vocabulary-sharded round (a
// tensor-parallel LM head: each rank holds one contiguous vocabulary slice
// [v0, v1) of every drafter and target row).
//
//  * shard_stream_kernel -- rows streamed through per-warp rings by clusters of
//    two CTAs (below); every call but those that stream_plan leaves to the next.
//  * shard_partials_kernel -- one CTA per row of the slice.  Each thread
//    streams its 16-byte vectors (ascending), keeping the online-softmax state
//    of its entries relative to an integer reference in log2 units (a new
//    maximum rescales the sums by an exact power of two), the first index of
//    its maximum and the drafter entropy accumulator; on target rows of a
//    round with the top-k rule each warp keeps its kcap highest-ranked
//    vectors in a list held one key per lane.  The CTA merges the threads'
//    states in thread order and selects the slice's kcap largest entries
//    (value descending, index ascending), then one thread writes the row's
//    record.  Logits are floored at -2^23 as in the
//    streaming kernel; entries past the slice width weigh nothing.
//
// The records of all slices are merged, and every rule of the round runs, in
// decide_kernel (rules.cuh: merge_row_shards); the draw that follows the
// exchange of the slices' draw-row masses is shard_draw_kernel (decide.cu).
#include <algorithm>
#include <atomic>

#include "scan.cuh"
#include "rules.cuh"

namespace sdd {

namespace {

// One CTA of four warps per row and eight CTAs per SM (64 registers): a c3
// slice holds 1,040 rows, one wave on 152 SMs.  (With 256-thread CTAs, four
// per SM, and per-thread candidate lists in shared memory, a half-vocabulary
// slice took 84 us; as here, ~55 us.)
constexpr int kShardThreads = 128;
constexpr int kShardMinCtas = 8;
constexpr int kShardU = 4;   // 16-byte vectors per thread in flight

// Order key of a candidate: larger value first, then lower index (an
// unsigned comparison of the keys is that order; a real entry's key is > 0).
__device__ __forceinline__ uint64_t cand_key(float z, int v) {
    uint32_t u = __float_as_uint(z);
    u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    return (static_cast<uint64_t>(u) << 32) | static_cast<uint32_t>(~static_cast<uint32_t>(v));
}
__device__ __forceinline__ float cand_value(uint64_t key) {
    const uint32_t e = static_cast<uint32_t>(key >> 32);
    return __uint_as_float((e & 0x80000000u) ? (e & 0x7FFFFFFFu) : ~e);
}
__device__ __forceinline__ int cand_index(uint64_t key) {
    return static_cast<int>(~static_cast<uint32_t>(key));
}

__device__ __forceinline__ uint64_t warp_max_u64(uint64_t v) {
    const uint32_t hi = static_cast<uint32_t>(v >> 32);
    const uint32_t mh = __reduce_max_sync(0xFFFFFFFFu, hi);
    const uint32_t ml = __reduce_max_sync(0xFFFFFFFFu, hi == mh ? static_cast<uint32_t>(v) : 0u);
    return (static_cast<uint64_t>(mh) << 32) | ml;
}

// The rare paths of the per-element work, kept out of line so that the
// common path is not compiled into predicated copies of them.
//
// The first index (ascending) of the value m in one vector whose entries
// start at index idx0; m is one of them.
template <int DT>
__device__ __noinline__ int vector_first_index(uint4 w, int idx0, float m) {
    constexpr int EPV = (DT == SDD_BF16) ? 8 : 4;
    for (int e = 0; e < EPV; ++e)
        if (vec_elem_sel<DT>(w, e) == m) return idx0 + e;
    return INT32_MAX;
}

// One key into a warp's candidate list: lane k < kl holds the list's k-th
// key (descending; 0 = empty), every lane returns its new entry.
__device__ __forceinline__ uint64_t warp_list_insert(uint64_t lk, uint64_t key, int kl, int lane) {
    const int pos = __popc(__ballot_sync(0xFFFFFFFFu, lk > key));   // keys ranking before it
    const uint64_t up = __shfl_up_sync(0xFFFFFFFFu, lk, 1);
    if (lane < kl && lane > pos) return up;
    if (lane < kl && lane == pos) return key;
    return lk;
}

// The running state of one thread's entries of a row.
struct ShardAcc {
    SoftState st;
    float s_hi, s_lo;   // exp-sum relative to 2^r, as an unevaluated pair
    bool nan;
    uint64_t lk;        // candidate rows: this lane's entry of the warp's list
    float wthr;         // value of the list's last key once full, else -inf
};

// One chunk (kShardU vectors per lane, lane-contiguous) of a row.  DRAFT: a
// drafter row (entropy accumulator, compensated sums); CANDL: a target row
// of a round with the top-k rule (the warp's candidate list); FULL: every
// vector of the warp's chunk lies inside the slice and before a ragged last
// vector (no guards).  Warp-uniform: every lane of the warp runs the same
// chunk, lanes past the end on floored -inf vectors that weigh nothing.
template <int DT, bool DRAFT, bool CANDL, bool FULL>
__device__ __forceinline__ void shard_chunk(const char *row, const ShardParams &sp, int v0, int kl, int lane,
                                            ShardAcc &a) {
    constexpr int EPV = (DT == SDD_BF16) ? 8 : 4;
    constexpr int PAIRS = EPV / 2;
    uint4 w[kShardU];
    float vm[kShardU];   // each vector's maximum (floored; NaN kept)
#pragma unroll
    for (int u = 0; u < kShardU; ++u) {
        const int vec = v0 + u * kShardThreads;
        if (FULL || vec < sp.RVs) {
            w[u] = __ldcs(reinterpret_cast<const uint4 *>(row) + vec);
        } else {
            const uint32_t ni = (DT == SDD_BF16) ? kNegInfPairBf16 : 0xFF800000u;
            w[u] = make_uint4(ni, ni, ni, ni);
        }
    }
    float cm = clamp_floor();
#pragma unroll
    for (int u = 0; u < kShardU; ++u) {
        const int vec = v0 + u * kShardThreads;
        if (!FULL && vec < sp.RVs && (vec + 1) * EPV > sp.Vs) mask_tail<DT>(w[u], sp.Vs - vec * EPV);
        w[u] = clamp_vec<DT>(w[u]);   // entries past the slice and masked ones: the floor
        const uint32_t *q = reinterpret_cast<const uint32_t *>(&w[u]);
        if (DT == SDD_BF16) {
            const uint32_t m2 = bf16x2_max_nan(bf16x2_max_nan(q[0], q[1]), bf16x2_max_nan(q[2], q[3]));
            vm[u] = fmax_nan(bf16_lo(m2), bf16_hi(m2));
        } else {
            vm[u] = fmax_nan(fmax_nan(__uint_as_float(q[0]), __uint_as_float(q[1])),
                             fmax_nan(__uint_as_float(q[2]), __uint_as_float(q[3])));
        }
        cm = fmax_nan(cm, vm[u]);
    }
    a.nan |= isnan(cm);
    if (cm > a.st.m) {
        // a new maximum (rare): its first index, in the first vector that holds it
        int us = kShardU - 1;
#pragma unroll
        for (int u = kShardU - 2; u >= 0; --u) us = (vm[u] == cm) ? u : us;
        uint4 ws = w[kShardU - 1];
#pragma unroll
        for (int u = kShardU - 2; u >= 0; --u) ws = (u == us) ? w[u] : ws;
        a.st.amax = vector_first_index<DT>(ws, (v0 + us * kShardThreads) * EPV, cm);
        // t2 against the maximum (as in the streaming kernel)
        if (DRAFT) a.st.t2 = fmaf((a.st.m - cm) * kLog2e, a.s_hi + a.s_lo, a.st.t2);
        a.st.m = cm;
        const float rn = ceilf(cm * kLog2e);
        if (rn > a.st.r) {
            const float sc = pow2f_int(a.st.r - rn);   // exact power of two (0 below the normal range)
            if (DRAFT) a.st.t2 *= sc;
            a.s_hi *= sc;
            a.s_lo *= sc;
            a.st.r = rn;
        }
    }
    if (CANDL) {
#pragma unroll
        for (int u = 0; u < kShardU; ++u) {
            const int vec = v0 + u * kShardThreads;
            // (a vector tying the last key has a larger index: it ranks after it)
            unsigned pend = __ballot_sync(0xFFFFFFFFu, vm[u] > a.wthr && (FULL || vec < sp.RVs));
            if (pend) {
                const uint64_t mine = cand_key(vm[u], vec);
                while (pend) {
                    const int src = __ffs(pend) - 1;
                    pend &= pend - 1;
                    a.lk = warp_list_insert(a.lk, __shfl_sync(0xFFFFFFFFu, mine, src), kl, lane);
                }
                const uint64_t last = __shfl_sync(0xFFFFFFFFu, a.lk, kl - 1);
                a.wthr = (last != 0ull) ? cand_value(last) : -INFINITY;
            }
        }
    }
    // the exp-sums, two entries at a time (drafter rows: compensated, so
    // that the small terms of a peaked row survive next to its peak)
    const f2_t L2 = f2_pack(kLog2e, kLog2e);
    const float nr = -a.st.r;
    const f2_t NR = f2_pack(nr, nr);
    const float dm = fmaf(a.st.m, kLog2e, nr);
    const f2_t DM = f2_pack(dm, dm);
    f2_t sa = f2_pack(0.f, 0.f), ca = sa, ta = sa;
#pragma unroll
    for (int u = 0; u < kShardU; ++u) {
        const uint32_t *q = reinterpret_cast<const uint32_t *>(&w[u]);
#pragma unroll
        for (int h = 0; h < PAIRS; ++h) {
            const f2_t z = (DT == SDD_BF16) ? f2_pack(bf16_lo(q[h]), bf16_hi(q[h]))
                                            : f2_pack(__uint_as_float(q[2 * h]), __uint_as_float(q[2 * h + 1]));
            const f2_t y = f2_fma(z, L2, NR);
            float y0, y1;
            f2_unpack(y, y0, y1);
            const f2_t e = f2_pack(ex2(y0), ex2(y1));
            if (DRAFT) {
                const f2_t yk = f2_sub(e, ca), t = f2_add(sa, yk);
                ca = f2_sub(f2_sub(t, sa), yk);
                sa = t;
                ta = f2_fma(e, f2_sub(y, DM), ta);
            } else {
                sa = f2_add(sa, e);
            }
        }
    }
    float a0, a1, h, e1, e2;
    f2_unpack(sa, a0, a1);
    two_sum(a.s_hi, a0, h, e1);
    two_sum(h, a1, a.s_hi, e2);
    if (DRAFT) {
        float c0, c1, t0, t1;
        f2_unpack(ca, c0, c1);
        f2_unpack(ta, t0, t1);
        a.s_lo += (e1 + e2) - (c0 + c1);
        a.st.t2 += t0 + t1;
    } else {
        a.s_lo += e1 + e2;
    }
}

// A thread's part of a row: chunks v0 = tid + c * kShardThreads * kShardU,
// run while the warp's first lane is inside the row.
template <int DT, bool DRAFT, bool CANDL>
__device__ __forceinline__ ShardAcc shard_row(const char *row, const ShardParams &sp, int kl, int tid) {
    constexpr int EPV = (DT == SDD_BF16) ? 8 : 4;
    const int lane = tid & 31;
    ShardAcc a;
    a.st = soft_identity();
    a.s_hi = a.s_lo = 0.f;
    a.nan = false;
    a.lk = 0ull;
    a.wthr = -INFINITY;
    const int rvf = (sp.Vs % EPV == 0) ? sp.RVs : sp.RVs - 1;   // vectors wholly inside the slice
    for (int v0 = tid; v0 - lane < sp.RVs; v0 += kShardThreads * kShardU) {
        if ((v0 - lane) + 31 + (kShardU - 1) * kShardThreads < rvf)
            shard_chunk<DT, DRAFT, CANDL, true>(row, sp, v0, kl, lane, a);
        else
            shard_chunk<DT, DRAFT, CANDL, false>(row, sp, v0, kl, lane, a);
    }
    return a;
}

template <int DT, bool CAND>
__global__ void __launch_bounds__(kShardThreads, kShardMinCtas) shard_partials_kernel(const __grid_constant__ ShardParams sp) {
    constexpr int EPV = (DT == SDD_BF16) ? 8 : 4;
    constexpr int NW = kShardThreads / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t r = blockIdx.x;
    const int64_t nd = static_cast<int64_t>(sp.B) * sp.gamma;
    griddep_wait();
    const bool drafter = r < nd;
    const char *row;
    int tok = -1;
    bool has_tok;
    if (drafter) {
        row = sp.zd + r * sp.stride_bytes;
        tok = __ldg(sp.tokens + r);
        has_tok = true;
    } else {
        const int64_t rr = r - nd;
        const int b = static_cast<int>(rr / (sp.gamma + 1)), j = static_cast<int>(rr % (sp.gamma + 1));
        row = sp.zt + rr * sp.stride_bytes;
        has_tok = j < sp.gamma;
        if (has_tok) tok = __ldg(sp.tokens + static_cast<int64_t>(b) * sp.gamma + j);
    }
    const bool tok_out = has_tok && (tok < 0 || tok >= sp.V);
    const bool in_slice = has_tok && !tok_out && tok >= sp.v0 && tok < sp.v0 + sp.Vs;
    const bool cand = CAND && !drafter;

    // target rows: the warp's kcap highest-ranked vectors, ranked by their
    // maximum (larger first, then lower vector index), held one key per lane
    // in descending order.  The kcap largest entries of the slice lie in the
    // slice's kcap highest-ranked vectors (an entry outside them has kcap
    // vectors ranked above its own, each holding an entry that ranks before
    // it), so the CTA selects those vectors at the end and takes the kcap
    // largest of their entries.
    const int kl = cand ? sp.kcap : 0;   // list length
    ShardAcc acc = drafter ? shard_row<DT, true, false>(row, sp, 0, tid)
                           : (cand ? shard_row<DT, false, CAND>(row, sp, kl, tid)
                                   : shard_row<DT, false, false>(row, sp, 0, tid));
    SoftState st = acc.st;
    const uint64_t lk = acc.lk;
    const bool nan = acc.nan;
    const float s_hi = acc.s_hi, s_lo = acc.s_lo;
    if (nan) st.m = qnan();
    st.sh = s_hi;
    st.sl = s_lo;
    st.rank = 0;

    // CTA merge of the threads' states, in thread order
    __shared__ SoftState s_st[NW];
    const SoftState wst = soft_warp_reduce(st);
    if (lane == 0) s_st[warp] = wst;

    // the slice's kcap highest-ranked vectors: the warps' lists in shared
    // memory, kcap rounds of a warp maximum over them (one warp); then the
    // kcap largest entries of those vectors (one warp, kcap rounds)
    __shared__ uint64_t s_wl[NW * SDD_SHARD_KMAX];
    __shared__ uint64_t s_top[SDD_SHARD_KMAX];
    __shared__ uint64_t s_ent[SDD_SHARD_KMAX * 8];
    const int kc = cand ? sp.kcap : 0;
    if (lane < kc) s_wl[warp * SDD_SHARD_KMAX + lane] = lk;
    __syncthreads();
    if (kc > 0 && warp == 0) {
        constexpr int PER = (NW * SDD_SHARD_KMAX + 31) / 32;
        uint64_t mk[PER];
#pragma unroll
        for (int t = 0; t < PER; ++t) {
            const int i = lane + 32 * t;
            mk[t] = (i < NW * SDD_SHARD_KMAX && (i % SDD_SHARD_KMAX) < kc) ? s_wl[i] : 0ull;
        }
        for (int round = 0; round < kc; ++round) {
            uint64_t mine = 0ull;
#pragma unroll
            for (int t = 0; t < PER; ++t) mine = (mk[t] > mine) ? mk[t] : mine;
            const uint64_t best = warp_max_u64(mine);
#pragma unroll
            for (int t = 0; t < PER; ++t) mk[t] = (best != 0ull && mk[t] == best) ? 0ull : mk[t];   // unique keys
            if (lane == 0) s_top[round] = best;
        }
    }
    __syncthreads();
    if (kc > 0) {
        // the entries of the selected vectors (re-read: kc x 16 bytes), keyed by value and global index
        if (tid < kc) {
            const uint64_t vk = s_top[tid];
            uint4 wv = make_uint4(0, 0, 0, 0);
            const int vec = (vk != 0ull) ? cand_index(vk) : -1;
            if (vec >= 0) wv = clamp_vec<DT>(__ldg(reinterpret_cast<const uint4 *>(row) + vec));
#pragma unroll
            for (int e = 0; e < EPV; ++e) {
                const int idx = vec * EPV + e;
                const float x = vec_elem<DT>(wv, e);
                s_ent[tid * 8 + e] = (vec >= 0 && idx < sp.Vs && !isnan(x)) ? cand_key(x, sp.v0 + idx) : 0ull;
            }
#pragma unroll
            for (int e = EPV; e < 8; ++e) s_ent[tid * 8 + e] = 0ull;
        }
        __syncthreads();
        if (warp == 0) {
            const int n = kc * 8;
            for (int round = 0; round < kc; ++round) {
                uint64_t mine = 0ull;
                int at = -1;
                for (int t = lane; t < n; t += 32)
                    if (s_ent[t] > mine) {
                        mine = s_ent[t];
                        at = t;
                    }
                const uint64_t best = warp_max_u64(mine);
                if (best != 0ull && mine == best) s_ent[at] = 0ull;   // unique keys: one lane takes it
                if (lane == 0) s_top[round] = best;
                __syncwarp();
            }
        }
    }
    __syncthreads();   // (every warp's state in s_st; the selection done)

    if (tid == 0) {
        SoftState a = s_st[0];
#pragma unroll
        for (int q = 1; q < NW; ++q) a = soft_merge(a, s_st[q]);
        sdd_shard_partial rec;
        rec.m = a.m;
        rec.r = a.r;
        rec.t2 = a.t2;
        rec.sh = a.sh;
        rec.sl = a.sl;
        rec.amax = (a.amax == INT32_MAX) ? INT32_MAX : sp.v0 + a.amax;
        rec.g = qnan();
        if (in_slice) {
            const int li = tok - sp.v0;
            float x;
            if (DT == SDD_BF16) {
                const uint16_t h = __ldg(reinterpret_cast<const unsigned short *>(row) + li);
                x = __uint_as_float(static_cast<uint32_t>(h) << 16);
            } else {
                x = __ldg(reinterpret_cast<const float *>(row) + li);
            }
            rec.g = fmax_nan(x, clamp_floor());
        }
        int nc = 0;
#pragma unroll
        for (int k = 0; k < SDD_SHARD_KMAX; ++k) {
            const uint64_t key = (k < kc) ? s_top[k] : 0ull;
            rec.cz[k] = (key != 0ull) ? cand_value(key) : -INFINITY;
            rec.cv[k] = (key != 0ull) ? cand_index(key) : INT32_MAX;
            nc += (key != 0ull) ? 1 : 0;
        }
        rec.info = (in_slice ? 1 : 0) | (tok_out ? 2 : 0) | (nc << 8);
        sp.out[r] = rec;
    }
}

// ---------------------------------------------------------------------------
// The streaming form: rows of the slice by clusters of two CTAs, one CTA per
// SM.  A cluster takes whole rows (as even a cost as whole rows allow: a
// drafter row 10, a target row 9), its 32 warps an equal run of their vectors
// each, streamed through the rings of the one-GPU pass (scan.cuh:
// process_tile).  A warp's piece of a row leaves its state and, for target
// rows of a round with the top-k rule, its kcap highest entries in the shared
// memory of the CTA that holds the row's first vector (the row that crosses
// the cluster's middle over distributed shared memory); after one cluster
// barrier each CTA merges its rows' pieces, a warp a row, into the records.
//
// Candidates: each lane keeps its kCandList largest tile maxima
// (group_update).  With T the kcap-th largest of all lanes' maxima, the piece's
// kcap highest entries are at least T and lie in the groups whose maximum is
// at least T: the warp re-reads those (about kcap of them), keeps the entries
// of at least T and ranks them by (value, index).  When more groups or entries
// reach T than there is room for, or a lane's whole list does (it may have
// dropped one), the piece is read again with the exact per-vector list
// (piece_candidates): ties in their hundreds, or short pieces.
//
// Bound by HBM and, at the end, by the last pieces' chain of selection and
// merge.  GB300, half of a 151,936 vocabulary, 16 x 32 positions, bf16 (158
// MB): 36.5 us with the top-k rule (k <= 10), 29.5 us without (5.35 TB/s),
// against 52.9 and 37.2 us with one CTA per row and register loads.
// ---------------------------------------------------------------------------
constexpr int kCandList = 7;      // tile maxima a lane keeps
constexpr int kCandGroups = 32;   // groups a piece re-reads at most
constexpr int kCandKeys = 64;     // entries it ranks at most

// A piece's slot: its partial, then its candidate keys, descending (0: none).
constexpr int kSlotBytes = static_cast<int>(sizeof(Partial)) + SDD_SHARD_KMAX * 8;

struct StreamParams {
    ShardParams sp;
    int32_t rows, nd;        // all rows, drafter rows
    int32_t slots;           // piece slots of a CTA
    uint32_t wait_polls;
    int32_t drop_copy;       // failure-detection test hook: the first warp never issues its first copy
};

__device__ __forceinline__ uint32_t slice_cta_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// A shared-memory address of this CTA in the cluster's CTA `rank`.
__device__ __forceinline__ uint32_t slice_map(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_slice_v4(uint32_t addr, uint4 v) {
    asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}
__device__ __forceinline__ void st_slice_u64(uint32_t addr, uint64_t v) {
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}

__device__ __forceinline__ const char *slice_row_base(const StreamParams &p, int r) {
    return r < p.nd ? p.sp.zd + r * p.sp.stride_bytes : p.sp.zt + (r - p.nd) * p.sp.stride_bytes;
}

// The kcap highest entries of vectors [kb, ke) of a row, exactly, by one warp:
// a list of the kcap highest vectors held one key per lane (larger maximum
// first, then lower index; a later vector that ties the last one ranks after
// it), then the kcap highest of their entries.  Lane k returns the k-th key.
template <int DT>
__device__ __noinline__ uint64_t piece_candidates(const char *row, int kb, int ke, int Vs, int v0, int kc) {
    constexpr int EPV = (DT == SDD_BF16) ? 8 : 4;
    const int lane = threadIdx.x & 31;
    uint64_t lk = 0ull;
    float thr = -INFINITY;
    for (int b = kb; b < ke; b += 32) {
        const int vec = b + lane;
        float vm = -INFINITY;
        if (vec < ke) {
            uint4 w = __ldg(reinterpret_cast<const uint4 *>(row) + vec);
            if ((vec + 1) * EPV > Vs) mask_tail<DT>(w, Vs - vec * EPV);
            w = clamp_vec<DT>(w);
#pragma unroll
            for (int e = 0; e < EPV; ++e) vm = fmaxf(vm, vec_elem<DT>(w, e));
        }
        unsigned pend = __ballot_sync(0xFFFFFFFFu, vm > thr);
        const uint64_t mine = cand_key(vm, vec);
        while (pend) {
            const int src = __ffs(pend) - 1;
            pend &= pend - 1;
            lk = warp_list_insert(lk, __shfl_sync(0xFFFFFFFFu, mine, src), kc, lane);
        }
        const uint64_t last = __shfl_sync(0xFFFFFFFFu, lk, kc - 1);
        thr = (last != 0ull) ? cand_value(last) : -INFINITY;
    }
    uint64_t key[8];
    const int vec = (lane < kc && lk != 0ull) ? cand_index(lk) : -1;
    uint4 w = make_uint4(0, 0, 0, 0);
    if (vec >= 0) w = clamp_vec<DT>(__ldg(reinterpret_cast<const uint4 *>(row) + vec));
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        key[e] = 0ull;
        if (e < EPV && vec >= 0 && vec * EPV + e < Vs) {
            const float x = vec_elem<DT>(w, e);
            if (!isnan(x)) key[e] = cand_key(x, v0 + vec * EPV + e);
        }
    }
    uint64_t out = 0ull;
    for (int k = 0; k < kc; ++k) {
        uint64_t mine = 0ull;
#pragma unroll
        for (int e = 0; e < 8; ++e) mine = key[e] > mine ? key[e] : mine;
        const uint64_t best = warp_max_u64(mine);
        if (lane == k) out = best;
#pragma unroll
        for (int e = 0; e < 8; ++e) key[e] = (key[e] == best) ? 0ull : key[e];   // (unique keys)
    }
    return out;
}

// The same from the lanes' lists of tile maxima; s_key: kCandKeys keys of
// scratch for this warp.
template <int DT>
__device__ __forceinline__ uint64_t group_candidates(const char *row, int kb, int ke, int Vs, int v0, int kc,
                                                     uint32_t (&ck)[kCandList], uint32_t (&ct)[kCandList],
                                                     uint64_t *s_key) {
    constexpr int EPV = (DT == SDD_BF16) ? 8 : 4;
    const int lane = threadIdx.x & 31;
    int first = -1, groups = 0, popped = 0;   // lane g < groups: group g's first vector
    uint32_t T = 0u;                          // the kcap-th maximum's key (its upper half for bf16)
    bool fits = true;
#pragma unroll 1
    for (;;) {
        const uint32_t m = __reduce_max_sync(0xFFFFFFFFu, ck[0]);
        const uint32_t mv = (DT == SDD_BF16) ? (m & 0xFFFF0000u) : m;
        if (m == 0u || (groups >= kc && mv < T)) break;
        if (groups == kCandGroups) {
            fits = false;
            break;
        }
        if (groups < kc) T = mv;
        const int owner = __ffs(__ballot_sync(0xFFFFFFFFu, ck[0] == m)) - 1;
        const uint32_t tile = (DT == SDD_BF16) ? (m & 0xFFFFu) : __shfl_sync(0xFFFFFFFFu, ct[0], owner);
        if (lane == groups) first = kb + static_cast<int>(tile) * kTileVec + owner;
        ++groups;
        if (lane == owner) {
            ++popped;
#pragma unroll
            for (int j = 0; j + 1 < kCandList; ++j) {
                ck[j] = ck[j + 1];
                if (DT != SDD_BF16) ct[j] = ct[j + 1];
            }
            ck[kCandList - 1] = 0u;
        }
    }
    // a piece of fewer groups than kcap: every entry counts
    if (groups < kc || __any_sync(0xFFFFFFFFu, popped == kCandList)) fits = false;
    int n = 0;
    if (fits) {
        const float thr = fkey_inv(DT == SDD_BF16 && !(T & 0x80000000u) ? (T | 0xFFFFu) : T);
        for (int u0 = 0; u0 < 8 * groups; u0 += 128) {
            uint4 w[4];
            int vec[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int u = u0 + 32 * h + lane;
                const int f = __shfl_sync(0xFFFFFFFFu, first, (u >> 3) & 31);
                const int v = f + 32 * (u & 7);
                vec[h] = (u < 8 * groups && v < ke) ? v : -1;
                w[h] = (vec[h] >= 0) ? __ldg(reinterpret_cast<const uint4 *>(row) + vec[h]) : make_uint4(0, 0, 0, 0);
            }
            // the lane's entries of at least T, a bit each; then a place for each
            uint32_t in = 0u;
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                w[h] = clamp_vec<DT>(w[h]);
#pragma unroll
                for (int e = 0; e < EPV; ++e)
                    if (vec[h] >= 0 && vec[h] * EPV + e < Vs && vec_elem<DT>(w[h], e) >= thr)
                        in |= 1u << (h * EPV + e);
            }
            const int mine = __popc(in);
            int incl = mine;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int t = __shfl_up_sync(0xFFFFFFFFu, incl, off);
                if (lane >= off) incl += t;
            }
            int at = n + incl - mine;
            n += __shfl_sync(0xFFFFFFFFu, incl, 31);
            while (in) {
                const int bit = __ffs(in) - 1, h = bit / EPV, e = bit % EPV;
                in &= in - 1;
                const uint4 c = (h < 2) ? (h == 0 ? w[0] : w[1]) : (h == 2 ? w[2] : w[3]);
                const int v = (h < 2) ? (h == 0 ? vec[0] : vec[1]) : (h == 2 ? vec[2] : vec[3]);
                if (at < kCandKeys) s_key[at] = cand_key(vec_elem_sel<DT>(c, e), v0 + v * EPV + e);
                ++at;
            }
        }
        if (n > kCandKeys) fits = false;
    }
    if (!fits) return piece_candidates<DT>(row, kb, ke, Vs, v0, kc);
    __syncwarp();
    // every key's rank among the n (they are unique); the kcap highest go back in order
    const uint64_t a = (lane < n) ? s_key[lane] : 0ull, b = (lane + 32 < n) ? s_key[lane + 32] : 0ull;
    int ra = 0, rb = 0;
    for (int t = 0; t < n; ++t) {
        const uint64_t o = s_key[t];
        ra += o > a ? 1 : 0;
        rb += o > b ? 1 : 0;
    }
    __syncwarp();
    if (a != 0ull && ra < kc) s_key[ra] = a;
    if (b != 0ull && rb < kc) s_key[rb] = b;
    __syncwarp();
    const uint64_t out = (lane < kc && lane < n) ? s_key[lane] : 0ull;
    __syncwarp();   // (the scratch serves the warp's next piece)
    return out;
}

template <int DT, bool CAND>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    shard_stream_kernel(const __grid_constant__ StreamParams p) {
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int EPV = (DT == SDD_BF16) ? 8 : 4;
    const ShardParams &sp = p.sp;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rank = static_cast<int>(slice_cta_rank());
    unsigned char *ring = smem + warp * (kStages * kTileBytes);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kWarpsPerCta * kStages * kTileBytes) + warp * kStages;
    unsigned char *slots = smem + kScanSmem;
    uint64_t *s_key = reinterpret_cast<uint64_t *>(slots + p.slots * kSlotBytes) + warp * kCandKeys;
    if (lane == 0) {
#pragma unroll
        for (int s = 0; s < kStages; ++s) mbar_init(&bars[s], 1);
        fence_mbar_init();
    }
    __syncwarp();
    // (the peer has started before anything is written to its shared memory)
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    griddep_wait();

    // the cluster's rows [ra, rb), this warp's vectors [v0, v1) of them
    const int cl = static_cast<int>(blockIdx.x) >> 1, G = static_cast<int>(gridDim.x) >> 1;
    const int bnd = slice_row(p.nd, p.rows, cl + (lane & 1), G);
    const int ra = __shfl_sync(0xFFFFFFFFu, bnd, 0), rb = __shfl_sync(0xFFFFFFFFu, bnd, 1);
    const int RV = sp.RVs, tail = sp.Vs % EPV;
    const int64_t Tc = static_cast<int64_t>(rb - ra) * RV;
    const int gw = rank * kWarpsPerCta + warp;
    const int64_t v0 = slice_start(Tc, gw), v1 = slice_start(Tc, gw + 1);
    const int n0 = slice_half(Tc, RV);   // CTA 0 owns the first n0 rows

    struct Cur {
        int64_t v;
        int l, k;   // row of the cluster, vector in it
    };
    Cur pc{v0, static_cast<int>(v0 / RV), 0};
    pc.k = static_cast<int>(v0 - static_cast<int64_t>(pc.l) * RV);
    Cur cc = pc;
    const char *prow = slice_row_base(p, ra + pc.l);
    const uint64_t pol = l2_evict_first_policy();
    uint32_t pending = 0, phase = 0;
    bool drop = p.drop_copy != 0 && cl == 0 && gw == 0;
    auto issue = [&](int slot) {
        const int n = static_cast<int>(min(static_cast<int64_t>(min(kTileVec, RV - pc.k)), v1 - pc.v));
        if (drop) {   // (test hook: nothing completes this slot's barrier, and nothing is in flight for the drain)
            drop = false;
        } else {
            if (lane == 0) {
                mbar_arrive_expect_tx(&bars[slot], static_cast<uint32_t>(n) * 16u);
                bulk_g2s(ring + slot * kTileBytes, prow + static_cast<int64_t>(pc.k) * 16,
                         static_cast<uint32_t>(n) * 16u, &bars[slot], pol);
            }
            pending |= 1u << slot;
        }
        pc.v += n;
        pc.k += n;
        if (pc.k == RV && pc.v < v1) {
            pc.k = 0;
            pc.l += 1;
            prow = slice_row_base(p, ra + pc.l);
        }
    };
    for (int s = 0; s < kStages && pc.v < v1; ++s) issue(s);

    SoftState st = soft_identity();
    uint32_t ck[kCandList], ct[kCandList];
    int kb = 0, slot = 0;
    float s_hi = 0.f, s_lo = 0.f;
    bool in_piece = false, ent = false, timed_out = false;
    const char *crow = nullptr;
    while (cc.v < v1) {
        const int n = static_cast<int>(min(static_cast<int64_t>(min(kTileVec, RV - cc.k)), v1 - cc.v));
        if (!in_piece) {
            st = soft_identity();
            s_hi = s_lo = 0.f;
#pragma unroll
            for (int k = 0; k < kCandList; ++k) ck[k] = ct[k] = 0u;
            kb = cc.k;
            ent = ra + cc.l < p.nd;
            crow = slice_row_base(p, ra + cc.l);
            in_piece = true;
        }
        if (!__any_sync(0xFFFFFFFFu, mbar_wait_bounded(&bars[slot], (phase >> slot) & 1u, p.wait_polls))) {
            timed_out = true;
            break;
        }
        uint4 *tile = reinterpret_cast<uint4 *>(ring + slot * kTileBytes);
        const bool row_end = cc.k + n == RV;
        const bool pad = n < kTileVec || (row_end && tail);
        if (pad) pad_tile<DT>(tile, n, lane, row_end, tail);
        const float cm = ent ? process_tile<DT, true>(tile, cc.k, lane, st, s_hi, s_lo)
                             : process_tile<DT, false>(tile, cc.k, lane, st, s_hi, s_lo);
        if (CAND && !ent) group_update<DT>(cm, static_cast<uint32_t>(cc.k - kb) / kTileVec, ck, ct);
        __syncwarp();
        phase ^= 1u << slot;
        pending &= ~(1u << slot);
        if (pad) fence_proxy_async_smem();   // generic writes of pad_tile
        if (pc.v < v1) issue(slot);
        slot = (slot + 1 == kStages) ? 0 : slot + 1;
        cc.v += n;
        cc.k += n;
        if (row_end || cc.v == v1) {
            // the piece's end, as in the one-GPU pass (scan_warp)
            const float M = fkey_inv(__reduce_max_sync(0xFFFFFFFFu, fkey(st.m)));
            const bool holds = st.m == M && st.amax != INT32_MAX;
            const int va = (holds ? st.amax : 0) + lane;
            uint4 aw[kVPL];
#pragma unroll
            for (int i = 0; i < kVPL; ++i)
                aw[i] = (holds && va + 32 * i < RV) ? __ldg(reinterpret_cast<const uint4 *>(crow) + va + 32 * i)
                                                    : make_uint4(0, 0, 0, 0);
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
                const uint4 c = clamp_vec<DT>(aw[i]);
#pragma unroll
                for (int e = EPV - 1; e >= 0; --e)
                    if ((va + 32 * i) * EPV + e < sp.Vs && vec_elem<DT>(c, e) == M) idx = (va + 32 * i) * EPV + e;
            }
            idx = __reduce_min_sync(0xFFFFFFFFu, holds ? idx : INT32_MAX);
            uint64_t key = 0ull;
            if (CAND && !ent) key = group_candidates<DT>(crow, kb, cc.k, sp.Vs, sp.v0, sp.kcap, ck, ct, s_key);
            const int own = cc.l >= n0 ? 1 : 0;
            const uint32_t dst = slice_map(smem_addr(slots + slice_slot(cc.l, n0, gw) * kSlotBytes), static_cast<uint32_t>(own));
            if (lane < 2) {
                Partial pt;
                pt.m = M;
                pt.r = rM;
                pt.t2 = t2;
                pt.sh = sh;
                pt.sl = sl;
                pt.amax = idx;
                pt.rank = 0;
                pt.g = 0.f;
                const uint4 *q = reinterpret_cast<const uint4 *>(&pt);
                st_slice_v4(dst + 16 * lane, lane == 0 ? q[0] : q[1]);
            }
            if (CAND && !ent && lane < SDD_SHARD_KMAX)
                st_slice_u64(dst + static_cast<uint32_t>(sizeof(Partial)) + 8 * lane, key);
            in_piece = false;
            if (row_end) {
                cc.k = 0;
                cc.l += 1;
            }
        }
    }
    // (a warp that gave up leaves its pieces' slots as they were, so the rows'
    // records are undefined; it meets the cluster's barrier below all the same)
    if (timed_out) {
        if (lane == 0) status_or(sp.status, SDD_DEV_TIMEOUT);
        for (int s = 0; s < kStages; ++s)
            if (pending & (1u << s)) (void)mbar_wait_bounded(&bars[s], (phase >> s) & 1u, kWaitPolls);
    }
    // the records of this CTA's rows, a warp a row; the drafted token and its
    // logit (two dependent loads) of the warp's first row ahead of the barrier
    const int l0 = rank ? n0 : 0, l1 = rank ? rb - ra : min(n0, rb - ra);
    bool tok_out = false, in_slice = false;
    float g = qnan();
    auto token = [&](int l) {
        const int r = ra + l;
        int tok = -1;
        bool has_tok = true;
        if (r < p.nd) {
            tok = __ldg(sp.tokens + r);
        } else {
            const int rr = r - p.nd, b = rr / (sp.gamma + 1), j = rr - b * (sp.gamma + 1);
            has_tok = j < sp.gamma;
            if (has_tok) tok = __ldg(sp.tokens + static_cast<int64_t>(b) * sp.gamma + j);
        }
        tok_out = has_tok && (tok < 0 || tok >= sp.V);
        in_slice = has_tok && !tok_out && tok >= sp.v0 && tok < sp.v0 + sp.Vs;
        g = in_slice ? fmax_nan(logit_at<DT>(slice_row_base(p, r), tok - sp.v0), clamp_floor()) : qnan();
    };
    if (l0 + warp < l1) token(l0 + warp);
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    for (int l = l0 + warp; l < l1; l += kWarpsPerCta) {
        const int r = ra + l;
        const bool drafter = r < p.nd;
        if (l > l0 + warp) token(l);
        // the warps that hold its first and last vector
        const int64_t f = static_cast<int64_t>(l) * RV;
        const int fw = slice_owner(Tc, f), lw = slice_owner(Tc, f + RV - 1);
        const bool on = fw + lane <= lw;
        SoftState a = soft_identity();
        const unsigned char *piece = slots + slice_slot(l, n0, fw + lane) * kSlotBytes;
        if (on) {
            const Partial pt = *reinterpret_cast<const Partial *>(piece);
            a.m = pt.m;
            a.r = pt.r;
            a.t2 = pt.t2;
            a.sh = pt.sh;
            a.sl = pt.sl;
            a.amax = pt.amax;
        }
        for (int off = 1; off <= lw - fw; off <<= 1) a = soft_merge(a, soft_shfl_down(a, off));   // (lane 0: the row)
        const uint64_t *list = reinterpret_cast<const uint64_t *>(piece + sizeof(Partial));
        const int kc = (CAND && !drafter) ? sp.kcap : 0;
        int head = 0, nc = 0;
        uint64_t mine = (on && kc > 0) ? list[0] : 0ull, top = 0ull;   // lane k: the row's k-th key
        for (int k = 0; k < kc; ++k) {
            const uint64_t best = warp_max_u64(mine);
            if (best == 0ull) break;
            ++nc;
            if (lane == k) top = best;
            if (mine == best) mine = (++head < kc) ? list[head] : 0ull;   // (unique keys)
        }
        sdd_shard_partial *rec = sp.out + r;
        if (lane == 0) {
            rec->m = a.m;
            rec->r = a.r;
            rec->t2 = a.t2;
            rec->sh = a.sh;
            rec->sl = a.sl;
            rec->amax = (a.amax == INT32_MAX) ? INT32_MAX : sp.v0 + a.amax;
            rec->g = g;
            rec->info = (in_slice ? 1 : 0) | (tok_out ? 2 : 0) | (nc << 8);
        }
        if (lane < SDD_SHARD_KMAX) {
            rec->cz[lane] = (top != 0ull) ? cand_value(top) : -INFINITY;
            rec->cv[lane] = (top != 0ull) ? cand_index(top) : INT32_MAX;
        }
    }
}

}  // namespace

namespace {

// [bf16][candidates]
void (*const kStream[2][2])(StreamParams) = {{shard_stream_kernel<SDD_F32, false>, shard_stream_kernel<SDD_F32, true>},
                                             {shard_stream_kernel<SDD_BF16, false>, shard_stream_kernel<SDD_BF16, true>}};

size_t stream_smem(int slots) {
    return static_cast<size_t>(kScanSmem) + static_cast<size_t>(slots) * kSlotBytes +
           static_cast<size_t>(kWarpsPerCta) * kCandKeys * sizeof(uint64_t);
}

// The streaming form's launch facts on the current device.
struct StreamDev {
    int clusters, smem;   // clusters of two one-CTA SMs; shared memory of a CTA
};
constexpr int kMaxDevices = 64;
std::atomic<int> g_stream_ready[kMaxDevices];
StreamDev g_stream_dev[kMaxDevices];

cudaError_t stream_device(StreamDev &out) {
    int dev = 0, sms = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    if (!g_stream_ready[dev].load(std::memory_order_acquire)) {
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        for (const auto &row : kStream)
            for (auto k : row)
                if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
        if (e != cudaSuccess) return e;
        g_stream_dev[dev] = StreamDev{sms / 2, optin};
        g_stream_ready[dev].store(1, std::memory_order_release);
    }
    out = g_stream_dev[dev];
    return cudaSuccess;
}

// The clusters of the streaming form for `rows` rows of a slice, and a CTA's
// piece slots; 0 where one CTA per row takes the call: slices of under two
// tiles a row, whose pieces would be mostly their ends; without candidates,
// rows of under kRowFormVec vectors whose CTAs are all resident at once (GB300,
// one CTA per row / streaming, 17 rows: 8,000 bf16 entries 4.0 / 7.2 us, 16,000 5.4
// / 7.0, 24,000 6.8 / 7.0, 38,000 9.6 / 7.0; 1,040 rows 7.7 / 10.1, 10.9 / 12.1, 14.8
// / 14.8, 21.5 / 18.9; 2,080 rows of 8,000 13.8 / 12.4; 17 rows of 12,000 fp32 entries
// 5.9 / 6.2); and batches whose clusters' pieces exceed the shared memory (~900 rows a cluster).  GB300, one
// CTA per row / streaming, bf16 halves with k = 10: 1 x 32 positions of 75,968
// entries 35.0 / 11.8 us, 8 x 32 41.6 / 24.0, 64 x 64 315 / 207; 16 x 32 of
// 4,500 entries 18.0 / 15.8, 1 x 32 13.6 / 11.5.
constexpr int kRowFormVec = 3000;
int stream_plan(const ShardParams &sp, int64_t rows, const StreamDev &dev, int32_t &slots) {
    slots = 0;
    if (dev.clusters < 1 || rows >= (int64_t(1) << 27)) return 0;
    if (sp.RVs < 2 * kTileVec) return 0;
    if (sp.kcap == 0 && rows <= static_cast<int64_t>(2 * kShardMinCtas) * dev.clusters && sp.RVs < kRowFormVec) return 0;
    slots = slice_slots(rows, dev.clusters);
    return stream_smem(slots) <= static_cast<size_t>(dev.smem) ? dev.clusters : 0;
}

}  // namespace

cudaError_t launch_shard_partials(const ShardParams &sp, cudaStream_t stream) {
    const int64_t rows = static_cast<int64_t>(sp.B) * (2 * sp.gamma + 1);
    if (rows == 0) return cudaSuccess;
    const bool bf = sp.dtype == SDD_BF16, cand = sp.kcap > 0;
    StreamDev dev;
    cudaError_t e = stream_device(dev);
    if (e != cudaSuccess) return e;
    StreamParams p;
    const int clusters = stream_plan(sp, rows, dev, p.slots);
    if (clusters > 0) {
        p.sp = sp;
        p.rows = static_cast<int32_t>(rows);
        p.nd = sp.B * sp.gamma;
        get_scan_wait_hooks(p.wait_polls, p.drop_copy);
        return launch_dependent(kStream[bf][cand], dim3(2 * clusters), dim3(kThreads), stream_smem(p.slots), stream, p);
    }
    void (*const k)(ShardParams) = bf ? (cand ? shard_partials_kernel<SDD_BF16, true> : shard_partials_kernel<SDD_BF16, false>)
                                      : (cand ? shard_partials_kernel<SDD_F32, true> : shard_partials_kernel<SDD_F32, false>);
    return launch_dependent(k, dim3(static_cast<unsigned>(rows)), dim3(kShardThreads), 0, stream, sp);
}

}  // namespace sdd
