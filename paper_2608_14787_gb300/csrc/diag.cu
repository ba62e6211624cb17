// diag.cu -- offline diagnostics over logged blocks (scores q [B, gamma] and
// strict accepted lengths L [B] of Strict SDD / shadow-verified rounds):
//
//  * the permutation diagnostic behind Table 1 (Sec. 5, H1 mechanism): at every
//    position j the (score, label) pairs are permuted across the blocks valid
//    there (all blocks; for the conditional signal those with L >= j - 1, j
//    1-based), which keeps every positionwise distribution and breaks the
//    association of positions within a block; the feasible prefix length
//    (Eq. 3's gates, before K_min or staleness) is recomputed per block;
//  * positionwise offline metrics (App. offline metrics): BCE of the scores
//    against the labels 1{L >= j}, the position-only baseline (the positive
//    rate at j), and AUROC (Mann-Whitney, ties count one half).
//
// perm_build_kernel  -- one CTA per (repetition, position): Fisher-Yates over
//                       the valid blocks in shared memory (order-preserving
//                       compaction by ballots; Philox partners drawn in
//                       parallel; the swaps resolved in parallel up to
//                       kPermPar blocks, in order by one thread above); it
//                       writes, for every block, the block whose score it takes.
// perm_prefix_kernel -- one thread per (repetition, block): the gates of Eq. 3
//                       on the permuted scores, position by position until the
//                       local gate fails (the schedule's double-floats, added
//                       one after another where it adds them in a tree: a sum
//                       within their rounding of its threshold, ~2^-43, may
//                       fall on the other side); integer sums per repetition (exact, order-free).
// metrics_kernel     -- one cluster of CTAs per position: fp64 BCE sums, integer
//                       pair counts.
#include <atomic>

#include "rules.cuh"

namespace sdd {
namespace {

constexpr uint32_t kPurposePerm = 3;
// The permutation builder's threads: every phase below is a pass over the n
// valid blocks between two barriers, so with 256 threads a 2,048-block log
// takes 8 elements a thread and phase, and seven CTAs (28 KiB each) share an
// SM.  Bound by issue (72 % of the slots), of which the ten Philox rounds are
// about a third.  GB300, 2,048 blocks x 32 positions x 100 repetitions: 61 us;
// with the chains followed by pointer jumping between barriers 75 us; with 64
// threads a CTA, buckets by a counting sort and the scores gathered here 265 us.
constexpr int kPermThreads = 256;

// Logs of at most this many blocks are shuffled by the parallel construction
// below; longer ones by the serial swap loop.
constexpr int kPermPar = 4096;

// Shared memory of the permutation builder for B logged blocks: the validity
// bits of position j [ceil(B/32) words] and their exclusive prefix popcounts
// [ceil(B/32)]; for B <= kPermPar the parallel construction's arrays (one [B]
// of 32-bit list heads, five [B] of 16-bit indices), above it the block list
// [B] (32-bit).
__host__ __device__ inline size_t perm_smem_bytes(int B) {
    const size_t words = (static_cast<size_t>(B) + 31) / 32;
    const size_t per = (B <= kPermPar) ? sizeof(int32_t) + 5 * sizeof(int16_t) : sizeof(int32_t);
    return 2 * words * sizeof(int32_t) + static_cast<size_t>(B) * per;
}

// pi: [n_rep][gamma][B] 16-bit block indices (B <= 50,000): block b of
// position j takes the score of block pi[r][j][b] in repetition r.
__global__ void __launch_bounds__(kPermThreads) perm_build_kernel(const int32_t *L, int B, int gamma, int conditional,
                                                                  uint64_t seed, uint16_t *pi) {
    extern __shared__ int32_t s_dyn[];
    griddep_wait();
    const int words = (B + 31) / 32;
    uint32_t *s_mask = reinterpret_cast<uint32_t *>(s_dyn);                // validity bits
    int32_t *s_wpre = s_dyn + words;                                       // valid blocks before each word
    int32_t *s_rest = s_wpre + words;
    __shared__ __align__(16) int32_t s_k[kPermThreads];   // swap partners of the current batch of slots
    __shared__ int s_n;
    const int r = blockIdx.x / gamma, j = blockIdx.x % gamma;
    const int tid = threadIdx.x, lane = tid & 31;
    uint16_t *row = pi + (static_cast<int64_t>(r) * gamma + j) * B;
    // validity bits (the loads of several chunks in flight together)
#pragma unroll 4
    for (int c = 0; c < B; c += kPermThreads) {
        const int b = c + tid;
        const bool v = b < B && (!conditional || __ldg(L + b) >= j);
        const unsigned m = __ballot_sync(0xFFFFFFFFu, v);
        if (lane == 0 && b < B) s_mask[b >> 5] = m;   // (b: the warp's first block, a multiple of 32)
    }
    __syncthreads();
    // exclusive prefix popcounts of the words (one warp)
    if (tid < 32) {
        int carry = 0;
        for (int w0 = 0; w0 < words; w0 += 32) {
            const int w = w0 + lane;
            const int c = (w < words) ? __popc(s_mask[w]) : 0;
            int incl = c;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int t = __shfl_up_sync(0xFFFFFFFFu, incl, off);
                if (lane >= off) incl += t;
            }
            if (w < words) s_wpre[w] = carry + incl - c;
            carry += __shfl_sync(0xFFFFFFFFu, incl, 31);
        }
        if (lane == 0) s_n = carry;
    }
    __syncthreads();
    const int n = s_n;
    // the valid blocks in index order (the order defines the draw): block b is
    // the (s_wpre + popcount)-th of them, or the b-th where all are valid
    const bool all = n == B;
    auto rank_of = [&](int b, bool &valid) {
        if (all) {
            valid = true;
            return b;
        }
        const uint32_t m = s_mask[b >> 5], bit = 1u << (b & 31);
        valid = (m & bit) != 0;
        return s_wpre[b >> 5] + __popc(m & (bit - 1u));
    };
    // Fisher-Yates from the top: slot i swaps with k_i = floor(w (i + 1) / 2^32),
    // w the first Philox word of counter (i, j, r, purpose), for i = n-1 .. 1.
    const uint2 key = make_uint2(static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32));
    auto partner = [&](int i) {
        const uint4 o = philox4x32_10(make_uint4(static_cast<uint32_t>(i), static_cast<uint32_t>(j),
                                                 static_cast<uint32_t>(r), kPurposePerm),
                                      key);
        return static_cast<int32_t>((static_cast<uint64_t>(o.x) * static_cast<uint64_t>(i + 1)) >> 32);
    };
    if (B <= kPermPar) {
        // The same permutation without the serial loop.  Step a moves the
        // value then at slot a to slot k_a and fixes slot a.  Let P(s) be the
        // value at slot s just before step s (slot 0: at the end); the last
        // step before a that wrote slot s is the smallest a' > a with
        // k_a' = s, and it wrote P(a').  So, with bucket(s) = {a : k_a = s}:
        //   P(s) = P(min{a' in bucket(s), a' > s}), or the s-th valid block;
        //   final[a] = P(min{a' in bucket(k_a), a' > a}), or the k_a-th;
        //   final[0] = P(0).
        // Each bucket is a linked list in any order (one atomic exchange per
        // step); both minima are taken by walking a bucket, whose length is
        // about ln(n / s), and P follows the "first step above" chains, about
        // as short, to their ends.
        int32_t *s_head = s_rest;                                  // a bucket's first step (0: none; steps are >= 1)
        int16_t *s_list = reinterpret_cast<int16_t *>(s_head + B); // the valid blocks
        int16_t *s_kk = s_list + B;                                // k_a
        int16_t *s_link = s_kk + B;                                // the bucket's next step (0: none)
        int16_t *s_nxt = s_link + B;                               // the bucket's first step above a (0: none)
        int16_t *s_ptr = s_nxt + B;                                // chain links (the slot itself at an end)
        for (int b = tid; b < B; b += kPermThreads) {
            s_head[b] = 0;
            bool valid;
            const int t = rank_of(b, valid);
            if (valid && !all) s_list[t] = static_cast<int16_t>(b);
        }
        __syncthreads();
        for (int a = 1 + tid; a < n; a += kPermThreads) {
            const int k = partner(a);
            s_kk[a] = static_cast<int16_t>(k);
            s_link[a] = static_cast<int16_t>(atomicExch(&s_head[k], a));
        }
        __syncthreads();
        for (int t = tid; t < n; t += kPermThreads) {
            int above = n;   // slot t's chain: it ends at t when no step above t targets t
            for (int u = s_head[t]; u != 0; u = s_link[u])
                if (u > t && u < above) above = u;
            s_ptr[t] = static_cast<int16_t>(above < n ? above : t);
            if (t > 0) {
                int nx = n;
                for (int u = s_head[s_kk[t]]; u != 0; u = s_link[u])
                    if (u > t && u < nx) nx = u;
                s_nxt[t] = static_cast<int16_t>(nx < n ? nx : 0);
            }
        }
        __syncthreads();
        for (int b = tid; b < B; b += kPermThreads) {
            bool valid;
            const int a = rank_of(b, valid);
            int src = b;
            if (valid) {
                // the slot whose first block step a takes: k_a, or the end of
                // the chain of the bucket's next step (of slot 0 itself)
                int u = (a > 0) ? s_nxt[a] : 0;
                if (a > 0 && u == 0) {
                    u = s_kk[a];
                } else {
                    for (int v = s_ptr[u]; v != u; v = s_ptr[u]) u = v;
                }
                src = all ? u : s_list[u];
            }
            row[b] = static_cast<uint16_t>(src);
        }
        return;
    }
    // serial: the partners of kPermThreads slots drawn in parallel, the swaps
    // then in order
    int32_t *s_list = s_rest;
    for (int b = tid; b < B; b += kPermThreads) {
        bool valid;
        const int t = rank_of(b, valid);
        if (valid) s_list[t] = b;
    }
    __syncthreads();
    for (int top = n - 1; top > 0; top -= kPermThreads) {
        const int i = top - tid;
        if (i > 0) s_k[tid] = partner(i);
        __syncthreads();
        if (tid == 0) {
            // slots top, top - 1, ..., top - cnt + 1 (all > 0); x carries the
            // value at slot a, re-read after each swap (which may have written
            // slot a - 1), so one shared-memory round trip bounds an iteration;
            // the partners come four at a time
            const int cnt = min(kPermThreads, top);
            int32_t x = s_list[top];
            for (int u = 0; u < cnt; u += 4) {
                const int4 kk = *reinterpret_cast<const int4 *>(s_k + u);
                const int ks[4] = {kk.x, kk.y, kk.z, kk.w};
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    if (u + h >= cnt) break;
                    const int a = top - u - h, k = ks[h];
                    const int32_t y = (k == a) ? x : s_list[k];
                    s_list[k] = x;
                    s_list[a] = y;
                    x = s_list[a - 1];
                }
            }
        }
        __syncthreads();
    }
    for (int b = tid; b < B; b += kPermThreads) {
        bool valid;
        const int a = rank_of(b, valid);
        row[b] = static_cast<uint16_t>(valid ? s_list[a] : b);
    }
}

// Grid: ceil(B / kPrefixThreads) CTAs for each of n_rep + 1 repetitions, the
// last of which is the logged order.  Neighbouring threads are neighbouring blocks, so a repetition's
// indices are read in whole lines, and a score is gathered only while the
// block's local gate holds; the positions go in groups of kPrefixU whose
// loads are in flight together, the indices of a group loaded beside the scores
// of the one before.  Bound by the gathers' latency.  GB300, 2,048 x 32 x 100:
// 20 us; with a warp per (repetition, block), its lanes on scores 4 B bytes
// apart, 112 us.  The whole diagnostic of 512 blocks, groups of 2 / 4 / 8:
// 31.0 / 31.1 / 31.7 us; with a group's indices loaded before its scores, 4: 33.0.
constexpr int kPrefixThreads = 256;
constexpr int kPrefixU = 2;
__global__ void __launch_bounds__(kPrefixThreads) perm_prefix_kernel(const float *q, const uint16_t *pi, int B,
                                                                     int gamma, int n_rep, int signal, df eta_loc,
                                                                     df log_eta_c, unsigned long long *sums) {
    griddep_wait();
    const int per = (B + kPrefixThreads - 1) / kPrefixThreads;
    const int r = blockIdx.x / per, b = static_cast<int>(blockIdx.x % per) * kPrefixThreads + threadIdx.x;
    int Kh = 0;
    if (b < B) {
        const uint16_t *row = pi + static_cast<int64_t>(r) * gamma * B + b;
        int kb = 0, best = 0;   // leading positions passing the local gate; the largest prefix meeting Eq. 3
        bool open = true;
        df S = df{0.f, 0.f};
        int src[kPrefixU];   // the group's source blocks, loaded a group ahead
        auto load_src = [&](int j0) {
#pragma unroll
            for (int u = 0; u < kPrefixU; ++u)
                src[u] = (r < n_rep && j0 + u < gamma) ? __ldg(row + static_cast<int64_t>(j0 + u) * B) : b;
        };
        load_src(0);
        for (int j0 = 0; j0 < gamma && open; j0 += kPrefixU) {
            float qj[kPrefixU];
#pragma unroll
            for (int u = 0; u < kPrefixU; ++u)
                qj[u] = (j0 + u < gamma) ? __ldg(q + static_cast<int64_t>(src[u]) * gamma + j0 + u) : qnan();
            load_src(j0 + kPrefixU);
#pragma unroll
            for (int u = 0; u < kPrefixU; ++u) {
                // (past gamma: NaN closes the gate)
                open = open && isfinite(qj[u]) && df_ge(df{qj[u], 0.f}, eta_loc);
                if (!open) continue;
                kb = j0 + u + 1;
                if (signal == SDD_SIG_MARGINAL) continue;
                S = df_add(S, df{logf(qj[u]), 0.f});
                const bool pass = (signal == SDD_SIG_RAW) ? df_ge(S, df_mul_f(log_eta_c, static_cast<float>(kb)))
                                                          : df_ge(S, log_eta_c);
                if (pass) best = kb;
            }
        }
        Kh = (signal == SDD_SIG_MARGINAL) ? kb : best;
    }
    Kh = __reduce_add_sync(0xFFFFFFFFu, Kh);
    if ((threadIdx.x & 31) == 0 && Kh > 0) atomicAdd(sums + r, static_cast<unsigned long long>(Kh));
}

// Positionwise metrics.  The pair counts of the AUROC are what costs: a
// position of a log of B blocks has up to B^2 / 4 (positive, negative) pairs.
// A cluster of kMetCluster CTAs takes a position; CTA c takes the blocks of
// its c-th part of the log as the positives (and their BCE terms: fp64
// logarithms, which issue slowly here, so they too are spread over the SMs)
// against every negative of the log.  The positives are compacted into shared
// memory and sorted there, a tile at a time, and each negative finds the
// numbers of positives below and at it by bisection.  Sums meet in CTA 0 by
// distributed shared memory and are added in rank order, so the results are
// deterministic.  Bound by the chain of staging, sort, fp64 logarithms and the
// cluster's sums.  GB300, 2,048 x 32: 22.6 us (4.0 M warp instructions); 30 us
// (9.3 M) with every pair compared, positives in registers against negatives in
// shared memory; 24.1 us with a thread's bisections one after another.
constexpr int kMetThreads = 256;
constexpr int kMetCluster = 8;
constexpr int kMetPos = 1024;    // positives of a tile (a power of two)
constexpr int kMetU = 4;         // blocks a thread loads together
struct MetSums {
    double bce;
    unsigned long long np, nn, gt, eq;
};

__device__ __forceinline__ void st_cluster_u64(uint32_t addr, unsigned long long v) {
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}

// The scores of the positives (valid, L >= j + 1; NaN counts in no pair) of
// blocks [b0, b1) compacted into dst, in any order; *s_cnt receives their number.
__device__ __forceinline__ void met_stage(const float *q, const int32_t *L, int gamma, int j, int conditional, int b0,
                                          int b1, float *dst, int *s_cnt) {
    __syncthreads();   // the previous tile has been read
    if (threadIdx.x == 0) *s_cnt = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int c = b0; c < b1; c += kMetU * kMetThreads) {
        int l[kMetU];
        float x[kMetU];
#pragma unroll
        for (int u = 0; u < kMetU; ++u) {
            const int b = c + u * kMetThreads + static_cast<int>(threadIdx.x);
            l[u] = (b < b1) ? __ldg(L + b) : 0;
            x[u] = (b < b1) ? __ldg(q + static_cast<int64_t>(b) * gamma + j) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < kMetU; ++u) {
            const int b = c + u * kMetThreads + static_cast<int>(threadIdx.x);
            const bool in = b < b1 && !(conditional && l[u] < j) && l[u] >= j + 1 && x[u] == x[u];
            const unsigned m = __ballot_sync(0xFFFFFFFFu, in);
            int at = 0;
            if (lane == 0 && m) at = atomicAdd(s_cnt, __popc(m));
            at = __shfl_sync(0xFFFFFFFFu, at, 0);
            if (in) dst[at + __popc(m & ((1u << lane) - 1u))] = x[u];
        }
    }
    __syncthreads();
}

// a[0, n) ascending, n a power of two: bitonic, a pair per thread and step.  A
// step of stride s <= 32 stays within the 64 entries that its warp's 32 pairs
// cover, so only strides above need the CTA's barrier.
__device__ __forceinline__ void met_sort(float *a, int n) {
    for (int k = 2; k <= n; k <<= 1) {
        for (int s = k >> 1; s > 0; s >>= 1) {
            for (int t = threadIdx.x; t < (n >> 1); t += kMetThreads) {
                const int i = ((t & ~(s - 1)) << 1) | (t & (s - 1));
                const float x = a[i], y = a[i + s];
                if ((x > y) == ((i & k) == 0)) {
                    a[i] = y;
                    a[i + s] = x;
                }
            }
            // the next step's stride: s / 2, or k (of the next k) behind s = 1
            if (s > 32 || (s == 1 && k > 32))
                __syncthreads();
            else
                __syncwarp();
        }
    }
    __syncthreads();
}

// How many of the n ascending entries (n a power of two) are below each v (or,
// with EQ, at most v); the U bisections step together.  (NaN: 0.)
template <bool EQ, int U>
__device__ __forceinline__ void met_rank(const float *a, int n, const float (&v)[U], int (&at)[U]) {
#pragma unroll
    for (int u = 0; u < U; ++u) at[u] = 0;
    for (int s = n >> 1; s > 0; s >>= 1)
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float x = a[at[u] + s - 1];
            if (EQ ? x <= v[u] : x < v[u]) at[u] += s;
        }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const float x = a[at[u]];   // (at <= n - 1)
        at[u] += (EQ ? x <= v[u] : x < v[u]) ? 1 : 0;
    }
}

__global__ void __cluster_dims__(kMetCluster, 1, 1) __launch_bounds__(kMetThreads)
    metrics_kernel(const float *q, const int32_t *L, int B, int gamma, int conditional, double *bce, double *bce_base,
                   double *auroc, int32_t *n_pos, int32_t *n_neg) {
    // (CTA 0 has started before the others write to its shared memory: the wait
    // for this arrival is ahead of those writes)
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    griddep_wait();
    const int j = blockIdx.x / kMetCluster, rank = blockIdx.x % kMetCluster;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ float s_pos[kMetPos];
    __shared__ int s_np;
    __shared__ MetSums s_w[kMetThreads / 32];
    __shared__ MetSums s_all[kMetCluster];   // (CTA 0)
    const int part = (B + kMetCluster - 1) / kMetCluster;
    const int p0 = min(B, rank * part), p1 = min(B, p0 + part);
    MetSums a{0.0, 0, 0, 0, 0};
    for (int b = p0 + tid; b < p1; b += kMetThreads) {
        const int l = __ldg(L + b);
        if (conditional && l < j) continue;
        const bool y = l >= j + 1;
        const double qc = fmin(fmax(static_cast<double>(__ldg(q + static_cast<int64_t>(b) * gamma + j)), 1e-7),
                               1.0 - 1e-7);
        // one fp64 logarithm for both classes: 1 - qc = h + l exactly, and
        // ln(h + l) = ln h + l / h to (l / h)^2 < 2^-104
        const double h = 1.0 - qc, l2 = (1.0 - h) - qc;
        const double corr = static_cast<double>(static_cast<float>(l2) / static_cast<float>(h));
        a.bce -= log(y ? qc : h) + (y ? 0.0 : corr);
        a.np += y ? 1 : 0;
        a.nn += y ? 0 : 1;
    }
    for (int c = p0; c < p1; c += kMetPos) {
        met_stage(q, L, gamma, j, conditional, c, min(p1, c + kMetPos), s_pos, &s_np);
        const int P = s_np;
        if (P == 0) continue;
        int n = 1;   // sorted with infinities behind the P positives
        while (n < P) n <<= 1;
        for (int t = P + tid; t < n; t += kMetThreads) s_pos[t] = INFINITY;
        __syncthreads();
        met_sort(s_pos, n);
        for (int b0 = tid; b0 < B; b0 += kMetU * kMetThreads) {
            int l[kMetU], lt[kMetU];
            float x[kMetU];
#pragma unroll
            for (int u = 0; u < kMetU; ++u) {
                const int b = b0 + u * kMetThreads;
                l[u] = (b < B) ? __ldg(L + b) : INT32_MAX;
                x[u] = (b < B) ? __ldg(q + static_cast<int64_t>(b) * gamma + j) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < kMetU; ++u)   // valid negatives; NaN counts in no pair
                if (l[u] >= j + 1 || (conditional && l[u] < j)) x[u] = qnan();
            met_rank<false>(s_pos, n, x, lt);
#pragma unroll
            for (int u = 0; u < kMetU; ++u) {
                if (!(x[u] == x[u])) continue;
                const int below = min(P, lt[u]);
                int le[1] = {below};
                if (below < P && s_pos[below] == x[u]) {
                    const float v[1] = {x[u]};
                    met_rank<true>(s_pos, n, v, le);
                    le[0] = min(P, le[0]);
                }
                a.gt += static_cast<unsigned>(P - le[0]);
                a.eq += static_cast<unsigned>(le[0] - below);
            }
        }
    }
    // fixed-order sums: lanes, warps, CTAs
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        a.bce += __shfl_down_sync(0xFFFFFFFFu, a.bce, off);
        a.np += __shfl_down_sync(0xFFFFFFFFu, a.np, off);
        a.nn += __shfl_down_sync(0xFFFFFFFFu, a.nn, off);
        a.gt += __shfl_down_sync(0xFFFFFFFFu, a.gt, off);
        a.eq += __shfl_down_sync(0xFFFFFFFFu, a.eq, off);
    }
    if (lane == 0) s_w[warp] = a;
    __syncthreads();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (tid == 0) {
#pragma unroll
        for (int w = 1; w < kMetThreads / 32; ++w) {
            a.bce += s_w[w].bce;
            a.np += s_w[w].np;
            a.nn += s_w[w].nn;
            a.gt += s_w[w].gt;
            a.eq += s_w[w].eq;
        }
        uint32_t dst;
        asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(dst) : "r"(smem_addr(&s_all[rank])));
        st_cluster_u64(dst, static_cast<unsigned long long>(__double_as_longlong(a.bce)));
        st_cluster_u64(dst + 8, a.np);
        st_cluster_u64(dst + 16, a.nn);
        st_cluster_u64(dst + 24, a.gt);
        st_cluster_u64(dst + 32, a.eq);
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (rank == 0 && lane == 0 && warp < 3) {
        // (a warp for each result: their fp64 chains run side by side)
        MetSums t = s_all[0];
#pragma unroll
        for (int c = 1; c < kMetCluster; ++c) {
            t.bce += s_all[c].bce;
            t.np += s_all[c].np;
            t.nn += s_all[c].nn;
            t.gt += s_all[c].gt;
            t.eq += s_all[c].eq;
        }
        const double P = static_cast<double>(t.np), N = static_cast<double>(t.nn), n = P + N;
        const double nan = __longlong_as_double(0x7FF8000000000000ll);
        if (warp == 0) {
            bce[j] = (n > 0) ? t.bce / n : nan;
            if (n_pos) n_pos[j] = static_cast<int32_t>(t.np);
            if (n_neg) n_neg[j] = static_cast<int32_t>(t.nn);
        } else if (warp == 1) {
            const double pr = (n > 0) ? P / n : nan;
            bce_base[j] = (n > 0) ? ((pr > 0.0 && pr < 1.0) ? -(pr * log(pr) + (1.0 - pr) * log1p(-pr)) : 0.0) : nan;
        } else {
            auroc[j] =
                (P > 0 && N > 0) ? (static_cast<double>(t.gt) + 0.5 * static_cast<double>(t.eq)) / (P * N) : nan;
        }
    }
}

constexpr int kMaxDevices = 64;
std::atomic<int> g_perm_ready[kMaxDevices];

// Per-device opt-in of the builder to all the dynamic shared memory that its
// static part leaves, once: the limit of 48 KiB without it is on the two
// together, and a limit set for one call's log would be another thread's too.
cudaError_t perm_prepare() {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    if (g_perm_ready[dev].load(std::memory_order_acquire)) return cudaSuccess;
    cudaFuncAttributes attr;
    e = cudaFuncGetAttributes(&attr, perm_build_kernel);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(perm_build_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 optin - static_cast<int>(attr.sharedSizeBytes));
    if (e == cudaSuccess) g_perm_ready[dev].store(1, std::memory_order_release);
    return e;
}

}  // namespace

cudaError_t launch_perm_diag(const float *q, const int32_t *L, int B, int gamma, int signal, df eta_loc,
                             df log_eta_c, int n_rep, uint64_t seed, uint16_t *pi, unsigned long long *sums,
                             cudaStream_t stream) {
    cudaError_t e = cudaMemsetAsync(sums, 0, sizeof(unsigned long long) * (n_rep + 1), stream);
    if (e != cudaSuccess) return e;
    const size_t smem = perm_smem_bytes(B);
    if (n_rep > 0) {
        e = perm_prepare();
        if (e != cudaSuccess) return e;
        e = launch_dependent(perm_build_kernel, dim3(n_rep * gamma), dim3(kPermThreads), smem, stream, L, B, gamma,
                             signal == SDD_SIG_CONDITIONAL ? 1 : 0, seed, pi);
        if (e != cudaSuccess) return e;
    }
    const int per = (B + kPrefixThreads - 1) / kPrefixThreads;
    return launch_dependent(perm_prefix_kernel,
                            dim3(static_cast<unsigned>(per) * static_cast<unsigned>(n_rep + 1)), dim3(kPrefixThreads), 0,
                            stream, q, pi, B, gamma, n_rep, signal, eta_loc, log_eta_c, sums);
}

cudaError_t launch_position_metrics(const float *q, const int32_t *L, int B, int gamma, int conditional, double *bce,
                                    double *bce_base, double *auroc, int32_t *n_pos, int32_t *n_neg,
                                    cudaStream_t stream) {
    return launch_dependent(metrics_kernel, dim3(gamma * kMetCluster), dim3(kMetThreads), 0, stream, q, L, B, gamma,
                            conditional, bce, bce_base, auroc, n_pos, n_neg);
}

}  // namespace sdd
