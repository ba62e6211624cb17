// mlp.cu -- the learned-scorer stand-ins of the decode-loop workload on the
// 5th-generation tensor cores (App. A.7's form, random weights):
//
//   one layer:  s[m] = sigmoid(w2 . GELU(W1 h[m] + b1) + b2),
//   deep:       a1 = bf16(GELU(W1 [h ; f] + b1)), a2 = bf16(GELU(W2 a1 + b2)),
//               s[m] = sigmoid(w4 . GELU(W3 a2 + b3) + b4),
//   GELU(z) = z Phi(z) (erf form), fp32 accumulation throughout,
//
// and the scalar-feature block f of the deep scorer's input.
//
// As many 128-row tiles as clusters of four fit the SMs (a decode round's batch):
// first layer (mlp_kernel): a cluster of S = 4 CTAs per 128-row tile splits K;
// each CTA streams its K quarter through a four-stage ring of 48 KiB (A tile
// 128 x 64, B tile 256 x 64, K-major, 128-byte swizzle) filled by 2D TMA, one
// thread issues tcgen05.mma.kind::f16 (M = 128, N = 256, K = 16) into a
// 256-column TMEM accumulator; the partial accumulators meet through an L2
// workspace (stores, one cluster barrier, loads) and CTA q finishes
// output columns [64 q, 64 q + 64) with the fused epilogue.
// Layers 2-3 of the deep scorer (mlp_tail_kernel): a cluster of four CTAs per
// tile, each computing 64 output columns of both layers, a2 through the
// workspace and back by TMA.
// Larger batches (mlp_plan): whole waves of one tile per SM run unsplit
// (mlp_kernel with S = 1; the deep scorer all layers in one CTA,
// mlp_deep_kernel), the tiles left over as above with S = 4 or 2.  However its
// tile is run, a row's sum over K is taken in the same chains (kMlpChains).
#include <cuda.h>
#include <cudaTypedefs.h>

#include <atomic>
#include <mutex>

#include "internal.h"

namespace sdd {
namespace {

constexpr int kMlpN = 256;           // hidden units = UMMA N
constexpr int kMlpBM = 128;          // rows per CTA = UMMA M
constexpr int kMlpBK = 64;           // K per stage: 64 bf16 = one 128-byte swizzle row
constexpr int kMlpStages = 4;
// Warps 0-15: epilogue.  The TMA producer is lane 0 of warp kRole, the MMA
// issuer lane 0 of the next: epilogue warps, or warps of their own where the
// epilogue warps read finished chains (kMlpChains) beside the main loop.
constexpr int kMlpThreads = 512, kMlpThreadsChains = kMlpThreads + 64;
constexpr uint32_t kATileBytes = kMlpBM * kMlpBK * 2;   // 16 KiB
constexpr uint32_t kBTileBytes = kMlpN * kMlpBK * 2;    // 32 KiB
constexpr uint32_t kStageBytes = kATileBytes + kBTileBytes;
constexpr int kMlpSmem = kMlpStages * kStageBytes + 1024 + 256;   // + alignment slack + barriers
constexpr uint32_t kTmemCols = 256;
// A tile's sum over K is taken in this many chains (quarters of K), each
// accumulated by the tensor cores from zero, added in fp32 in their order: a
// CTA of S splits takes kMlpChains / S of them.  The tensor cores' fp32
// accumulation loses about in proportion to a chain's length: error of the
// scores against 64 bits (2-norm), K = 3584: one chain 3.9e-7, two 1.9e-7, four
// 0.98e-7; K = 2048: 2.2e-7, 1.1e-7, 0.66e-7.  Four against one chain cost
// (S = 1) 28.0 against 27.4 us at 12,000 rows, 33.1 / 32.9 at 16,384, 35.4 /
// 35.4 at 19,456, and two against one (S = 2) 20.4 / 20.1 at 8,192.
// Under eight slices of K two chains or one, as measured there (K = 448: one
// chain 0.64e-7 and 10.0 us at 19,456 rows, four 0.48e-7 and 11.1).
constexpr int kMlpChains = 4;
__host__ __device__ constexpr int mlp_chains(int slices) {
    return slices >= 2 * kMlpChains ? kMlpChains : (slices >= kMlpChains && slices % 2 == 0) ? 2 : 1;
}

struct MlpParams {
    int32_t M, K;
    int32_t Ka;             // K columns of the first A operand (the rest come from the second)
    const float *b1;        // [256]
    const uint16_t *w2;     // [256] bf16 bits (head mode)
    float b2;
    float *out;             // [M] (head mode)
    uint16_t *act;          // [M, 256] bf16 bits: GELU(W1 x + b1) (activation mode)
    float *ws;              // [tiles][S][256][128] fp32: partial accumulators (column-major per source CTA)
    int32_t *status;
    int32_t tile0;          // the launch's first tile
};

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int c0, int c1, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
        : "memory");
}

// Shared-memory matrix descriptor of a K-major operand tile with the 128-byte
// swizzle: rows of 128 bytes, 8-row core groups 1024 bytes apart (SBO); the
// leading-dimension offset is unused for this layout; descriptor version 1.
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t addr) {
    uint64_t d = static_cast<uint64_t>((addr >> 4) & 0x3FFFu);
    d |= static_cast<uint64_t>(1) << 16;                // LBO (unused): 16 bytes
    d |= static_cast<uint64_t>(1024 >> 4) << 32;        // SBO: 1024 bytes
    d |= static_cast<uint64_t>(1) << 46;                // version
    d |= static_cast<uint64_t>(2) << 61;                // 128-byte swizzle
    return d;
}

// Instruction descriptor of kind::f16: fp32 D, bf16 A and B, both K-major, N, M = 128.
__host__ __device__ constexpr uint32_t idesc_f16(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(n >> 3) << 17) |
           (static_cast<uint32_t>(kMlpBM >> 4) << 24);
}

template <int N = kMlpN>
__device__ __forceinline__ void umma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc_f16(N)), "r"(accumulate)
        : "memory");
}

// Arrive on `bar` once every tcgen05 operation this thread issued so far completes.
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 16 consecutive fp32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// 16 consecutive fp32 columns into this thread's TMEM lane.
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float *v) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
        "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]), "f"(v[9]),
        "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15])
        : "memory");
}
// 16 columns of this thread's TMEM lane, or zeros when the accumulator is not valid.
__device__ __forceinline__ void tmem_ld16_or0(bool ok, uint32_t taddr, uint32_t (&v)[16]) {
    if (ok) {
        tmem_ld16(taddr, v);
    } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = 0u;
    }
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Address of the same shared-memory location in cluster CTA `rank`.
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// Orders this thread's generic-proxy global stores before later async-proxy
// (TMA) reads of them, by any thread that synchronises with this one.
__device__ __forceinline__ void fence_proxy_async_global() {
    asm volatile("fence.proxy.async.global;" ::: "memory");
}

__device__ __forceinline__ void st_cluster_f32(uint32_t addr, float a) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(a) : "memory");
}

// Two fp32 values rounded to bf16 (round to nearest even), packed (a low).
__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
    uint32_t d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
    return d;
}

__device__ __forceinline__ float gelu_erf(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }

// The first layer's main loop over K slices [kt0, kt0 + nk) of the tile at row
// m0, in C chains (chain c: slices [c nk / C, (c + 1) nk / C), into the 256 TMEM
// columns at tmem + 256 (c & 1)).  Warp ROLE lane 0 fills the ring, the next
// warp's lane 0 issues the products; done[c] completes with chain c, and chain
// c >= 2 starts once drained[c - 2] says that its columns have been read.  The
// ring is idle when both lanes have left (once the last chain has completed).
template <int ROLE>
__device__ __forceinline__ void mlp_mainloop(unsigned char *smem, uint64_t *full, uint64_t *empty, uint64_t *done,
                                             uint64_t *drained, const CUtensorMap *tmA, const CUtensorMap *tmA2,
                                             const CUtensorMap *tmB, int Ka, int m0, int kt0, int nk, int C,
                                             uint32_t tmem, int *s_abort) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == ROLE && lane == 0) {
        // TMA producer: stage s holds K slice kt0 + t of the A tile (rows
        // m0..m0+127) and of the B tile (all 256 hidden units)
        int t = 0;
        for (; t < nk; ++t) {
            const int s = t % kMlpStages;
            const uint32_t ph = static_cast<uint32_t>(t / kMlpStages) & 1u;
            if (t >= kMlpStages && !mbar_wait_bounded(&empty[s], ph ^ 1u, kWaitPolls)) {
                *s_abort = 1;
                break;
            }
            mbar_arrive_expect_tx(&full[s], kStageBytes);
            const uint32_t a = smem_addr(smem + s * kStageBytes);
            const int k = (kt0 + t) * kMlpBK;
            if (k < Ka)
                tma_load_2d(a, tmA, k, m0, smem_addr(&full[s]));
            else
                tma_load_2d(a, tmA2, k - Ka, m0, smem_addr(&full[s]));
            tma_load_2d(a + kATileBytes, tmB, k, 0, smem_addr(&full[s]));
        }
        // let every issued load land before the ring is reused or the CTA
        // leaves (already true unless a wait gave up): the last load per stage
        for (int s = 0; s < kMlpStages && s < t; ++s) {
            const int last = ((t - 1 - s) / kMlpStages) * kMlpStages + s;
            (void)mbar_wait_bounded(&full[s], static_cast<uint32_t>(last / kMlpStages) & 1u, kWaitPolls);
        }
    } else if (warp == ROLE + 1 && lane == 0) {
        // MMA issuer: four K = 16 steps per stage, the 128-byte rows advanced
        // by 32 bytes per step
        bool ok = true;
        int t = 0;
        for (int c = 0; c < C; ++c) {
            const int first = t, end = (c + 1) * nk / C;
            const uint32_t d = tmem + (c & 1) * kTmemCols;
            if (ok && c >= 2) {
                ok = mbar_wait_bounded(&drained[c - 2], 0u, kWaitPolls);
                tc_fence_after();
            }
            for (; ok && t < end; ++t) {
                const int s = t % kMlpStages;
                const uint32_t ph = static_cast<uint32_t>(t / kMlpStages) & 1u;
                if (!mbar_wait_bounded(&full[s], ph, kWaitPolls)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t a = smem_addr(smem + s * kStageBytes), b = a + kATileBytes;
#pragma unroll
                for (int kk = 0; kk < kMlpBK / 16; ++kk)
                    umma_f16(d, umma_desc_sw128(a + kk * 32), umma_desc_sw128(b + kk * 32),
                             (t != first || kk != 0) ? 1u : 0u);
                umma_commit(smem_addr(&empty[s]));   // the stage is free once these MMAs have read it
            }
            umma_commit(smem_addr(&done[c]));        // the chain is complete (at once when nothing was issued)
        }
        if (!ok) *s_abort = 1;
    }
}

// The chains of a CTA that takes the whole of K, added in order by the epilogue
// warps while the later ones run: warp w its 32 TMEM lanes (tlane) and columns
// [64 (w / 4), + 64), the sum left in the first 256 columns.  Every warp of the
// CTA calls it; epi: the epilogue warps.  False when a wait gave up.
__device__ __forceinline__ bool mlp_drain(uint64_t *done, uint64_t *drained, int C, bool epi, uint32_t tlane, int part) {
    bool ok = true;
    float acc[64];
#pragma unroll
    for (int j = 0; j < 64; ++j) acc[j] = 0.f;
#pragma unroll 1
    for (int c = 0; c < C && ok; ++c) {
        ok = __all_sync(0xFFFFFFFFu, mbar_wait_bounded(&done[c], 0u, kWaitPolls));
        tc_fence_after();
        if (!ok || !epi || C == 1) continue;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t v[16];
            tmem_ld16(tlane + (c & 1) * kTmemCols + part * 64 + 16 * q, v);
#pragma unroll
            for (int j = 0; j < 16; ++j) acc[16 * q + j] += __uint_as_float(v[j]);
        }
        if (c + 2 < C) {   // a later chain takes these columns
            tc_fence_before();
            __syncwarp();
            if ((threadIdx.x & 31) == 0) mbar_arrive(&drained[c]);
        }
    }
    if (ok && epi && C > 1) {
#pragma unroll
        for (int q = 0; q < 4; ++q) tmem_st16(tlane + part * 64 + 16 * q, acc + 16 * q);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    return ok;
}

// Grid: (M tiles x S) CTAs in clusters of S along x (S = 1, 2 or 4 splits of
// K).  CTA rank r of a cluster multiplies K slices [r nk/S, (r+1) nk/S) of its
// 128-row tile into its own TMEM.  Columns [q W, (q+1) W) of the tile (W =
// 256/S) are finished by CTA q: every CTA stores the other columns of its
// partial to the workspace (L2; distributed shared memory moves these 96 KiB
// per CTA several times slower), a cluster barrier orders the stores before
// the loads, and each CTA sums the S partials of its columns in rank order
// (its own from TMEM) and runs the epilogue.  A thread's loads of the other
// partials (48 with S = 4, a warp's each 128 contiguous bytes) are in flight
// together, straight to registers: GB300, 4,096 x 3,584, 13.85 us per call
// against 14.47 with the partials brought into the idle ring by bulk copies
// (one more round trip and pass through shared memory; 14.2-14.3 with that
// form's tighter epilogue).  What bounds it: the main loop's bytes (5.7 us of
// it, 31 MB), then the chain of the exchange and the GELUs.
//
// The A operand is the concatenation [A1 | A2] along K: slices below p.Ka come
// from tmA, the rest from tmA2 (the scalar features of the deep scorer).
// HEAD: the epilogue fuses GELU, the w2 dot product and the sigmoid (one
// float per row); otherwise it writes the layer's activations GELU(z + b1)
// as bf16 rows of p.act for the next layer (S > 1: whole tiles of the deep
// scorer are mlp_deep_kernel's).
// The CTA's K is taken in 4 / S chains (as its slices allow): S = 2 adds its two
// where it reads them, S = 1 its four beside the main loop (mlp_drain).
__host__ __device__ constexpr int mlp_threads(int S) { return S == 1 ? kMlpThreadsChains : kMlpThreads; }
template <int S, bool HEAD>
__global__ void __launch_bounds__(mlp_threads(S), 1) mlp_kernel(const __grid_constant__ CUtensorMap tmA,
                                                            const __grid_constant__ CUtensorMap tmA2,
                                                            const __grid_constant__ CUtensorMap tmB,
                                                            const __grid_constant__ MlpParams p) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                            ~static_cast<uintptr_t>(1023));
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + kMlpStages * kStageBytes);
    uint64_t *empty = full + kMlpStages;
    uint64_t *done = empty + kMlpStages;      // a barrier a chain
    uint64_t *drained = done + kMlpChains;    // [kMlpChains - 2]
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(drained + kMlpChains - 2);
    constexpr int kRole = S == 1 ? kMlpThreads / 32 : 0;
    constexpr uint32_t kCols = S < kMlpChains ? 2 * kTmemCols : kTmemCols;
    __shared__ int s_abort;
    __shared__ float s_b1[kMlpN], s_w2[kMlpN];   // epilogue constants, widened once per CTA
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = (S > 1) ? cluster_rank() : 0u;
    const int m0 = (p.tile0 + static_cast<int>(blockIdx.x) / S) * kMlpBM;
    const int slices = p.K / kMlpBK;
    const int kt0 = static_cast<int>(rank) * slices / S;                // K slices of this CTA
    const int nk = (static_cast<int>(rank) + 1) * slices / S - kt0;
    const int C = max(mlp_chains(slices) / S, 1);

    if (tid == 0) {
        for (int i = 0; i < 2 * kMlpStages + kMlpChains; ++i) mbar_init(&full[i], 1);
        for (int i = 0; i < kMlpChains - 2; ++i) mbar_init(&drained[i], kMlpThreads / 32);
        fence_mbar_init();
        s_abort = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                     "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // launched as a programmatic dependent: the setup above overlaps the end
    // of the work ahead in the stream; nothing is read before that completes
    // (earlier grids' writes are visible only behind this grid's own wait: the
    // launch ahead having waited for them promises nothing here)
    griddep_wait();
    for (int n = tid; n < kMlpN; n += mlp_threads(S)) {
        s_b1[n] = __ldg(p.b1 + n);
        s_w2[n] = HEAD ? __uint_as_float(static_cast<uint32_t>(__ldg(p.w2 + n)) << 16) : 0.f;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    mlp_mainloop<kRole>(smem, full, empty, done, drained, &tmA, &tmA2, &tmB, p.Ka, m0, kt0, nk, C, tmem, &s_abort);
    __syncwarp();

    // Exchange through the workspace.  CTA q of the cluster finishes the
    // column block [q W, (q + 1) W) (W = 256 / S) of all 128 rows: its own
    // partial of the block stays in its TMEM, every other column of its
    // partial goes to ws[tile][q][column][row] (a warp's 32 rows of one column
    // are 128 contiguous bytes), from where the owner of the column loads it.
    // Warp w reads TMEM lanes 32 (w % 4) .. + 31 (tile rows); the four warps
    // of a lane quarter share the columns in 16-column chunks.
    constexpr int W = kMlpN / S;
    const int quarter = warp & 3, part = warp >> 2;   // (part 4: the producer's and the issuer's warps of S = 1)
    const bool epi = warp < kMlpThreads / 32;
    const int row = quarter * 32 + lane;
    const uint32_t tbase = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
    bool ok;
    if (S == 1) {
        ok = mlp_drain(done, drained, C, epi, tbase, part);
    } else {   // (the last chain's products end after the first's)
        ok = __all_sync(0xFFFFFFFFu, mbar_wait_bounded(&done[C - 1], 0u, kWaitPolls));
        tc_fence_after();
    }
    // 16 columns of this CTA's sum
    auto own16 = [&](int c, uint32_t (&v)[16]) {
        tmem_ld16_or0(ok, tbase + c, v);
        if (S == 2 && C == 2) {
            uint32_t w[16];
            tmem_ld16_or0(ok, tbase + kTmemCols + c, w);
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) + __uint_as_float(w[j]));
        }
    };
    if (!ok) s_abort = 1;
    griddep_launch_dependents();   // the next launch may set up (it still waits for this grid)
    float *ws_tile = p.ws + static_cast<int64_t>(blockIdx.x / S) * S * kMlpN * kMlpBM;
    if (S > 1) {
        float *mine = ws_tile + static_cast<int64_t>(rank) * kMlpN * kMlpBM;
        int idx = 0;   // remote chunks in column order, round robin over the quarter's four warps
#pragma unroll 1
        for (int c = 0; c < kMlpN; c += 16) {
            if (c / W == static_cast<int>(rank)) continue;
            if ((idx++ & 3) != part) continue;
            uint32_t v[16];
            own16(c, v);
#pragma unroll
            for (int j = 0; j < 16; ++j) __stcg(mine + (c + j) * kMlpBM + row, __uint_as_float(v[j]));
        }
        cluster_sync();               // every partial of the tile is in the workspace (release / acquire)
    }

    // epilogue: z = the partials summed in rank order, then bias and GELU;
    // this warp's columns [rank W + part W / 4, + W / 4) of its 32 rows
    const int grow = m0 + row;
    float t2 = 0.f;   // HEAD: this thread's part of the w2 dot product, a sum of 16 columns at a time
#pragma unroll 1
    for (int c = static_cast<int>(rank) * W + part * (W / 4);
         epi && c < static_cast<int>(rank) * W + (part + 1) * (W / 4); c += 16) {
        float rem[S][16];   // the other CTAs' partials: all loads in flight together
#pragma unroll
        for (int r = 0; r < S; ++r)
            if (r != static_cast<int>(rank)) {
                const float *src = ws_tile + (static_cast<int64_t>(r) * kMlpN + c) * kMlpBM + row;
#pragma unroll
                for (int j = 0; j < 16; ++j) rem[r][j] = __ldcg(src + j * kMlpBM);
            }
        uint32_t own[16];
        own16(c, own);
        float g[16];   // the partials' sum, then the activations
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            g[j] = 0.f;
#pragma unroll
            for (int r = 0; r < S; ++r) {
                const float x = (r == static_cast<int>(rank)) ? __uint_as_float(own[j]) : rem[r][j];
                g[j] = (r == 0) ? x : g[j] + x;
            }
        }
        float t = 0.f;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const int n = c + j;
            g[j] = gelu_erf(g[j] + s_b1[n]);
            if (HEAD) t = fmaf(s_w2[n], g[j], t);
        }
        t2 += t;
        if (!HEAD && ok && grow < p.M) {
            // 16 bf16 activations (round to nearest even) in two 16-byte stores
            uint32_t w[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) w[q] = pack_bf16x2(g[2 * q], g[2 * q + 1]);
            uint4 *dst = reinterpret_cast<uint4 *>(p.act + static_cast<int64_t>(grow) * kMlpN + c);
            dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
            dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
        }
    }
    if (HEAD) {
        // the row's dot product: the four warps of the quarter in order, then
        // the S column blocks in rank order (CTA 0 of the cluster finishes)
        __shared__ float s_part[3][kMlpBM];
        __shared__ float s_head[S][kMlpBM];
        if (epi && part > 0) s_part[part - 1][row] = t2;
        __syncthreads();
        if (part == 0) {
            const float t = ((t2 + s_part[0][row]) + s_part[1][row]) + s_part[2][row];
            if (S > 1)
                st_cluster_f32(map_rank(smem_addr(&s_head[rank][row]), 0u), t);
            else
                s_head[0][row] = t;
        }
        if (S > 1)
            cluster_sync();
        else
            __syncthreads();
        if (rank == 0 && part == 0 && ok && grow < p.M) {
            float t = s_head[0][row];
#pragma unroll
            for (int r = 1; r < S; ++r) t += s_head[r][row];
            p.out[grow] = 1.f / (1.f + expf(-(t + p.b2)));
        }
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && s_abort) status_or(p.status, SDD_DEV_TIMEOUT);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
}

// ---------------------------------------------------------------------------
// Layers 2 and 3 and the head of the deep scorer (K -> 256 -> 256 -> 256 -> 1):
// a cluster of four CTAs per 128-row tile, CTA q producing output columns
// [64 q, 64 q + 64) of both layers, so that the GELU epilogues (ALU-bound:
// 32 K activations per tile and layer) spread over four SMs.
//   1. TMA: the tile's first-layer activations a1 (128 x 256 bf16, four
//      64-column slices, 128-byte swizzle), rows [64 q, +64) of W2 and of W3.
//   2. z2 = W2_q a1 (M = 128, N = 64) into TMEM columns 0..63; the epilogue
//      writes a2 = bf16(GELU(z2 + b2)) for its 64 columns to the workspace.
//   3. Cluster barrier; every CTA loads the whole a2 tile back by TMA (L2)
//      into the swizzled K-major layout over a1.
//   4. z3 = W3_q a2 into TMEM columns 64..127; each row's dot product
//      w4 . GELU(z3 + b3) over the CTA's 64 columns goes to CTA 0, which adds
//      the four in rank order, adds b4 and applies the sigmoid.
// ---------------------------------------------------------------------------
constexpr int kTailCluster = 4;
constexpr int kTailN = kMlpN / kTailCluster;               // 64 output columns per CTA
constexpr uint32_t kTailASlice = kMlpBM * kMlpBK * 2;      // 16 KiB: 128 rows x 64 bf16
constexpr uint32_t kTailWSlice = kTailN * kMlpBK * 2;      // 8 KiB: 64 rows x 64 bf16
constexpr int kTailSlices = kMlpN / kMlpBK;                // 4
constexpr uint32_t kTailA = kTailSlices * kTailASlice;     // 64 KiB
constexpr uint32_t kTailW = kTailSlices * kTailWSlice;     // 32 KiB
// PAIR: W3 takes W2's place, so that two CTAs share an SM (launches of more
// clusters than fit at one CTA per SM: one's round trips run under the other's
// epilogue); otherwise both are loaded ahead.
constexpr int tail_smem(bool pair) { return static_cast<int>(kTailA + (pair ? 1 : 2) * kTailW) + 1024 + 256; }
constexpr uint32_t kTailTmemCols = 128;
constexpr int kTailThreads = 512;   // 16 warps: four per TMEM lane quarter, 16 columns each

struct TailParams {
    int32_t M;
    int32_t tile0;          // the launch's first tile
    const float *b2, *b3;   // [256]
    const uint16_t *w4;     // [256] bf16 bits
    float b4;
    uint16_t *a2;           // [tiles * 128, 256] bf16 bits (workspace)
    float *out;             // [M]
    int32_t *status;
};

template <bool PAIR>
__global__ void __launch_bounds__(kTailThreads, PAIR ? 2 : 1) mlp_tail_kernel(const __grid_constant__ CUtensorMap tmAct,
                                                                 const __grid_constant__ CUtensorMap tmW2,
                                                                 const __grid_constant__ CUtensorMap tmW3,
                                                                 const __grid_constant__ CUtensorMap tmAct2,
                                                                 const __grid_constant__ TailParams p) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                            ~static_cast<uintptr_t>(1023));
    unsigned char *bufA = smem, *bufW2 = smem + kTailA;   // a1, then a2; W2
    unsigned char *bufW3 = PAIR ? bufW2 : bufW2 + kTailW;
    uint64_t *bar = reinterpret_cast<uint64_t *>(bufW3 + kTailW);
    uint64_t *fullA = bar, *fullW2 = bar + 1, *fullW3 = bar + 2, *mma2 = bar + 3, *mma3 = bar + 4, *fullA2 = bar + 5;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bar + 6);
    __shared__ int s_abort;
    __shared__ float s_b2[kTailN], s_b3[kTailN], s_w4[kTailN];
    __shared__ float s_part[3][kMlpBM];             // warps 1..3 of a quarter: their parts of each row's dot product
    __shared__ float s_head[kTailCluster][kMlpBM];  // (CTA 0) each CTA's dot product of each row
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_rank();
    const int m0 = (p.tile0 + static_cast<int>(blockIdx.x) / kTailCluster) * kMlpBM;
    const int n0 = static_cast<int>(rank) * kTailN;
    if (tid == 0) {
        for (int i = 0; i < 6; ++i) mbar_init(&bar[i], 1);
        fence_mbar_init();
        s_abort = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                     "r"(kTailTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    auto load_w3 = [&] {
        mbar_arrive_expect_tx(fullW3, kTailW);
        for (int c = 0; c < kTailSlices; ++c)
            tma_load_2d(smem_addr(bufW3 + c * kTailWSlice), &tmW3, c * kMlpBK, n0, smem_addr(fullW3));
    };
    // launched as a programmatic dependent of the first layer: a1 (and the
    // workspace, which a2 overwrites) only once that grid has completed, and
    // the weights too, which a grid ahead of it may have written
    griddep_wait();
    if (tid == 0) {
        mbar_arrive_expect_tx(fullA, kTailA);
        mbar_arrive_expect_tx(fullW2, kTailW);
        for (int c = 0; c < kTailSlices; ++c) {
            tma_load_2d(smem_addr(bufA + c * kTailASlice), &tmAct, c * kMlpBK, m0, smem_addr(fullA));
            tma_load_2d(smem_addr(bufW2 + c * kTailWSlice), &tmW2, c * kMlpBK, n0, smem_addr(fullW2));
        }
        if (!PAIR) load_w3();
    }
    for (int n = tid; n < kTailN; n += kTailThreads) {
        s_b2[n] = __ldg(p.b2 + n0 + n);
        s_b3[n] = __ldg(p.b3 + n0 + n);
        s_w4[n] = __uint_as_float(static_cast<uint32_t>(__ldg(p.w4 + n0 + n)) << 16);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 1 && lane == 0) {
        const bool okA = mbar_wait_bounded(fullA, 0u, kWaitPolls), okB = mbar_wait_bounded(fullW2, 0u, kWaitPolls);
        if (okA && okB) {
            tc_fence_after();
#pragma unroll 1
            for (int c = 0; c < kTailSlices; ++c)
#pragma unroll
                for (int kk = 0; kk < kMlpBK / 16; ++kk)
                    umma_f16<kTailN>(tmem, umma_desc_sw128(smem_addr(bufA + c * kTailASlice) + kk * 32),
                                     umma_desc_sw128(smem_addr(bufW2 + c * kTailWSlice) + kk * 32),
                                     (c | kk) != 0 ? 1u : 0u);
        } else {
            s_abort = 1;
        }
        umma_commit(smem_addr(mma2));   // (arrives at once when nothing was issued)
    }
    __syncwarp();

    // layer-2 epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 (tile
    // rows), columns 16 (w / 4) .. + 15 of this CTA's 64
    const int quarter = warp & 3, part = warp >> 2;
    const int row = quarter * 32 + lane;
    const uint32_t tlane = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
    bool ok = __all_sync(0xFFFFFFFFu, mbar_wait_bounded(mma2, 0u, kWaitPolls));
    tc_fence_after();
    // layer 2's products have read W2: W3 into its place, under the epilogue
    const bool w3_issued = !PAIR || ok;   // (thread 0's)
    if (PAIR && tid == 0 && ok) load_w3();
    {
        uint32_t v[16];
        tmem_ld16_or0(ok, tlane + part * 16, v);
        uint32_t w[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int j = 2 * q;
            w[q] = pack_bf16x2(gelu_erf(__uint_as_float(v[j]) + s_b2[part * 16 + j]),
                               gelu_erf(__uint_as_float(v[j + 1]) + s_b2[part * 16 + j + 1]));
        }
        uint4 *dst = reinterpret_cast<uint4 *>(p.a2 + static_cast<int64_t>(m0 + row) * kMlpN + n0 + part * 16);
        __stcg(dst, make_uint4(w[0], w[1], w[2], w[3]));
        __stcg(dst + 1, make_uint4(w[4], w[5], w[6], w[7]));
    }
    fence_proxy_async_global();   // the stores, before the other CTAs' TMA loads read them
    cluster_sync();               // the four column blocks of a2 are in the workspace (release / acquire)

    // the a2 tile into bufA (a1 was consumed by the finished layer-2 MMAs)
    if (tid == 0) {
        mbar_arrive_expect_tx(fullA2, kTailA);
        for (int c = 0; c < kTailSlices; ++c)
            tma_load_2d(smem_addr(bufA + c * kTailASlice), &tmAct2, c * kMlpBK, m0, smem_addr(fullA2));
    }
    if (warp == 1 && lane == 0) {
        if (ok && mbar_wait_bounded(fullA2, 0u, kWaitPolls) && mbar_wait_bounded(fullW3, 0u, kWaitPolls)) {
            tc_fence_after();
#pragma unroll 1
            for (int c = 0; c < kTailSlices; ++c)
#pragma unroll
                for (int kk = 0; kk < kMlpBK / 16; ++kk)
                    umma_f16<kTailN>(tmem + kTailN, umma_desc_sw128(smem_addr(bufA + c * kTailASlice) + kk * 32),
                                     umma_desc_sw128(smem_addr(bufW3 + c * kTailWSlice) + kk * 32),
                                     (c | kk) != 0 ? 1u : 0u);
        } else {
            s_abort = 1;
        }
        umma_commit(smem_addr(mma3));
    }
    __syncwarp();

    // layer-3 epilogue and head: this thread's part of the row's dot product
    ok = __all_sync(0xFFFFFFFFu, mbar_wait_bounded(mma3, 0u, kWaitPolls)) && ok;
    tc_fence_after();
    griddep_launch_dependents();   // whatever follows may set up (it still waits for this grid)
    float t = 0.f;
    {
        uint32_t v[16];
        tmem_ld16_or0(ok, tlane + kTailN + part * 16, v);
#pragma unroll
        for (int j = 0; j < 16; ++j)
            t = fmaf(s_w4[part * 16 + j], gelu_erf(__uint_as_float(v[j]) + s_b3[part * 16 + j]), t);
    }
    if (part > 0) s_part[part - 1][row] = t;
    tc_fence_before();
    __syncthreads();
    if (part == 0)
        st_cluster_f32(map_rank(smem_addr(&s_head[rank][row]), 0u),
                       ((t + s_part[0][row]) + s_part[1][row]) + s_part[2][row]);
    cluster_sync();   // CTA 0 holds the four parts of every row
    if (rank == 0 && part == 0 && ok && m0 + row < p.M)
        p.out[m0 + row] = 1.f / (1.f + expf(-((((s_head[0][row] + s_head[1][row]) + s_head[2][row]) +
                                                s_head[3][row]) + p.b4)));
    if (tid == 0) {
        // every load this CTA issued has landed before its shared memory goes away
        for (int i : {0, 1, 5}) (void)mbar_wait_bounded(&bar[i], 0u, kWaitPolls);
        if (w3_issued) (void)mbar_wait_bounded(fullW3, 0u, kWaitPolls);
        if (s_abort || !ok) status_or(p.status, SDD_DEV_TIMEOUT);
    }
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTailTmemCols)
                     : "memory");
}

// ---------------------------------------------------------------------------
// The deep scorer of one 128-row tile in one CTA (whole waves of tiles): the
// first layer with K in kMlpChains chains, then layers 2 and 3 and the head
// without a2 or partial sums leaving the SM; every sum in the order of the
// split form, so that a row's score does not depend on the batch.  After the main loop the ring's 192 KiB
// hold the activations (64 KiB, written by the epilogues in the operands'
// swizzled layout) and one 256 x 256 weight matrix (128 KiB: W2 as soon as the
// main loop's products have read the ring, W3 once layer 2's have read W2,
// each under the epilogue before it).  TMEM columns 0-255 hold z1, 256-511 z2,
// 0-255 z3 (and the main loop's chains all of them in turn).  a1 is also written to
// p.act.
//
// Bound by the main loop's operands (2.9 MB into each SM, ~22 us) and then by
// the issue of 3 x 32 K erf-form GELUs an SM.  GB300, K = 3584 + 256: 51.7 us
// for 128 tiles (16,384 rows) against 93.8 us with K split four ways, clusters
// of four and a second launch for the tail (61.4 us with K not split and the
// tail in a second launch); 20,000 rows 71.7 against 116 us.
// ---------------------------------------------------------------------------
struct DeepParams {
    int32_t M, K, Ka, tile0;
    const float *b1, *b2, *b3;   // [256]
    const uint16_t *w4;          // [256] bf16 bits
    float b4;
    uint16_t *act;               // [M, 256] bf16 bits: a1
    float *out;                  // [M]
    int32_t *status;
};
constexpr uint32_t kDeepW = 4u * kBTileBytes;   // 128 KiB: a 256 x 256 bf16 matrix, four 64-column slices
static_assert(kTailA + kDeepW == kMlpStages * kStageBytes, "activations and weights share the ring");

// Address of the 16-byte chunk of columns 8 c8 .. 8 c8 + 7 of a row in the
// swizzled activations (64-column slices of 128 rows x 128 bytes).
__device__ __forceinline__ unsigned char *act_chunk(unsigned char *buf, int row, int c8) {
    return buf + (c8 >> 3) * kTailASlice + row * 128 + (((c8 & 7) ^ (row & 7)) << 4);
}

__global__ void __launch_bounds__(kMlpThreadsChains, 1) mlp_deep_kernel(const __grid_constant__ CUtensorMap tmA,
                                                                 const __grid_constant__ CUtensorMap tmA2,
                                                                 const __grid_constant__ CUtensorMap tmB,
                                                                 const __grid_constant__ CUtensorMap tmW2,
                                                                 const __grid_constant__ CUtensorMap tmW3,
                                                                 const __grid_constant__ DeepParams p) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                            ~static_cast<uintptr_t>(1023));
    unsigned char *bufA = smem, *bufW = smem + kTailA;
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + kMlpStages * kStageBytes);
    uint64_t *empty = full + kMlpStages;
    uint64_t *done = empty + kMlpStages;   // z1's chains, then z2, z3
    uint64_t *fullW = done + kMlpChains + 2;   // W2, W3
    uint64_t *drained = fullW + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(drained + kMlpChains - 2);
    __shared__ int s_abort;
    __shared__ float s_b[3][kMlpN], s_w4[kMlpN];
    __shared__ float s_part[3][kMlpBM];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = (p.tile0 + static_cast<int>(blockIdx.x)) * kMlpBM;

    if (tid == 0) {
        for (int i = 0; i < 2 * kMlpStages + kMlpChains + 4; ++i) mbar_init(&full[i], 1);
        for (int i = 0; i < kMlpChains - 2; ++i) mbar_init(&drained[i], kMlpThreads / 32);
        fence_mbar_init();
        s_abort = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                     "r"(2 * kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    griddep_wait();
    for (int n = tid; n < kMlpN; n += kMlpThreadsChains) {
        s_b[0][n] = __ldg(p.b1 + n);
        s_b[1][n] = __ldg(p.b2 + n);
        s_b[2][n] = __ldg(p.b3 + n);
        s_w4[n] = __uint_as_float(static_cast<uint32_t>(__ldg(p.w4 + n)) << 16);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const int nk = p.K / kMlpBK, C = mlp_chains(nk);
    mlp_mainloop<kMlpThreads / 32>(smem, full, empty, done, drained, &tmA, &tmA2, &tmB, p.Ka, m0, 0, nk, C, tmem, &s_abort);
    __syncwarp();

    // warp w: TMEM lanes 32 (w % 4) .. + 31 (tile rows), columns 64 (w / 4) .. + 63
    const int quarter = warp & 3, part = warp >> 2;
    const bool epi = warp < kMlpThreads / 32;
    const int row = quarter * 32 + lane, grow = m0 + row;
    const uint32_t tlane = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
    bool ok = true;
    float t = 0.f;   // this thread's part of the head's dot product
    int w_issued = 0;
#pragma unroll 1
    for (int layer = 0; layer < 3; ++layer) {
        // z of this layer is complete, and its products have read their operands
        if (layer == 0) {
            ok = mlp_drain(done, drained, C, epi, tlane, part);
        } else {
            ok = __all_sync(0xFFFFFFFFu, mbar_wait_bounded(&done[kMlpChains + layer - 1], 0u, kWaitPolls)) && ok;
            tc_fence_after();
        }
        if (!ok) s_abort = 1;
        if (layer == 0) {
            // (every warp: a CTA's threads have all passed the main loop)
            __syncthreads();   // the producer has left the ring
            griddep_launch_dependents();
        }
        if (tid == 0 && layer < 2 && ok) {
            mbar_arrive_expect_tx(&fullW[layer], kDeepW);
            for (int c = 0; c < kTailSlices; ++c)
                tma_load_2d(smem_addr(bufW + c * kBTileBytes), layer == 0 ? &tmW2 : &tmW3, c * kMlpBK, 0,
                            smem_addr(&fullW[layer]));
            w_issued = layer + 1;
        }
        const uint32_t z = tlane + (layer == 1 ? kTmemCols : 0u) + part * 64;
        const float *bias = s_b[layer];
#pragma unroll 1
        for (int c = 0; epi && c < 64; c += 16) {
            uint32_t v[16];
            tmem_ld16_or0(ok, z + c, v);
            float g[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) g[j] = gelu_erf(__uint_as_float(v[j]) + bias[part * 64 + c + j]);
            if (layer == 2) {
                float d = 0.f;
#pragma unroll
                for (int j = 0; j < 16; ++j) d = fmaf(s_w4[part * 64 + c + j], g[j], d);
                t += d;   // (16 columns at a time, as the tail kernel's warps)
                continue;
            }
            uint32_t w[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) w[q] = pack_bf16x2(g[2 * q], g[2 * q + 1]);
            const int c8 = part * 8 + (c >> 3);
            *reinterpret_cast<uint4 *>(act_chunk(bufA, row, c8)) = make_uint4(w[0], w[1], w[2], w[3]);
            *reinterpret_cast<uint4 *>(act_chunk(bufA, row, c8 + 1)) = make_uint4(w[4], w[5], w[6], w[7]);
            if (layer == 0 && ok && grow < p.M) {
                uint4 *dst = reinterpret_cast<uint4 *>(p.act + static_cast<int64_t>(grow) * kMlpN + part * 64 + c);
                dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
                dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
            }
        }
        if (layer == 2) break;
        fence_proxy_async_smem();   // the activations, before the tensor cores read them
        tc_fence_before();
        __syncthreads();
        if (warp == 1 && lane == 0) {
            tc_fence_after();
            if (ok && mbar_wait_bounded(&fullW[layer], 0u, kWaitPolls)) {
                const uint32_t d = tmem + (layer == 0 ? kTmemCols : 0u);
#pragma unroll 1
                for (int c = 0; c < kTailSlices; ++c)
#pragma unroll
                    for (int kk = 0; kk < kMlpBK / 16; ++kk)
                        umma_f16(d, umma_desc_sw128(smem_addr(bufA + c * kTailASlice) + kk * 32),
                                 umma_desc_sw128(smem_addr(bufW + c * kBTileBytes) + kk * 32),
                                 (c | kk) != 0 ? 1u : 0u);
            } else {
                s_abort = 1;
            }
            umma_commit(smem_addr(&done[kMlpChains + layer]));   // (arrives at once when nothing was issued)
        }
        __syncwarp();
    }
    if (epi && part > 0) s_part[part - 1][row] = t;
    tc_fence_before();
    __syncthreads();
    if (part == 0 && ok && grow < p.M) {
        t = ((t + s_part[0][row]) + s_part[1][row]) + s_part[2][row];
        p.out[grow] = 1.f / (1.f + expf(-(t + p.b4)));
    }
    if (tid == 0) {
        // every weight load has landed before the shared memory goes away
        for (int i = 0; i < w_issued; ++i) (void)mbar_wait_bounded(&fullW[i], 0u, kWaitPolls);
        if (s_abort) status_or(p.status, SDD_DEV_TIMEOUT);
    }
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * kTmemCols)
                     : "memory");
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
    }
    return fn;
}

// Row-major bf16 [rows, K] as a 2D tensor map with (64 x box_rows) boxes and the 128-byte swizzle.
bool make_map(CUtensorMap *map, const void *base, int64_t rows, int K, int box_rows) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
    if (!enc) return false;
    const cuuint64_t dims[2] = {static_cast<cuuint64_t>(K), static_cast<cuuint64_t>(rows)};
    const cuuint64_t strides[1] = {static_cast<cuuint64_t>(K) * 2};
    const cuuint32_t box[2] = {static_cast<cuuint32_t>(kMlpBK), static_cast<cuuint32_t>(box_rows)};
    const cuuint32_t estr[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Encoded maps of recent (address, rows, K) operands: a decode loop passes the
// same weights every round and often the same hidden-state buffer.
struct MapCache {
    struct Entry {
        const void *base;
        int64_t rows;
        int K, box;
        CUtensorMap map;
    };
    static constexpr int kSlots = 16;
    Entry e[kSlots];
    int n = 0, next = 0;
    std::mutex mu;
    bool get(CUtensorMap *out, const void *base, int64_t rows, int K, int box) {
        std::lock_guard<std::mutex> g(mu);
        for (int i = 0; i < n; ++i)
            if (e[i].base == base && e[i].rows == rows && e[i].K == K && e[i].box == box) {
                *out = e[i].map;
                return true;
            }
        if (!make_map(out, base, rows, K, box)) return false;
        e[next] = Entry{base, rows, K, box, *out};
        next = (next + 1) % kSlots;
        n = n < kSlots ? n + 1 : n;
        return true;
    }
};
MapCache g_maps;
constexpr int kMaxDevices = 64;
std::atomic<int> g_attr_ready[kMaxDevices];
// What fits a device at once: CTAs of the first layer's kernels one per SM, and
// clusters of 4 and of 2 of them (a GPC's SMs are not a multiple of four: 36
// clusters of 4 on 152 SMs, 76 of 2).
struct MlpDev {
    int sms, c4, c2;
};
MlpDev g_dev[kMaxDevices];

cudaError_t max_clusters(int *n, void (*kernel)(CUtensorMap, CUtensorMap, CUtensorMap, MlpParams), int S) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(S);
    cfg.blockDim = dim3(mlp_threads(S));
    cfg.dynamicSmemBytes = kMlpSmem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = S;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(n, kernel, &cfg);
}

// Per-device opt-in of every kernel here to its dynamic shared memory.
cudaError_t mlp_prepare(MlpDev *out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    if (g_attr_ready[dev].load(std::memory_order_acquire)) {
        *out = g_dev[dev];
        return cudaSuccess;
    }
    for (auto fn : {mlp_kernel<1, true>, mlp_kernel<2, true>, mlp_kernel<4, true>, mlp_kernel<2, false>,
                    mlp_kernel<4, false>}) {
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMlpSmem);
        if (e != cudaSuccess) return e;
    }
    MlpDev d = {};
    e = cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = max_clusters(&d.c4, mlp_kernel<4, true>, 4);
    if (e == cudaSuccess) e = max_clusters(&d.c2, mlp_kernel<2, true>, 2);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(mlp_tail_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, tail_smem(false));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(mlp_tail_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, tail_smem(true));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(mlp_deep_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMlpSmem);
    if (e != cudaSuccess) return e;
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    if (!g_attr_ready[dev].load(std::memory_order_acquire)) {
        g_dev[dev] = d;
        g_attr_ready[dev].store(1, std::memory_order_release);
    }
    *out = d;
    return cudaSuccess;
}

// How M rows' tiles are run: `full` of them, whole waves of one tile per SM,
// with K not split (no operand read twice, nothing exchanged), and the `rest`
// after them with K split S ways, as far as their clusters all fit at once (one
// wave again: 13.9 us with S = 4 at 32 tiles of K = 3584, 14.6 at 36, and 25.4 at
// 37, whose last cluster waits for another; 18.2 with S = 2 there, 22.4 at 76; a
// full wave with S = 1 35.4).  A larger rest runs unsplit too (it is then part of
// `full`), and so do, of fewer than eight slices of K, a rest that two splits
// would take (K = 448, 47 tiles: 9.4 us against 9.9) and one behind whole waves
// (196 tiles: 18.3 against 20.0).  GB300,
// one-layer scorer, K = 3584, three inputs in turn, against all tiles split four
// ways: 8,192 rows 20.3 / 28.9 us, 12,000 28.2 / 43.7, 16,384 33.3 / 58.0,
// 20,000 44.9 / 71.9, 32,768 64.4 / 111.9.
struct MlpPlan {
    int full, rest, S;
};
MlpPlan mlp_plan(int M, int K, const MlpDev &dev) {
    const int tiles = (M + kMlpBM - 1) / kMlpBM, nk = K / kMlpBK;
    MlpPlan q{tiles / dev.sms * dev.sms, tiles % dev.sms, 1};
    if (q.rest > 0) q.S = (q.rest <= dev.c4 && nk >= 4) ? 4 : (q.rest <= dev.c2 && nk >= 2) ? 2 : 1;
    if (nk < 2 * kMlpChains && (q.S == 2 || q.full > 0)) q.S = 1;
    if (q.S == 1) q = MlpPlan{tiles, 0, 1};
    return q;
}

// The first layer: A = [A1 | A2] (A2 may be absent: Ka = K), W1 [256, K].
// head: fused GELU / w2 / sigmoid into out; else bf16 activations into act, of
// the plan's rest only (its whole waves are mlp_deep_kernel's).
cudaError_t launch_layer1(const void *a1, int Ka, const void *a2, int M, int K, const void *W1, const float *b1,
                          const void *w2, float b2, float *out, uint16_t *act, bool head, float *ws, int32_t *status,
                          cudaStream_t stream, const char **why) {
    CUtensorMap tmA, tmA2, tmB;
    if (!g_maps.get(&tmA, a1, M, Ka, kMlpBM) || !g_maps.get(&tmB, W1, kMlpN, K, kMlpN) ||
        !g_maps.get(&tmA2, a2 ? a2 : a1, M, a2 ? K - Ka : Ka, kMlpBM)) {
        *why = "cuTensorMapEncodeTiled failed";
        return cudaErrorInvalidValue;
    }
    MlpDev dev;
    cudaError_t e = mlp_prepare(&dev);
    if (e != cudaSuccess) return e;
    MlpParams p;
    p.M = M;
    p.K = K;
    p.Ka = Ka;
    p.b1 = b1;
    p.w2 = static_cast<const uint16_t *>(w2);
    p.b2 = b2;
    p.out = out;
    p.act = act;
    p.ws = ws;
    p.status = status;
    // Tiles [t0, t0 + n) with K split S ways.
    auto launch = [&](int t0, int n, int S) {
        p.tile0 = t0;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(n * S);
        cfg.blockDim = dim3(mlp_threads(S));
        cfg.dynamicSmemBytes = kMlpSmem;
        cfg.stream = stream;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = S;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // setup overlaps the work ahead
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        // (a plan's rest has S = 4 or 2)
        const auto kernel = S == 4   ? (head ? mlp_kernel<4, true> : mlp_kernel<4, false>)
                            : S == 2 ? (head ? mlp_kernel<2, true> : mlp_kernel<2, false>)
                                     : mlp_kernel<1, true>;
        return cudaLaunchKernelEx(&cfg, kernel, tmA, tmA2, tmB, p);
    };
    const MlpPlan plan = mlp_plan(M, K, dev);
    if (head && plan.full > 0) {
        e = launch(0, plan.full, 1);
        if (e != cudaSuccess) return e;
    }
    return plan.rest > 0 ? launch(plan.full, plan.rest, plan.S) : cudaSuccess;
}

}  // namespace

size_t mlp_workspace_bytes(int M) {
    const int64_t tiles = (static_cast<int64_t>(M) + kMlpBM - 1) / kMlpBM;
    return static_cast<size_t>(tiles) * 4 * kMlpN * kMlpBM * sizeof(float);   // K split at most four ways
}

cudaError_t launch_mlp(const void *h, int M, int K, const void *W1, const float *b1, const void *w2, float b2,
                       float *out, void *ws, int32_t *status, cudaStream_t stream, const char **why) {
    *why = nullptr;
    if (M == 0) return cudaSuccess;
    return launch_layer1(h, K, nullptr, M, K, W1, b1, w2, b2, out, nullptr, true, static_cast<float *>(ws), status,
                         stream, why);
}

cudaError_t launch_scorer_deep(const void *h, int Kh, const void *f, int M, const void *W1, const float *b1,
                               const void *W2, const float *b2, const void *W3, const float *b3, const void *w4,
                               float b4, uint16_t *act, float *out, void *ws, int32_t *status, cudaStream_t stream,
                               const char **why) {
    *why = nullptr;
    if (M == 0) return cudaSuccess;
    MlpDev dev;
    cudaError_t e = mlp_prepare(&dev);
    if (e != cudaSuccess) return e;
    const int K = Kh + kMlpN;
    const MlpPlan plan = mlp_plan(M, K, dev);
    if (plan.full > 0) {
        CUtensorMap tmA, tmA2, tmB, tmW2, tmW3;
        if (!g_maps.get(&tmA, h, M, Kh, kMlpBM) || !g_maps.get(&tmA2, f, M, kMlpN, kMlpBM) ||
            !g_maps.get(&tmB, W1, kMlpN, K, kMlpN) || !g_maps.get(&tmW2, W2, kMlpN, kMlpN, kMlpN) ||
            !g_maps.get(&tmW3, W3, kMlpN, kMlpN, kMlpN)) {
            *why = "cuTensorMapEncodeTiled failed";
            return cudaErrorInvalidValue;
        }
        DeepParams d;
        d.M = M;
        d.K = K;
        d.Ka = Kh;
        d.tile0 = 0;
        d.b1 = b1;
        d.b2 = b2;
        d.b3 = b3;
        d.w4 = static_cast<const uint16_t *>(w4);
        d.b4 = b4;
        d.act = act;
        d.out = out;
        d.status = status;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(plan.full);
        cfg.blockDim = dim3(kMlpThreadsChains);
        cfg.dynamicSmemBytes = kMlpSmem;
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, mlp_deep_kernel, tmA, tmA2, tmB, tmW2, tmW3, d);
        if (e != cudaSuccess || plan.rest == 0) return e;
    }
    e = launch_layer1(h, Kh, f, M, K, W1, b1, nullptr, 0.f, nullptr, act, false, static_cast<float *>(ws), status,
                      stream, why);
    if (e != cudaSuccess || *why) return e;
    const int64_t rows_pad = ((static_cast<int64_t>(M) + kMlpBM - 1) / kMlpBM) * kMlpBM;
    CUtensorMap tmAct, tmW2, tmW3, tmAct2;
    if (!g_maps.get(&tmAct, act, M, kMlpN, kMlpBM) || !g_maps.get(&tmW2, W2, kMlpN, kMlpN, kTailN) ||
        !g_maps.get(&tmW3, W3, kMlpN, kMlpN, kTailN) || !g_maps.get(&tmAct2, ws, rows_pad, kMlpN, kMlpBM)) {
        *why = "cuTensorMapEncodeTiled failed";
        return cudaErrorInvalidValue;
    }
    const bool pair = plan.rest > dev.c4;   // (more clusters of 4 than fit one CTA per SM)
    TailParams p;
    p.M = M;
    p.tile0 = plan.full;
    p.b2 = b2;
    p.b3 = b3;
    p.w4 = static_cast<const uint16_t *>(w4);
    p.b4 = b4;
    p.a2 = static_cast<uint16_t *>(ws);   // the first layer's partials are dead once it has finished
    p.out = out;
    p.status = status;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(plan.rest * kTailCluster);
    cfg.blockDim = dim3(kTailThreads);
    cfg.dynamicSmemBytes = tail_smem(pair);
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kTailCluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // weight loads overlap the first layer
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, pair ? mlp_tail_kernel<true> : mlp_tail_kernel<false>, tmAct, tmW2, tmW3, tmAct2, p);
}

// ---------------------------------------------------------------------------
// The learned scorer's scalar-feature block (App. A.7's list): one warp per
// position writes its 256 bf16 columns (lane u: columns 8u .. 8u + 7), zero
// except the logits-side features and the position ones.
// ---------------------------------------------------------------------------
namespace {
__global__ void scorer_features_kernel(const float *maxprob, const float *entropy, const float *margin,
                                       const float *top5, int64_t M, int gamma, float gen, uint16_t *f) {
    const int64_t w = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    griddep_wait();
    if (w >= M) return;
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = 0.f;
    if (lane == 0) {   // columns 4..7: top-1 probability, its log, entropy, its negative
        const float mp = __ldg(maxprob + w), h = __ldg(entropy + w);
        v[4] = mp;
        v[5] = logf(mp);
        v[6] = h;
        v[7] = -h;
    } else if (lane == 1) {   // columns 8, 9: margin, top-5 mass; 14, 15: block position, generated length
        v[0] = __ldg(margin + w);
        v[1] = __ldg(top5 + w);
        v[6] = static_cast<float>(w % gamma) / static_cast<float>(gamma);
        v[7] = gen;
    }
    const uint4 u = make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]),
                               pack_bf16x2(v[6], v[7]));
    reinterpret_cast<uint4 *>(f + w * kMlpN)[lane] = u;
}
}  // namespace

cudaError_t launch_scorer_features(const float *maxprob, const float *entropy, const float *margin, const float *top5,
                                   int64_t M, int gamma, float gen, uint16_t *f, cudaStream_t stream) {
    if (M == 0) return cudaSuccess;
    const int64_t threads = M * 32;
    return launch_dependent(scorer_features_kernel, dim3(static_cast<unsigned>((threads + 255) / 256)), dim3(256), 0,
                            stream, maxprob, entropy, margin, top5, M, gamma, gen, f);
}

}  // namespace sdd
