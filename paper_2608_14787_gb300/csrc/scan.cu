// scan.cu -- the streaming kernel (the per-warp work is in scan.cuh).
#include <algorithm>
#include <atomic>

#include "scan.cuh"

namespace sdd {

namespace {

// FEAT: also the five largest logits of every drafter row piece (extended
// features).  KIND: a call over rows of one kind leaves the other's code out.
template <int DT, bool FEAT, int KIND>
__global__ void __launch_bounds__(kThreads, 1) scan_kernel(const __grid_constant__ ScanParams p) {
    extern __shared__ __align__(128) unsigned char smem[];
    // launched as a programmatic dependent of whatever precedes it in the
    // stream: nothing is read or written before that work has completed
    griddep_wait();
    scan_warp<DT, FEAT, KIND>(p, smem, threadIdx.x >> 5, blockDim.x >> 5);
}

// [bf16][mixed rows, drafter rows, target rows, drafter rows with the extended features]
void (*const kScanKernels[2][4])(ScanParams) = {
    {scan_kernel<SDD_F32, false, kRowsMixed>, scan_kernel<SDD_F32, false, kRowsDrafter>,
     scan_kernel<SDD_F32, false, kRowsTarget>, scan_kernel<SDD_F32, true, kRowsDrafter>},
    {scan_kernel<SDD_BF16, false, kRowsMixed>, scan_kernel<SDD_BF16, false, kRowsDrafter>,
     scan_kernel<SDD_BF16, false, kRowsTarget>, scan_kernel<SDD_BF16, true, kRowsDrafter>}};

}  // namespace

int scan_max_ctas_per_sm() {
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, scan_kernel<SDD_BF16, false, kRowsMixed>, kThreads, kScanSmem);
    return n;
}

// Opt every instantiation in to its dynamic shared memory on the current device.
cudaError_t scan_prepare_device() {
    for (const auto &row : kScanKernels)
        for (auto k : row) {
            const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kScanSmem);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

// The launch overhead of the streaming grid overlaps the tail of the work
// ahead of it in the stream (the kernel waits for that work to complete).
namespace {
std::atomic<uint32_t> g_wait_polls{0};
std::atomic<int> g_drop_copy{0};
}  // namespace

void set_scan_wait_hooks(uint32_t polls, int drop_copy) {
    g_wait_polls.store(polls, std::memory_order_relaxed);
    g_drop_copy.store(drop_copy ? 1 : 0, std::memory_order_relaxed);
}
void get_scan_wait_hooks(uint32_t &polls, int32_t &drop_copy) {
    const uint32_t n = g_wait_polls.load(std::memory_order_relaxed);
    polls = n ? n : kWaitPolls;
    drop_copy = g_drop_copy.load(std::memory_order_relaxed);
}

cudaError_t launch_scan(const ScanParams &p, cudaStream_t stream) {
    const bool bf = p.dtype == SDD_BF16, feat = p.feat != nullptr;
    const int kind = feat ? 3 : p.n_groups > 1 ? kRowsMixed : p.grp[0].kind == 0 ? kRowsDrafter : kRowsTarget;
    void (*const k)(ScanParams) = kScanKernels[bf][kind];
    ScanParams q = p;
    get_scan_wait_hooks(q.wait_polls, q.drop_copy);
    q.spread = (p.W + std::min(p.W, p.ctas) - 1) / std::min(p.W, p.ctas);
    return launch_dependent(k, dim3(std::min(p.W, p.ctas)), dim3(32 * q.spread), ring_bytes(kStages, q.spread), stream,
                            q);
}

}  // namespace sdd
