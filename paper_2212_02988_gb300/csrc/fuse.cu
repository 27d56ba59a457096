// fuse.cu — single-stream launch of the per-voxel map update; the device
// body is in fuse_dev.cuh.
#include <cuda/atomic>

#include "fuse_dev.cuh"
#include "kernels.h"
#include "render_dev.cuh"

namespace prism {

// The tiles in the frustum, appended to `list` (ctr[0] counts them), and those
// whose cells may read a voxel of them, to cells_list (ctr[1]).  rejected
// (nullable): a nonzero value lists no tile (the localisation of this step was
// rejected, so its frame is not fused).
// depth (nullable): the observed frame whose depth validity the blocks past the
// first cull_blocks write to mask.  The two are independent and short, and a
// launch each costs a map update of known pose about 3 us of its 36 (200^3,
// 251x189).
__global__ void __launch_bounds__(256) k_fuse_cull(KParams P, const float* __restrict__ w2c, int* __restrict__ list,
                                                   int* __restrict__ cells_list, unsigned int* __restrict__ ctr,
                                                   const int* __restrict__ rejected, int cull_blocks,
                                                   const float* __restrict__ depth, uint8_t* __restrict__ mask) {
    pdl_enter();
    if ((int)blockIdx.x >= cull_blocks) {
        const int p = ((int)blockIdx.x - cull_blocks) * (int)blockDim.x + (int)threadIdx.x;
        if (p < P.W * P.H) depth_mask_px(P, depth, mask, p);
        return;
    }
    __shared__ float sM[9], sb[3];
    load_w2c(w2c, sM, sb);
    __syncthreads();
    cull_tiles(P, sM, sb, blockIdx.x * blockDim.x + threadIdx.x, rejected && *rejected, list, cells_list, ctr);
}

// Persistent over the listed tiles (ctr[0] of them); a block reads its next
// tile of the list beside the current one.  Without empty-space skipping nothing
// reads the counters after it: the last block (ticket in ctr[1], which counts no
// tiles then) clears them (a memset behind it: 12.3 us an update of a
// 128^3 map from 320x240 against 10.9).  Bound by the latency of three
// dependent rounds of loads (pixel, update decision, colours) at half the warps.
template <bool BF16>
__global__ void __launch_bounds__(256, 4) k_fuse_list(KParams P, MapPlanes M, const float* __restrict__ w2c,
                                                   const float* __restrict__ depth, const float* __restrict__ rgb,
                                                   const uint8_t* __restrict__ mask, DevStats* __restrict__ stats,
                                                   const int* __restrict__ list, unsigned int* __restrict__ ctr) {
    pdl_enter();
    __shared__ float sM[9], sb[3];
    __shared__ unsigned int s_count[2];
    load_w2c(w2c, sM, sb);
    if (threadIdx.x < 2) s_count[threadIdx.x] = 0u;
    __syncthreads();
    const unsigned int count = min(ctr[0], (unsigned int)(P.nbx * P.nby * P.nbz));   // (the list's room)
    int tile = blockIdx.x < count ? list[blockIdx.x] : 0;
    for (unsigned int i = blockIdx.x; i < count; i += gridDim.x) {
        const int cur = tile;
        if (i + gridDim.x < count) tile = list[i + gridDim.x];
        fuse_tile<BF16>(P, M, sM, sb, depth, rgb, mask, s_count, (uint32_t)cur);
    }
    __syncthreads();
    add_fuse_counts(stats, s_count);
    if (!P.skip && threadIdx.x == 0) {
        cuda::atomic_ref<unsigned int, cuda::thread_scope_device> ticket(ctr[1]);
        if (ticket.fetch_add(1u, cuda::memory_order_acq_rel) == gridDim.x - 1) ctr[0] = ctr[1] = 0u;
    }
}

template <bool BF16>
static int fuse_grid() {
    static int cached = 0;
    if (!cached) {
        int dev = 0, sms = 0, per = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_fuse_list<BF16>, 256, 0);
        cached = (sms > 0 ? sms : 152) * (per > 0 ? per : 1);
    }
    return cached;
}

cudaError_t launch_fuse_listed(const KParams& P, const MapPlanes& M, const float* w2c, const float* depth,
                               const float* rgb, uint8_t* mask, bool mask_ready, DevStats* stats, int* list,
                               int* cells_list, unsigned int* ctr, const int* rejected, cudaStream_t s) {
    const int cull = (P.nbx * P.nby * P.nbz + 255) / 256, pix = mask_ready ? 0 : (P.W * P.H + 255) / 256;
    cudaError_t e = launch_pdl(k_fuse_cull, cull + pix, 256, s, P, w2c, list, cells_list, ctr, rejected, cull, depth,
                               mask);
    if (e != cudaSuccess) return e;
    if (P.bf16) return launch_pdl(k_fuse_list<true>, fuse_grid<true>(), 256, s, P, M, w2c, depth, rgb, (const uint8_t*)mask, stats,
                                  (const int*)list, ctr);
    return launch_pdl(k_fuse_list<false>, fuse_grid<false>(), 256, s, P, M, w2c, depth, rgb, (const uint8_t*)mask, stats,
                      (const int*)list, ctr);
}

}  // namespace prism
