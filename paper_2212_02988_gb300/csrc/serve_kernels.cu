// serve_kernels.cu — the batched filter step of the serving runtime: one
// persistent launch per kernel of the step over the work of every stream in
// the batch (see serve.h).  Items of unequal cost (render tiles,
// localisation blocks) are taken dynamically from a per-launch counter;
// uniform ones (pixel blocks, voxel tiles) by a grid stride.
#include "fuse_dev.cuh"
#include "render_dev.cuh"
#include "serve.h"
#include "state_dev.cuh"
#include "track_dev.cuh"

namespace prism {

namespace {

// Member whose item range [off[i], off[i + 1]) holds `item` (off[0] = 0).
__device__ __forceinline__ int find_member(const int* off, int n, int item) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= item) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// The block's next work item from a launch-wide counter.  The first barrier
// keeps every thread's use of the previous item (and of the block's shared
// memory) ahead of the next item's.
__device__ __forceinline__ int next_item(unsigned int* ctr) {
    __shared__ int s_item;
    __syncthreads();
    if (threadIdx.x == 0) s_item = (int)atomicAdd(ctr, 1u);
    __syncthreads();
    return s_item;
}

// The slot of member `k` in shared memory: the localisation and the map update
// read its configuration many times an item (52.9 -> 51.8 us a pass, 49 -> 45 us
// the map update of ten streams; the render keeps what it needs in registers and
// was 4 % slower from shared memory).  prev: the member staged before (-1: none).  Every thread calls it,
// after a barrier that follows the last use of *dst; the barrier here publishes it.
__device__ __forceinline__ void stage_slot(const SlotDesc* __restrict__ src, SlotDesc* dst, int k, int& prev) {
    static_assert(sizeof(SlotDesc) % 8 == 0, "copied in 8-byte words");
    if (k == prev) return;
    prev = k;
    for (int e = threadIdx.x; e < (int)(sizeof(SlotDesc) / 8); e += blockDim.x)
        reinterpret_cast<unsigned long long*>(dst)[e] = reinterpret_cast<const unsigned long long*>(src)[e];
    __syncthreads();
}

}  // namespace

// Prediction and the Gauss-Newton start pose matrices; block k runs the k-th
// localising member.
__global__ void __launch_bounds__(256) kb_predict(const SlotDesc* __restrict__ slots, const BatchDesc* __restrict__ b,
                                                  const double* __restrict__ imu) {
    pdl_enter();
    const int k = blockIdx.x;
    if (k >= b->n_loc) return;
    const BatchMember& m = b->m[b->loc[k]];
    const SlotDesc& S = slots[m.slot];
    predict_block<PREP_REL>(S.P, S.dev, imu + 7 * m.imu_off, m.n_imu, m.dt);
}

// Depth validity of the observed frames.
__global__ void __launch_bounds__(256) kb_mask(const SlotDesc* __restrict__ slots, const BatchDesc* __restrict__ b) {
    pdl_enter();
    const int total = b->pix_off[b->n];
    for (int item = blockIdx.x; item < total; item += gridDim.x) {
        const int i = find_member(b->pix_off, b->n, item);
        const SlotDesc& S = slots[b->m[i].slot];
        const int p = (item - b->pix_off[i]) * 256 + threadIdx.x;
        if (p < S.P.W * S.P.H) depth_mask_px(S.P, S.depth, S.o_mask, p);
    }
}

// The anchors' packing; item = one 32x8-pixel tile.  Pixel by pixel from global
// memory, with the validity of five pixels tested anew at each, a batch of nine
// streams of 160x120 to 640x480 took 45 us; by tiles 33 us.
__global__ void __launch_bounds__(256) kb_pack(const SlotDesc* __restrict__ slots, const BatchDesc* __restrict__ b) {
    pdl_enter();
    const int total = b->pack_off[b->n];
    for (int item = blockIdx.x; item < total; item += gridDim.x) {
        const int i = find_member(b->pack_off, b->n, item);
        const SlotDesc& S = slots[b->m[i].slot];
        const int t = item - b->pack_off[i], across = (S.P.W + kPackTW - 1) / kPackTW;
        anchor_pack_tile(S.P, S.a_depth, S.a_rgb, S.a0, S.a1, t % across, t / across);
        __syncthreads();   // the tile's shared memory is reused by the next item
    }
}

// One localisation pass of every localising member; item = one virtual block.
template <int MODE>
__global__ void __launch_bounds__(Block<MODE>::threads, 1) kb_track(const SlotDesc* __restrict__ slots, BatchDesc* __restrict__ b,
                                                int ctr) {
    pdl_enter();
    const int* off = MODE == TRACK_GN ? b->gn_off : b->lap_off;
    const int total = off[b->n_loc];
    __shared__ SlotDesc S;
    int prev = -1;
    for (;;) {
        const int item = next_item(&b->ctr[ctr]);
        if (item >= total) break;
        const int k = find_member(off, b->n_loc, item);
        stage_slot(&slots[b->m[b->loc[k]].slot], &S, k, prev);
        const int nvb = MODE == TRACK_GN ? S.grid_gn : S.grid_lap;
        track_item<MODE>(S.P, S.depth, S.rgb, S.o_mask, S.a0, S.a1, S.dev, S.partials, S.pstride, S.counter, S.stats,
                         item - off[k], nvb);
    }
}

// The tiles of every member that are in its new camera's frustum, appended to
// the member's list; item = 256 tiles, one a thread.  Testing every tile of
// every map inside the map update (one thread of a block testing, 255
// waiting) took 201 us with the update for ten streams of 64^3 to 256^3 maps
// (mean of a batch of one and a batch of nine); listed first, this kernel
// takes 6.6 us and the update 59 us.
__global__ void __launch_bounds__(256) kb_cull(const SlotDesc* __restrict__ slots, const BatchDesc* __restrict__ b) {
    pdl_enter();
    __shared__ float sM[9], sb[3];
    const int total = b->cull_off[b->n];
    for (int item = blockIdx.x; item < total; item += gridDim.x) {
        const int i = find_member(b->cull_off, b->n, item);
        const SlotDesc& S = slots[b->m[i].slot];
        load_w2c(S.dev->w2c, sM, sb);
        __syncthreads();
        // a rejected localisation lists no tile: its frame is not fused
        cull_tiles(S.P, sM, sb, (item - b->cull_off[i]) * 256 + (int)threadIdx.x, S.dev->rejected != 0, S.fuse_list,
                   S.P.skip ? S.cells_list : nullptr, S.fuse_count);
        __syncthreads();   // the shared matrices are reused by the next item
    }
}

// Item ranges of the members' lists (which = 0: fuse_list, 1: cells_list): the
// prefix sums of the counts kb_cull left on the device.  Returns the total.
__device__ __forceinline__ int list_offsets(const SlotDesc* __restrict__ slots, const BatchDesc* __restrict__ b, int which,
                                            int* s_off) {
    const int n = b->n;
    if (threadIdx.x < kServeMaxSlots)
        s_off[threadIdx.x + 1] = (int)threadIdx.x < n ? (int)slots[b->m[threadIdx.x].slot].fuse_count[which] : 0;
    __syncthreads();
    if (threadIdx.x == 0) {
        s_off[0] = 0;
        for (int i = 0; i < n; ++i) s_off[i + 1] += s_off[i];
    }
    __syncthreads();
    return s_off[n];
}

// The map update of every member's listed tiles.
template <bool BF16>
__global__ void __launch_bounds__(256, 4) kb_fuse(const SlotDesc* __restrict__ slots, const BatchDesc* __restrict__ b) {
    pdl_enter();
    __shared__ float sM[9], sb[3];
    __shared__ int s_off[kServeMaxSlots + 1];
    __shared__ unsigned int s_count[kServeMaxSlots][2];   // update counts by member
    if (threadIdx.x < 2 * kServeMaxSlots) s_count[threadIdx.x >> 1][threadIdx.x & 1] = 0u;
    const int n = b->n, total = list_offsets(slots, b, 0, s_off);
    __shared__ SlotDesc S;
    int prev = -1;
    for (int item = blockIdx.x; item < total; item += gridDim.x) {
        const int i = find_member(s_off, n, item);
        stage_slot(&slots[b->m[i].slot], &S, i, prev);
        load_w2c(S.dev->w2c, sM, sb);
        __syncthreads();
        fuse_tile<BF16>(S.P, S.M, sM, sb, S.depth, S.rgb, S.o_mask, s_count[i], (uint32_t)S.fuse_list[item - s_off[i]]);
        __syncthreads();   // the shared matrices are reused by the next item
    }
    __syncthreads();
    for (int i = 0; i < n; ++i) add_fuse_counts(slots[b->m[i].slot].stats, s_count[i]);
}

// The brick flags of every member's tiles that may read an updated voxel.
template <bool BF16>
__global__ void __launch_bounds__(256) kb_flags(const SlotDesc* __restrict__ slots, const BatchDesc* __restrict__ b) {
    pdl_enter();
    __shared__ int s_off[kServeMaxSlots + 1];
    const int n = b->n, total = list_offsets(slots, b, 1, s_off);
    for (int item = 2 * blockIdx.x; item < total; item += 2 * gridDim.x) {
        const int j = item + ((int)threadIdx.x >> 7), i = find_member(s_off, n, j < total ? j : item);
        const SlotDesc& S = slots[b->m[i].slot];
        const int tile[1] = {j < total ? S.cells_list[j - s_off[i]] : -1};
        render_detail::brick_flags_tiles<BF16, 1>(S.P, S.M, tile);
    }
}

// The box codes of every member; item = one 32^3 box.
__global__ void __launch_bounds__(256) kb_codes(const SlotDesc* __restrict__ slots, const BatchDesc* __restrict__ b) {
    pdl_enter();
    // the lists have been read: their counts start the next batch at zero
    if (blockIdx.x == 0 && (int)threadIdx.x < b->n) {
        unsigned int* c = slots[b->m[threadIdx.x].slot].fuse_count;
        c[0] = c[1] = 0u;
    }
    const int total = b->box_off[b->n];
    for (int item = blockIdx.x; item < total; item += gridDim.x) {
        const int i = find_member(b->box_off, b->n, item);
        const SlotDesc& S = slots[b->m[i].slot];
        render_detail::box_codes_block(S.P, S.M, item - b->box_off[i]);
    }
}

// The anchor render at each member's new state mean; item = one 16x8 tile.
template <bool BF16>
__global__ void __launch_bounds__(128) kb_render(const SlotDesc* __restrict__ slots, BatchDesc* __restrict__ b,
                                                 int ctr) {
    pdl_enter();
    __shared__ float sR[9], sc[3];
    const int total = b->tiles_off[b->n];
    for (;;) {
        const int item = next_item(&b->ctr[ctr]);
        if (item >= total) break;
        const int i = find_member(b->tiles_off, b->n, item);
        const SlotDesc& S = slots[b->m[i].slot];
        const int t = item - b->tiles_off[i];
        DevState* dev = S.dev;
        if (threadIdx.x < 12) {
            if (threadIdx.x < 9) sR[threadIdx.x] = dev->c2w[threadIdx.x];
            else sc[threadIdx.x - 9] = dev->c2w[threadIdx.x];
        }
        // the state mean (t[3], q[4], contiguous) becomes the anchor's pose
        if (t == 0 && threadIdx.x < 7) dev->anchor_pose[threadIdx.x] = dev->t[threadIdx.x];
        __syncthreads();
        const int tx = t % S.tiles_x, ty = t / S.tiles_x;
        switch (S.px_spec) {
            case 66: render_tile<BF16, false, 66>(S.P, sR, sc, S.M, S.a_depth, S.a_rgb, nullptr, nullptr, S.stats, tx, ty); break;
            case 130: render_tile<BF16, false, 130>(S.P, sR, sc, S.M, S.a_depth, S.a_rgb, nullptr, nullptr, S.stats, tx, ty); break;
            case 258: render_tile<BF16, false, 258>(S.P, sR, sc, S.M, S.a_depth, S.a_rgb, nullptr, nullptr, S.stats, tx, ty); break;
            default: render_tile<BF16, false, 0>(S.P, sR, sc, S.M, S.a_depth, S.a_rgb, nullptr, nullptr, S.stats, tx, ty);
        }
    }
}

// Each member's posterior (and device flags, which are cleared) to `out`.
__global__ void __launch_bounds__(256) kb_out(const SlotDesc* __restrict__ slots, const BatchDesc* __restrict__ b,
                                              ServeOut* __restrict__ out) {
    pdl_enter();
    const int i = blockIdx.x;
    if (i >= b->n) return;
    DevState* d = slots[b->m[i].slot].dev;
    ServeOut& o = out[i];
    for (int e = threadIdx.x; e < 144; e += blockDim.x) o.cov[e] = d->cov[e];
    if (threadIdx.x < 3) {
        o.t[threadIdx.x] = d->t[threadIdx.x];
        o.v[threadIdx.x] = d->v[threadIdx.x];
        o.w[threadIdx.x] = d->w[threadIdx.x];
    }
    if (threadIdx.x < 4) o.q[threadIdx.x] = d->q[threadIdx.x];
    if (threadIdx.x == 0) {
        o.n_localised = d->n_localised;
        o.flags = d->flags;
        d->flags = 0;
    }
}

// ----------------------------------------------------------------- host side
namespace {

template <typename K>
int grid_of(K kern, int threads) {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, threads, 0);
    return (sms > 0 ? sms : 152) * (per > 0 ? per : 1);
}

}  // namespace

int pack_tiles(const KParams& P) { return ((P.W + kPackTW - 1) / kPackTW) * ((P.H + kPackTH - 1) / kPackTH); }

cudaError_t batch_grids(bool bf16, BatchGrids* g) {
    g->pix = grid_of(kb_mask, 256);
    g->pack = grid_of(kb_pack, 256);
    g->codes = grid_of(kb_codes, 256);
    g->flags = bf16 ? grid_of(kb_flags<true>, 256) : grid_of(kb_flags<false>, 256);
    g->track_gn = grid_of(kb_track<TRACK_GN>, Block<TRACK_GN>::threads);
    g->track_lap = grid_of(kb_track<TRACK_LAPLACE>, Block<TRACK_LAPLACE>::threads);
    g->fuse = bf16 ? grid_of(kb_fuse<true>, 256) : grid_of(kb_fuse<false>, 256);
    g->render = bf16 ? grid_of(kb_render<true>, 128) : grid_of(kb_render<false>, 128);
    return cudaGetLastError();
}

cudaError_t launch_batch_step(const SlotDesc* slots, BatchDesc* batch, const double* imu, ServeOut* out, int n_gn,
                              bool bf16, const BatchGrids& g, cudaStream_t s) {
    cudaError_t e;
#define PRISM_BK(call)                        \
    do {                                      \
        if ((e = (call)) != cudaSuccess) return e; \
    } while (0)
    PRISM_BK(launch_pdl(kb_predict, kServeMaxSlots, 256, s, slots, batch, imu));
    PRISM_BK(launch_pdl(kb_mask, g.pix, 256, s, slots, batch));
    for (int it = 0; it < n_gn; ++it) PRISM_BK(launch_pdl(kb_track<TRACK_GN>, g.track_gn, Block<TRACK_GN>::threads, s, slots, batch, it));
    PRISM_BK(launch_pdl(kb_track<TRACK_LAPLACE>, g.track_lap, Block<TRACK_LAPLACE>::threads, s, slots, batch, n_gn));
    PRISM_BK(launch_pdl(kb_cull, g.pix, 256, s, slots, batch));
    if (bf16) PRISM_BK(launch_pdl(kb_fuse<true>, g.fuse, 256, s, slots, batch));
    else PRISM_BK(launch_pdl(kb_fuse<false>, g.fuse, 256, s, slots, batch));
    if (bf16) PRISM_BK(launch_pdl(kb_flags<true>, g.flags, 256, s, slots, batch));
    else PRISM_BK(launch_pdl(kb_flags<false>, g.flags, 256, s, slots, batch));
    PRISM_BK(launch_pdl(kb_codes, g.codes, 256, s, slots, batch));
    if (bf16) PRISM_BK(launch_pdl(kb_render<true>, g.render, 128, s, slots, batch, n_gn + 1));
    else PRISM_BK(launch_pdl(kb_render<false>, g.render, 128, s, slots, batch, n_gn + 1));
    PRISM_BK(launch_pdl(kb_pack, g.pack, 256, s, slots, batch));
    PRISM_BK(launch_pdl(kb_out, kServeMaxSlots, 256, s, slots, batch, out));
#undef PRISM_BK
    return cudaSuccess;
}

}  // namespace prism
