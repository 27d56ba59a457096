// mapio.cu — map initialisation and conversion between the caller's linear
// layout (z-major, x fastest, colour interleaved) and the padded planes
// (a ghost border holding copies of the edge voxels, prism_dev.cuh).
#include "kernels.h"
#include "prism_dev.cuh"
#include "render_dev.cuh"

namespace prism {

template <bool BF16>
__global__ void k_map_fill(KParams P, MapPlanes M, float occ, float rgb, float var, uint32_t n) {
    pdl_enter();
    // n = padded elements per plane; ghosts get the same prior values
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        map_store<BF16>(M.occ, i, occ);
        map_store<BF16>(M.r, i, rgb);
        map_store<BF16>(M.g, i, rgb);
        map_store<BF16>(M.b, i, rgb);
        map_store<BF16>(M.var_occ, i, var);
        map_store<BF16>(M.var_rgb, i, var);
    }
}

// The exchange of maps with the caller goes by segments of 128 voxels of one
// row, one a warp: every load and store is of 32 consecutive elements, all of a
// segment's loads (up to 24 a lane) are issued before the first store, and the
// interleaved colours are taken apart or put together in shared memory (stride
// 3: no bank conflicts).  No access wants more than the element's alignment.
// Bound by HBM: 256^3 voxels out 114 us and in 141 us (with cold caches; 815 MB
// move, 122 us at the measured copy rate) against 167 and 132 us an element a
// thread, with divisions for its coordinates and strided colours; out, in and
// out again 392 us against 601 (361 at the copy rate).  Streaming cache hints
// were slower (407 us).
constexpr int kSeg = 128;

// Every padded element (ghosts included) takes the caller's value of the
// voxel it clamps to: one warp per segment of a padded row; the first and last
// voxel of a row also fill the ghost beside them.
template <bool BF16>
__global__ void __launch_bounds__(256) k_map_load(KParams P, MapPlanes M, const float* __restrict__ occ,
                                                  const float* __restrict__ rgb, const float* __restrict__ vo,
                                                  const float* __restrict__ vr, uint32_t items, uint32_t segs) {
    pdl_enter();
    __shared__ float s_c[8][3 * kSeg];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* sc = s_c[warp];
    for (uint32_t it = blockIdx.x * 8 + warp; it < items; it += gridDim.x * 8) {
        const uint32_t row = it / segs, x0 = (it % segs) * kSeg;
        const int y = min(max((int)(row % P.py) - 1, 0), P.ny - 1), z = min(max((int)(row / P.py) - 1, 0), P.nz - 1);
        const int len = min(kSeg, P.nx - (int)x0);
        const size_t v0 = ((size_t)z * P.ny + y) * P.nx + x0;   // the segment's first voxel
        const uint32_t e0 = row * P.px + x0 + 1;                // and its padded element
        float c[12], o[4], a[4], b[4];
        if (rgb)
#pragma unroll
            for (int j = 0; j < 12; ++j) c[j] = lane + 32 * j < 3 * len ? rgb[3 * v0 + lane + 32 * j] : 0.0f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int x = lane + 32 * j;
            const bool in = x < len;
            o[j] = occ && in ? occ[v0 + x] : 0.0f;
            a[j] = vo && in ? vo[v0 + x] : 0.0f;
            b[j] = vr && in ? vr[v0 + x] : 0.0f;
        }
        if (rgb) {
            __syncwarp();   // the last segment's reads
#pragma unroll
            for (int j = 0; j < 12; ++j) sc[lane + 32 * j] = c[j];
            __syncwarp();
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int x = lane + 32 * j;
            if (x >= len) continue;
            auto put = [&](uint32_t e) {
                if (occ) map_store<BF16>(M.occ, e, o[j]);
                if (rgb) {
                    map_store<BF16>(M.r, e, sc[3 * x]);
                    map_store<BF16>(M.g, e, sc[3 * x + 1]);
                    map_store<BF16>(M.b, e, sc[3 * x + 2]);
                }
                if (vo) map_store<BF16>(M.var_occ, e, a[j]);
                if (vr) map_store<BF16>(M.var_rgb, e, b[j]);
            };
            put(e0 + x);
            if (x0 + x == 0) put(e0 - 1);
            if ((int)x0 + x == P.nx - 1) put(e0 + x + 1);
        }
    }
}

template <bool BF16>
__global__ void __launch_bounds__(256) k_map_store(KParams P, MapPlanes M, float* __restrict__ occ, float* __restrict__ rgb,
                                                   float* __restrict__ vo, float* __restrict__ vr, uint32_t items,
                                                   uint32_t segs) {
    pdl_enter();
    __shared__ float s_c[8][3 * kSeg];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* sc = s_c[warp];
    for (uint32_t it = blockIdx.x * 8 + warp; it < items; it += gridDim.x * 8) {
        const uint32_t row = it / segs, x0 = (it % segs) * kSeg;   // row: y + ny z
        const int len = min(kSeg, P.nx - (int)x0);
        const size_t v0 = (size_t)row * P.nx + x0;
        const uint32_t e0 = pad_index(P, (int)x0, (int)(row % (uint32_t)P.ny), (int)(row / (uint32_t)P.ny));
        float c[3][4], o[4], a[4], b[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int x = lane + 32 * j;
            const bool in = x < len;
            const uint32_t e = e0 + (in ? x : 0);
            if (rgb) {
                c[0][j] = map_load_rw<BF16>(M.r, e);
                c[1][j] = map_load_rw<BF16>(M.g, e);
                c[2][j] = map_load_rw<BF16>(M.b, e);
            }
            o[j] = occ ? map_load_rw<BF16>(M.occ, e) : 0.0f;
            a[j] = vo ? map_load_rw<BF16>(M.var_occ, e) : 0.0f;
            b[j] = vr ? map_load_rw<BF16>(M.var_rgb, e) : 0.0f;
        }
        if (rgb) {
            __syncwarp();   // the last segment's reads
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int k = 0; k < 3; ++k) sc[3 * (lane + 32 * j) + k] = c[k][j];
            __syncwarp();
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int x = lane + 32 * j;
            if (x >= len) continue;
            if (occ) occ[v0 + x] = o[j];
            if (vo) vo[v0 + x] = a[j];
            if (vr) vr[v0 + x] = b[j];
        }
        if (rgb)
#pragma unroll
            for (int j = 0; j < 12; ++j)
                if (lane + 32 * j < 3 * len) rgb[3 * v0 + lane + 32 * j] = sc[lane + 32 * j];
    }
}

// The empty-space index (render_dev.cuh): the brick flags of each 8^3 tile of
// the map or of the listed ones, two a block; then the box codes, one block per
// 32^3 box.
template <bool BF16, int T>
__global__ void __launch_bounds__(256) k_brick_flags(KParams P, MapPlanes M, const int* __restrict__ list,
                                                     const unsigned int* __restrict__ count) {
    pdl_enter();
    const unsigned int all = P.nbx * P.nby * P.nbz, n = list ? min(*count, all) : all;   // (a list has room for all)
    for (unsigned int i = 2 * T * blockIdx.x; i < n; i += 2 * T * gridDim.x) {
        int tile[T];
#pragma unroll
        for (int t = 0; t < T; ++t) {
            const unsigned int j = i + T * (threadIdx.x >> 7) + t;
            tile[t] = j < n ? (list ? list[j] : (int)j) : -1;
        }
        render_detail::brick_flags_tiles<BF16, T>(P, M, tile);
    }
}

__global__ void __launch_bounds__(256) k_box_codes(KParams P, MapPlanes M, unsigned int* ctr) {
    pdl_enter();
    if (ctr && blockIdx.x == 0 && threadIdx.x < 2) ctr[threadIdx.x] = 0u;
    render_detail::box_codes_block(P, M, blockIdx.x);
}

static unsigned int io_grid(uint32_t n) {
    uint32_t g = (n + 255) / 256;
    return g > 152u * 64u ? 152u * 64u : (g ? g : 1u);
}

// Blocks of 8 warps, one segment each (a persistent grid of 152 x 8 blocks was
// slower: 450 us against 412 for the three passes above).
static unsigned int seg_grid(uint32_t items) {
    return (items + 7) / 8;
}

cudaError_t launch_map_fill(const KParams& P, const MapPlanes& M, float occ, float rgb, float var, cudaStream_t s) {
    uint32_t n = P.npad;
    if (P.bf16) launch_pdl(k_map_fill<true>, io_grid(n), 256, s, P, M, occ, rgb, var, n);
    else launch_pdl(k_map_fill<false>, io_grid(n), 256, s, P, M, occ, rgb, var, n);
    return cudaGetLastError();
}

cudaError_t launch_map_load(const KParams& P, const MapPlanes& M, const float* occ, const float* rgb,
                            const float* var_occ, const float* var_rgb, cudaStream_t s) {
    const uint32_t segs = (uint32_t)(P.nx + kSeg - 1) / kSeg, items = P.npad / P.px * segs;
    if (P.bf16) launch_pdl(k_map_load<true>, seg_grid(items), 256, s, P, M, occ, rgb, var_occ, var_rgb, items, segs);
    else launch_pdl(k_map_load<false>, seg_grid(items), 256, s, P, M, occ, rgb, var_occ, var_rgb, items, segs);
    return cudaGetLastError();
}

cudaError_t launch_map_store(const KParams& P, const MapPlanes& M, float* occ, float* rgb, float* var_occ,
                             float* var_rgb, cudaStream_t s) {
    const uint32_t segs = (uint32_t)(P.nx + kSeg - 1) / kSeg, items = (uint32_t)P.ny * P.nz * segs;
    if (P.bf16) launch_pdl(k_map_store<true>, seg_grid(items), 256, s, P, M, occ, rgb, var_occ, var_rgb, items, segs);
    else launch_pdl(k_map_store<false>, seg_grid(items), 256, s, P, M, occ, rgb, var_occ, var_rgb, items, segs);
    return cudaGetLastError();
}

// A frame in pinned host memory that the device maps (s0, s1: device views of
// it) copied by the SMs' own loads: n0 floats s0 -> d0, n1 floats s1 -> d1.
// Each thread has four 16-byte loads in flight per round (the host memory's
// latency is the bound); single floats where an address is not 16-byte
// aligned, and for the tail.
__global__ void __launch_bounds__(256) k_frame_upload(const float* __restrict__ s0, float* __restrict__ d0,
                                                      size_t n0, const float* __restrict__ s1,
                                                      float* __restrict__ d1, size_t n1) {
    pdl_enter();
    const size_t tid = (size_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
    const float* src[2] = {s0, s1};
    float* dst[2] = {d0, d1};
    const size_t cnt[2] = {n0, n1};
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        const float* s = src[a];
        float* d = dst[a];
        const size_t n = cnt[a];
        size_t done = 0;
        if (((reinterpret_cast<uintptr_t>(s) | reinterpret_cast<uintptr_t>(d)) & 15) == 0) {
            const size_t nv = n / 4;
            const float4* s4 = reinterpret_cast<const float4*>(s);
            float4* d4 = reinterpret_cast<float4*>(d);
            size_t i = tid;
            for (; i + 3 * stride < nv; i += 4 * stride) {
                const float4 x0 = s4[i], x1 = s4[i + stride], x2 = s4[i + 2 * stride], x3 = s4[i + 3 * stride];
                d4[i] = x0;
                d4[i + stride] = x1;
                d4[i + 2 * stride] = x2;
                d4[i + 3 * stride] = x3;
            }
            for (; i < nv; i += stride) d4[i] = s4[i];
            done = nv * 4;
        }
        for (size_t i = done + tid; i < n; i += stride) d[i] = s[i];
    }
}

cudaError_t launch_frame_upload(const float* s0, float* d0, size_t n0, const float* s1, float* d1, size_t n1,
                                int blocks, cudaStream_t s) {
    k_frame_upload<<<blocks, 256, 0, s>>>(s0, d0, n0, s1, d1, n1);
    return cudaGetLastError();
}

cudaError_t launch_brick_flags(const KParams& P, const MapPlanes& M, const int* list, const unsigned int* count,
                               cudaStream_t s) {
    // One tile for each half of a block where latency counts: after a map update,
    // whose list is a few waves at most (an update 15.0 us against 15.5 with two at
    // 128^3, 15.9 against 17.4 at 160^3, 25.0 against 26.9 at 256^3), and over a whole
    // map of up to 160^3 voxels (a load of its occupancy 13.6 against 14.4 at 128^3,
    // 25.3 against 25.4 at 160^3).  Two over a larger map, where the rate counts (36.9
    // against 36.0 at 192^3, 79.3 against 76.3 at 256^3).
    const int tiles = P.nbx * P.nby * P.nbz;
    auto go = [&](auto kern, int per) {
        const int need = (tiles + per - 1) / per;
        return launch_pdl(kern, need < 152 * 8 || !list ? need : 152 * 8, 256, s, P, M, list, count);
    };
    if (list || tiles <= 8000) return P.bf16 ? go(k_brick_flags<true, 1>, 2) : go(k_brick_flags<false, 1>, 2);
    return P.bf16 ? go(k_brick_flags<true, 2>, 4) : go(k_brick_flags<false, 2>, 4);
}

cudaError_t launch_box_codes(const KParams& P, const MapPlanes& M, unsigned int* ctr, cudaStream_t s) {
    return launch_pdl(k_box_codes, P.ntx * P.nty * P.ntz, 256, s, P, M, ctr);
}

cudaError_t launch_map_index(const KParams& P, const MapPlanes& M, cudaStream_t s) {
    cudaError_t e = launch_brick_flags(P, M, nullptr, nullptr, s);
    return e != cudaSuccess ? e : launch_box_codes(P, M, nullptr, s);
}

}  // namespace prism
