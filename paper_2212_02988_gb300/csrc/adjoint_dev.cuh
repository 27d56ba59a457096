// adjoint_dev.cuh — device body of the render adjoint of App. B (the emission
// is differentiable), shared by the adjoint itself (render_bwd.cu) and the
// descent step on the map (mapping.cu): gradients of L with respect to the
// occupancy and colour means and to a world-frame perturbation of the camera
// pose (t' = t + dt, R' = Exp(dtheta) R).
//
// Nothing is stored by the forward: each ray is marched again (the forward's
// march, so it finds the same hit sample k) and then, with
// alpha = (tau - f0) / (f1 - f0) between samples k-1 and k,
//   dL/dalpha = gD eps / |dir_c| + sum_c gC_c (C_c(p_k) - C_c(p_{k-1})),
//   dL/df0 = dL/dalpha (alpha - 1) / (f1 - f0),  dL/df1 = -dL/dalpha alpha / (f1 - f0),
// each value's gradient goes to its 8 trilinear corners (FP32 atomics, the
// caller's linear map layout, edge corners clamped), and the pose gradient
// through the sample positions p_s = c + d_s r:
// dL/dt += gp_s, dL/dtheta += d_s (r x gp_s), gp_s = dL/dp_s.
//
// What bounds it: the march (as the render; before the empty-space index the
// adjoint evaluated every sample of a ray), then the atomics:
// 2 samples x 8 corners x 4 values a hit.  A warp's 8x4 pixels see one or two
// voxels, so most of those meet in a few cells: the warp sums them cell by
// cell (warp_reduce_scatter32) and adds each cell's 32 values with one atomic
// instruction.  640x480 on a 256^3 map: 487 us -> 66 us; 320x240 on 128^3: 98 us
// -> 29 us (54 us with the march alone and an atomic for each value; the same
// to the noise for 6, 12 or 24 cells).
#pragma once

#include "kernels.h"
#include "prism_dev.cuh"
#include "render_dev.cuh"

namespace prism {

namespace adjoint_detail {

using render_detail::Sample;

// The 8 corner values of a cell from a padded plane, order (x, y, z) bits.
template <bool BF16>
__device__ __forceinline__ void corners(const KParams& P, const void* plane, uint32_t base, float v[8]) {
    const uint32_t b1 = base + P.px, b2 = base + P.pxy, b3 = b2 + P.px;
    v[0] = map_load<BF16>(plane, base); v[1] = map_load<BF16>(plane, base + 1);
    v[2] = map_load<BF16>(plane, b1);   v[3] = map_load<BF16>(plane, b1 + 1);
    v[4] = map_load<BF16>(plane, b2);   v[5] = map_load<BF16>(plane, b2 + 1);
    v[6] = map_load<BF16>(plane, b3);   v[7] = map_load<BF16>(plane, b3 + 1);
}

// Trilinear value (the forward's lerp order) and its gradient in cell units.
__device__ __forceinline__ float tri_value_grad(const float v[8], float fx, float fy, float fz, float g[3]) {
    const float c00 = lerp_rn(v[0], v[1], fx), c10 = lerp_rn(v[2], v[3], fx);
    const float c01 = lerp_rn(v[4], v[5], fx), c11 = lerp_rn(v[6], v[7], fx);
    const float c0 = lerp_rn(c00, c10, fy), c1 = lerp_rn(c01, c11, fy);
    const float dx00 = v[1] - v[0], dx10 = v[3] - v[2], dx01 = v[5] - v[4], dx11 = v[7] - v[6];
    g[0] = lerp_rn(lerp_rn(dx00, dx10, fy), lerp_rn(dx01, dx11, fy), fz);
    g[1] = lerp_rn(c10 - c00, c11 - c01, fz);
    g[2] = c1 - c0;
    return lerp_rn(c0, c1, fz);
}

// Index in the caller's linear layout of corner c (bits x, y, z) of the cell
// with lower corner (ix, iy, iz), clamped to the grid.
__device__ __forceinline__ size_t corner_index(const KParams& P, int ix, int iy, int iz, int c) {
    const int x = min(max(ix + (c & 1), 0), P.nx - 1), y = min(max(iy + ((c >> 1) & 1), 0), P.ny - 1),
              z = min(max(iz + (c >> 2), 0), P.nz - 1);
    return ((size_t)z * P.ny + y) * P.nx + x;
}

// The trilinear weights of a cell's corners.
__device__ __forceinline__ void weights(const Sample& s, float w[8]) {
#pragma unroll
    for (int c = 0; c < 8; ++c)
        w[c] = (c & 1 ? s.fx : 1.0f - s.fx) * (c & 2 ? s.fy : 1.0f - s.fy) * (c & 4 ? s.fz : 1.0f - s.fz);
}

// One sample's gradient values g (occupancy, colours) added to its corners.
__device__ __forceinline__ void scatter(const KParams& P, float* g_occ, float* g_rgb, const Sample& s, const float g[4]) {
    float w[8];
    weights(s, w);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const size_t i = corner_index(P, s.ix, s.iy, s.iz, c);
        if (g_occ) atomicAdd(g_occ + i, g[0] * w[c]);
        if (g_rgb)
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) atomicAdd(g_rgb + 3 * i + ch, g[1 + ch] * w[c]);
    }
}

// Cells a warp sums before the rest of its samples go out one by one: a cell
// costs ~250 instructions, a lone sample 32 atomics.
constexpr int kCells = 12;

// The gradients of the warp's hits (on: this lane has one; samples s[0], s[1]
// with values g[0], g[1]) added to the map gradients.  Every lane calls it.
__device__ __forceinline__ void warp_scatter(const KParams& P, float* g_occ, float* g_rgb, bool on, const Sample s[2],
                                             const float g[2][4]) {
    const int lane = threadIdx.x & 31;
    uint32_t left[2];   // lanes whose sample is still to be added
    left[0] = left[1] = __ballot_sync(0xffffffffu, on);
    // this lane's value of a cell: 0..7 occupancy of corner `lane`; 8 + 6 (y + 2 z) + 3 x + channel
    const int q = lane - 8, row = q / 6, corner = lane < 8 ? lane : ((q % 6) / 3) | (row << 1), ch = q % 3;
    float w[2][8];
    weights(s[0], w[0]);
    weights(s[1], w[1]);
    for (int it = 0; it < kCells && (left[0] | left[1]); ++it) {
        const int j = left[0] ? 0 : 1, leader = __ffs(left[j]) - 1;
        const int ix = __shfl_sync(0xffffffffu, s[j].ix, leader), iy = __shfl_sync(0xffffffffu, s[j].iy, leader),
                  iz = __shfl_sync(0xffffffffu, s[j].iz, leader);
        float v[32];
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = 0.0f;
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const bool in = on && s[m].ix == ix && s[m].iy == iy && s[m].iz == iz;
            left[m] &= ~__ballot_sync(0xffffffffu, in);
            float h[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) h[k] = in ? g[m][k] : 0.0f;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const float wc = in ? w[m][c] : 0.0f;
                v[c] = fmaf(h[0], wc, v[c]);
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    float& t = v[8 + 6 * (c >> 1) + 3 * (c & 1) + k];
                    t = fmaf(h[1 + k], wc, t);
                }
            }
        }
        warp_reduce_scatter32(v);
        const size_t i = corner_index(P, ix, iy, iz, corner);
        float* dst = lane < 8 ? (g_occ ? g_occ + i : nullptr) : (g_rgb ? g_rgb + 3 * i + ch : nullptr);
        if (dst) atomicAdd(dst, v[0]);
    }
#pragma unroll
    for (int m = 0; m < 2; ++m)
        if ((left[m] >> lane) & 1u) scatter(P, g_occ, g_rgb, s[m], g[m]);
}

}  // namespace adjoint_detail

// One 16x8-pixel tile (128 threads).  `loss` supplies the gradients: want(p)
// says whether pixel p's ray is needed, get(p, d, c, gd, gc) gives
// dL/d(depth) and dL/d(colour) of a hit rendered as (d, c) (passed only if
// Loss::kImage) and returns whether any of them is not zero.  gpose: this
// thread's pose gradient (added to; of use only where get returns true for
// every ray wanted).  Returns the
// thread's hit sample index (0: none).
template <bool BF16, bool DETAIL, int PX, class Loss>
__device__ __forceinline__ int adjoint_tile(const KParams& P, const float* sR, const float* sc, const MapPlanes& M,
                                             Loss& loss, float* g_occ, float* g_rgb, float gpose[6], int& nsamp,
                                             unsigned int& uniq, int tile_x, int tile_y) {
    using namespace render_detail;
    using namespace adjoint_detail;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int u = tile_x * 16 + (warp & 1) * 8 + (lane & 7);
    const int v = tile_y * 8 + (warp >> 1) * 4 + (lane >> 3);
    const uint32_t px = PX > 0 ? (uint32_t)PX : P.px;
    const uint32_t pxy = PX > 0 ? (uint32_t)(PX * PX) : P.pxy;
    const int p = v * P.W + u;
    const bool want = u < P.W && v < P.H && loss.want(p);
    if (!__any_sync(0xffffffffu, want)) return 0;
    const Ray r = ray_of(P, sR, sc, u, v);
    const float k0 = P.skip && M.boxes != nullptr
                         ? beam_start(P, M, sR, r, (float)(tile_x * 16 + (warp & 1) * 8) + 3.5f,
                                      (float)(tile_y * 8 + (warp >> 1) * 4) + 1.5f)
                         : 1.0f;
    int steps = 0;
    const MarchHit h = march<BF16, DETAIL, PX>(P, M, r, want, k0, nsamp, steps, uniq);
    Sample s[2];
    float g[2][4] = {{0.0f, 0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f, 0.0f}};
    s[0] = s[1] = Sample{0u, 0.0f, 0.0f, 0.0f, 0, 0, 0};
    bool on = want && h.k >= 2;
    if (on) {
        float ds[2];
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            ds[m] = __fmul_rn((float)(h.k - 1 + m), P.eps32);
            s[m] = cell_of(px, pxy, __fmaf_rn(ds[m], r.rgx, r.cgx), __fmaf_rn(ds[m], r.rgy, r.cgy),
                           __fmaf_rn(ds[m], r.rgz, r.cgz));
        }
        on = PRISM_IN_RANGE(P, CHK_BWD_CORNER, (long long)s[0].base + P.pxy + P.px + 1, P.npad) &&
             PRISM_IN_RANGE(P, CHK_BWD_CORNER, (long long)s[1].base + P.pxy + P.px + 1, P.npad);
        if (on) {
            float vo[8], go[2][3], f[2];
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                corners<BF16>(P, M.occ, s[m].base, vo);
                f[m] = tri_value_grad(vo, s[m].fx, s[m].fy, s[m].fz, go[m]);
            }
            const float alpha = (P.tau32 - f[0]) / (f[1] - f[0]);
            const void* planes[3] = {M.r, M.g, M.b};
            float col[2][3], gcol[2][3][3];
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    float vc[8];
                    corners<BF16>(P, planes[c], s[m].base, vc);
                    col[m][c] = tri_value_grad(vc, s[m].fx, s[m].fy, s[m].fz, gcol[m][c]);
                }
            float gd = 0.0f, gc[3] = {0.0f, 0.0f, 0.0f};
            {   // the render's depth and colour
                float d = 0.0f, c[3] = {0.0f, 0.0f, 0.0f};
                if (Loss::kImage) {
                    d = fmaf(alpha, ds[1] - ds[0], ds[0]) * r.inv_n;
#pragma unroll
                    for (int k = 0; k < 3; ++k) c[k] = fmaf(alpha, col[1][k] - col[0][k], col[0][k]);
                }
                // (a ray that takes no part is not scattered: its zero gradient times a map
                // value or slope that is not finite is NaN)
                on = loss.get(p, d, c, gd, gc);
            }
            float gA = gd * (ds[1] - ds[0]) * r.inv_n;
            for (int c = 0; c < 3; ++c) gA += gc[c] * (col[1][c] - col[0][c]);
            const float inv_df = 1.0f / (f[1] - f[0]);
            const float gf[2] = {gA * (alpha - 1.0f) * inv_df, -gA * alpha * inv_df};
            const float wa[2] = {1.0f - alpha, alpha};
            const float rr[3] = {r.rx, r.ry, r.rz};
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                g[m][0] = gf[m];
#pragma unroll
                for (int c = 0; c < 3; ++c) g[m][1 + c] = gc[c] * wa[m];
                float gp[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    gp[a] = gf[m] * go[m][a];
#pragma unroll
                    for (int c = 0; c < 3; ++c) gp[a] += gc[c] * wa[m] * gcol[m][c][a];
                    gp[a] *= P.inv_vs32;
                }
                // dL/dt += gp; dL/dtheta += d (r x gp)
                gpose[0] += gp[0]; gpose[1] += gp[1]; gpose[2] += gp[2];
                gpose[3] += ds[m] * (rr[1] * gp[2] - rr[2] * gp[1]);
                gpose[4] += ds[m] * (rr[2] * gp[0] - rr[0] * gp[2]);
                gpose[5] += ds[m] * (rr[0] * gp[1] - rr[1] * gp[0]);
            }
        }
    }
    __syncwarp();
    if (g_occ || g_rgb) warp_scatter(P, g_occ, g_rgb, on, s, g);
    return h.k;
}

}  // namespace prism
