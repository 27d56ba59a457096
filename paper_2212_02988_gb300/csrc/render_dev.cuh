// render_dev.cuh — device bodies of the map-mean render of App. B and of the
// anchor it leaves for the localisation (App. E.3, App. F.3), shared by the
// single-stream kernels (render.cu) and the batched serving kernels
// (serve_kernels.cu).
//
// The render: one thread per pixel, 16x8-pixel blocks of 4 warps, each warp an
// 8x4 pixel tile so that a warp's rays stay close and their trilinear cells
// share cache lines.  Each ray marches d_k = k eps, k = 1, 2, ... through the
// occupancy plane (8 gathered corners per sample, FP32 lerps) and
// stops at the first sample with occupancy > tau (reading R1) or at the first
// sample outside the grid (R5).  The occupancy plane is linear with a ghost
// border (prism_dev.cuh), so a sample costs 8 loads at fixed offsets from
// one base index.  The hit depth and colour are the alpha
// interpolation between samples k-1 and k (App. B, R7); the colour planes are
// read only there.  The decision arithmetic follows the documented FP32
// recipe with explicitly rounded intrinsics (no contraction), so sample
// positions, corner indices and hit indices are reproducible bit for bit.
#pragma once

#include "kernels.h"
#include "prism_dev.cuh"

namespace prism {

namespace render_detail {

// Trilinear value at a cell given by its padded base index and in-cell
// weights: lerps along x, then y, then z (the FP32 recipe).  With PX > 0 the
// plane strides are compile-time constants (cubic grids of PX - 2 voxels a
// side), so the 8 loads are immediate offsets from one address.
template <bool BF16, int PX>
__device__ __forceinline__ float trilinear(const void* plane, uint32_t base, uint32_t px_rt, uint32_t pxy_rt,
                                           float fx, float fy, float fz) {
    const uint32_t px = PX > 0 ? (uint32_t)PX : px_rt;
    const uint32_t pxy = PX > 0 ? (uint32_t)(PX * PX) : pxy_rt;
    float v000, v100, v010, v110, v001, v101, v011, v111;
    if constexpr (BF16) {
        const __nv_bfloat16* q = reinterpret_cast<const __nv_bfloat16*>(plane) + base;
        v000 = __bfloat162float(__ldg(q)); v100 = __bfloat162float(__ldg(q + 1));
        v010 = __bfloat162float(__ldg(q + px)); v110 = __bfloat162float(__ldg(q + px + 1));
        v001 = __bfloat162float(__ldg(q + pxy)); v101 = __bfloat162float(__ldg(q + pxy + 1));
        v011 = __bfloat162float(__ldg(q + pxy + px)); v111 = __bfloat162float(__ldg(q + pxy + px + 1));
    } else {
        const float* q = reinterpret_cast<const float*>(plane) + base;
        v000 = __ldg(q); v100 = __ldg(q + 1);
        v010 = __ldg(q + px); v110 = __ldg(q + px + 1);
        v001 = __ldg(q + pxy); v101 = __ldg(q + pxy + 1);
        v011 = __ldg(q + pxy + px); v111 = __ldg(q + pxy + px + 1);
    }
    const float c00 = lerp_rn(v000, v100, fx);
    const float c10 = lerp_rn(v010, v110, fx);
    const float c01 = lerp_rn(v001, v101, fx);
    const float c11 = lerp_rn(v011, v111, fx);
    const float c0 = lerp_rn(c00, c10, fy);
    const float c1 = lerp_rn(c01, c11, fy);
    return lerp_rn(c0, c1, fz);
}

// Sample k of a ray in grid units: position g = fma(k eps, rg, cg), lower
// cell corner floor(g) as a padded base index, in-cell weights g - floor(g).
struct Sample {
    uint32_t base;
    float fx, fy, fz;
    int ix, iy, iz;   // lower corner (x0, y0, z0), x0 in [-1, n - 1]
};

// floor(g) for |g| < 2^22 without a conversion instruction: adding
// 1.5 * 2^23 with rounding toward -inf leaves floor(g) in the low mantissa
// bits (the sum's ulp is 1), and subtracting it back is exact.
constexpr float kFloorMagic = 12582912.0f;   // 1.5 * 2^23
constexpr uint32_t kFloorMagicBits = 0x4B400000u;

__device__ __forceinline__ Sample cell_of(uint32_t px, uint32_t pxy, float gx, float gy, float gz) {
    const float tx = __fadd_rd(gx, kFloorMagic), ty = __fadd_rd(gy, kFloorMagic), tz = __fadd_rd(gz, kFloorMagic);
    Sample s;
    s.fx = __fsub_rn(gx, __fsub_rn(tx, kFloorMagic));
    s.fy = __fsub_rn(gy, __fsub_rn(ty, kFloorMagic));
    s.fz = __fsub_rn(gz, __fsub_rn(tz, kFloorMagic));
    // (x0 + 1) + px ((y0 + 1) + py (z0 + 1)) with x0 = bits(tx) - magic, ...
    // in wrapping 32-bit arithmetic; the constant folds the offsets.
    const uint32_t c = (1u - kFloorMagicBits) * (1u + px + pxy);
    s.base = __float_as_uint(tx) + px * __float_as_uint(ty) + pxy * __float_as_uint(tz) + c;
    s.ix = (int)(__float_as_uint(tx) - kFloorMagicBits);
    s.iy = (int)(__float_as_uint(ty) - kFloorMagicBits);
    s.iz = (int)(__float_as_uint(tz) - kFloorMagicBits);
    return s;
}

// The empty-space index.  A trilinear value is a convex combination of its 8
// corners, so a cell whose largest corner is below tau by more than the
// lerps' rounding (7 lerps, each within ~3 2^-24 of the corners' magnitude:
// 2^-18 (1 + max |corner|) is a safe margin) holds no sample that can be a
// hit.  The index is 16 bits per 8^3 box of cells (those whose lower corner
// lies in [8 b, 8 b + 8) per axis; a lower corner of -1 reads voxel 0 only,
// which cell 0 reads too, and goes with cell 0):
//   bits 0-7   the 4^3 bricks of the box with a cell that may hold a hit;
//   bits 8-9   where there are none: c = 1, 2 or 3 for the largest aligned box
//              around it, 4 2^c = 8, 16 or 32 cells a side, without any;
//   bit 10     open: neither this box nor its 26 neighbours have any.
// 64 KB for 256^3 voxels, 32 bytes for 32x32x8 of them (box_index): the rays'
// lookups hit L1.
//
// How a warp's 32 rays use it.  First the warp goes together along the tile's
// centre ray, each lane testing one distance for open boxes (beam_start): one
// or two loads take all rays past the free space in front of the camera.
// Then each ray jumps out of empty boxes and bricks on one load a jump, and
// evaluates the samples in the remaining bricks, three at a time.  With 4^3
// bounds of floats and three coarser levels of them (2.4 MB, two dependent
// loads a jump), rays one by one from the camera, a call of 320 frames (640x480,
// 256^3 map) took 15.2 ms and a frame alone 66 us; now 8.7 ms and 44.5 us.
constexpr uint32_t kBoxOpen = 1u << 10;

// The word of box (x, y, z): the 4x4x4 boxes of a 32^3 box are consecutive.
__device__ __forceinline__ int box_index(const KParams& P, int x, int y, int z) {
    return 64 * ((x >> 2) + P.ntx * ((y >> 2) + P.nty * (z >> 2))) + ((x & 3) | ((y & 3) << 2) | ((z & 3) << 4));
}

// The flags of the 8 bricks of 2 T 8^3 tiles (256 threads, T tiles for each 128;
// a negative tile: none): a brick's cells read the 5^3 voxels from its lowest
// one on, and it may hold a hit unless the largest of them is below tau as
// above.  Warp w of a tile's four takes the layers z = 2 w .. 2 w + 2; its lane
// l < 27 reads voxel x = l % 9 of the rows y = 3 i + l / 9: 9 T loads in flight
// a lane.  Latency bound: 4.2 us for 512 tiles, 8.8 us for the ~3,400 of a
// 640x480 step, 36 us for the 32,768 of a 256^3 map (T = 1; a tile a block
// through shared memory: 4.3, 10.3 and 75 us; a tile a warp: 9.4, 10.8 and 43).
template <bool BF16, int T>
__device__ __forceinline__ void brick_flags_tiles(const KParams& P, const MapPlanes& M, const int (&tile)[T]) {
    __shared__ float2 s_b[2][T][4][4];   // [half][tile][warp][brick x + 2 y]: largest value and magnitude
    const int half = threadIdx.x >> 7, w = (threadIdx.x >> 5) & 3, lane = threadIdx.x & 31;
    const int l = lane < 27 ? lane : 26, x = l % 9, y0 = l / 9;
    float v[T][9];
    bool on[T];
#pragma unroll
    for (int t = 0; t < T; ++t) {
        on[t] = tile[t] >= 0 && PRISM_IN_RANGE(P, CHK_FUSE_TILE, tile[t], (long long)P.nbx * P.nby * P.nbz);
        const int q = on[t] ? tile[t] : 0, bx = q % P.nbx, by = (q / P.nbx) % P.nby, bz = q / (P.nbx * P.nby);
        const uint32_t base = pad_index(P, 8 * bx + x, 8 * by + y0, 8 * bz + 2 * w);
#pragma unroll
        for (int i = 0; i < 9; ++i) v[t][i] = map_load_rw<BF16>(M.occ, base + P.px * (3u * (i % 3)) + P.pxy * (i / 3));
    }
#pragma unroll
    for (int t = 0; t < T; ++t)
#pragma unroll
        for (int q = 0; q < 2; ++q) {   // y: 0 .. 4 (rows 3 r + y0), then 4 .. 8
            float m = -INFINITY, a = 0.0f;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const int r = i % 3;
                if (r == (q == 0 ? 2 : 0)) continue;
                const bool in = r != 1 || (q == 0 ? y0 <= 1 : y0 >= 1);
                m = fmaxf(m, in ? v[t][i] : -INFINITY);
                a = fmaxf(a, in ? fabsf(v[t][i]) : 0.0f);
            }
            // over the lanes' rows (l, l + 9, l + 18), then x = 0 .. 4 into lane 0 and 4 .. 8 into lane 4
            auto reduce = [&](float z) {
                const float r1 = __shfl_down_sync(0xffffffffu, z, 9), r2 = __shfl_down_sync(0xffffffffu, z, 18);
                z = fmaxf(fmaxf(z, r1), r2);
                const float s1 = fmaxf(z, __shfl_down_sync(0xffffffffu, z, 1));
                const float s2 = fmaxf(s1, __shfl_down_sync(0xffffffffu, s1, 2));
                return fmaxf(s2, __shfl_down_sync(0xffffffffu, z, 4));
            };
            m = reduce(m);
            a = reduce(a);
            if (lane == 0 || lane == 4) s_b[half][t][w][(lane >> 2) + 2 * q] = make_float2(m, a);
        }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < T; ++t)
        if (w == t) {   // lane: brick x + 2 y + 4 z
            const float2 b0 = s_b[half][t][2 * ((lane >> 2) & 1)][lane & 3], b1 = s_b[half][t][2 * ((lane >> 2) & 1) + 1][lane & 3];
            const uint32_t f = __ballot_sync(0xffffffffu, !(fmaxf(b0.x, b1.x) < P.tau32 - 0x1p-18f * (1.0f + fmaxf(b0.y, b1.y))));
            if (lane == 0 && on[t]) M.bricks[tile[t]] = (uint8_t)(f & 0xffu);
        }
    __syncthreads();   // s_b is reused by the next tiles
}

// The words of the 64 boxes of one 32^3 box, one 256-thread block: the flags
// of the 6^3 boxes around them go through shared memory; boxes past the map's
// edge count as empty.
__device__ __forceinline__ void box_codes_block(const KParams& P, const MapPlanes& M, int top) {
    __shared__ uint8_t s_f[6][6][6];   // [z][y][x], the 32^3 box's own at 1 .. 4
    __shared__ int s_all[2];
    const int t = threadIdx.x;
    const int x0 = 4 * (top % P.ntx), y0 = 4 * ((top / P.ntx) % P.nty), z0 = 4 * (top / (P.ntx * P.nty));
    if (t < 216) {
        const int i = t % 6, j = (t / 6) % 6, k = t / 36, x = x0 + i - 1, y = y0 + j - 1, z = z0 + k - 1;
        s_f[k][j][i] = x >= 0 && x < P.nbx && y >= 0 && y < P.nby && z >= 0 && z < P.nbz
                           ? M.bricks[x + P.nbx * (y + P.nby * z)] : (uint8_t)0;
    }
    __syncthreads();
    uint32_t f = 0u, near = 0u;
    int e1 = 0, e2 = 0;
    if (t < 64) {   // box (t & 3, (t >> 2) & 3, t >> 4)
        const int i = t & 3, j = (t >> 2) & 3, k = t >> 4;
        f = s_f[k + 1][j + 1][i + 1];
#pragma unroll
        for (int c = 0; c < 27; ++c) near |= s_f[k + c / 9][j + (c / 3) % 3][i + c % 3];
        e1 = f == 0u;
        e2 = e1 & __shfl_xor_sync(0xffffffffu, e1, 1);   // the 2x2x2 boxes of its 16^3 box
        e2 &= __shfl_xor_sync(0xffffffffu, e2, 4);
        e2 &= __shfl_xor_sync(0xffffffffu, e2, 16);
        const int all = __all_sync(0xffffffffu, e1);
        if ((t & 31) == 0) s_all[t >> 5] = all;
    }
    __syncthreads();
    if (t < 64) {
        const uint32_t code = e1 ? (e2 ? (s_all[0] & s_all[1] ? 3u : 2u) : 1u) : 0u;
        M.boxes[64 * (size_t)top + t] = (uint16_t)(f | (code << 8) | (near == 0u ? kBoxOpen : 0u));
    }
    __syncthreads();   // the shared flags are reused by the block's next item
}

// A ray in grid units: sample position g = fma(d, rg, cg), d = k eps.
struct Ray {
    float rx, ry, rz;      // unit world direction
    float rgx, rgy, rgz, cgx, cgy, cgz;
    float inv_n;           // 1 / |dir_c|
};

// The ray of pixel (u, v) (the FP32 recipe).
__device__ __forceinline__ Ray ray_of(const KParams& P, const float* sR, const float* sc, int u, int v) {
    Ray r;
    const float dx = __fmul_rn(__fsub_rn((float)u, P.cx32), P.ifx32);
    const float dy = __fmul_rn(__fsub_rn((float)v, P.cy32), P.ify32);
    const float w0 = __fmaf_rn(sR[0], dx, __fmaf_rn(sR[1], dy, sR[2]));
    const float w1 = __fmaf_rn(sR[3], dx, __fmaf_rn(sR[4], dy, sR[5]));
    const float w2 = __fmaf_rn(sR[6], dx, __fmaf_rn(sR[7], dy, sR[8]));
    r.inv_n = __fdiv_rn(1.0f, __fsqrt_rn(__fmaf_rn(w0, w0, __fmaf_rn(w1, w1, __fmul_rn(w2, w2)))));
    r.rx = __fmul_rn(w0, r.inv_n);
    r.ry = __fmul_rn(w1, r.inv_n);
    r.rz = __fmul_rn(w2, r.inv_n);
    r.rgx = __fmul_rn(r.rx, P.inv_vs32);
    r.rgy = __fmul_rn(r.ry, P.inv_vs32);
    r.rgz = __fmul_rn(r.rz, P.inv_vs32);
    r.cgx = __fmaf_rn(__fsub_rn(sc[0], P.o32[0]), P.inv_vs32, -0.5f);
    r.cgy = __fmaf_rn(__fsub_rn(sc[1], P.o32[1]), P.inv_vs32, -0.5f);
    r.cgz = __fmaf_rn(__fsub_rn(sc[2], P.o32[2]), P.inv_vs32, -0.5f);
    return r;
}

// One axis of a brick exit: the plane of the box's far side along the ray is
// lo + s e + m (s = 1, m = -1e-3 for a positive direction; s = 0, m = 1e-3
// for a negative one: pulled 1e-3 voxels inside, far above the rounding of
// the sample positions and of the quotient; a zero direction: never), its
// distance in samples (lo + s e + (m - cg)) / (rg eps).
struct ExitAxis {
    float s, c, ir;   // s; m - cg; 1 / (rg eps)
    __device__ __forceinline__ ExitAxis(float rg, float cg, float ieps) {
        s = rg > 0.0f ? 1.0f : 0.0f;
        c = (rg > 0.0f ? -1e-3f : (rg < 0.0f ? 1e-3f : 1e30f)) - cg;
        ir = rg != 0.0f ? ieps / rg : 1.0f;
    }
    // bits: the cell coordinate + kFloorMagicBits, clear: the bits below the box's
    // edge, ef: the edge
    __device__ __forceinline__ float dist(uint32_t bits, uint32_t clear, float ef) const {
        const float lo = __uint_as_float(bits & ~clear) - kFloorMagic;   // exact
        return (fmaf(s, ef, lo) + c) * ir;
    }
};

// The sample index from which the 32 rays of a warp (all lanes call it, rays
// or not) have to be marched: every sample before it lies in an open box or a
// neighbour of one.  Lane j of a round tests the middle of the piece [j, j + 1)
// S of the centre ray (unit direction rc), S = 8 voxels: a point of the piece
// is at most 4 voxels from its middle on any axis, a ray's sample at the same
// distance at most delta (j + 1) S more (delta: the largest difference of a
// lane's direction from rc on any axis), together below the 8 voxels that an
// open box has around it (0.1 voxel of margin, far above the rounding).  The
// centre must be one voxel inside the grid (cg in [0.5, h - 1]): no sample
// before the returned one has then left the grid and come back.
__device__ __forceinline__ float beam_start(const KParams& P, const MapPlanes& M, const float* sR, const Ray& r, float uc,
                                          float vc) {
    const float hx = (float)P.nx - 1.5f, hy = (float)P.ny - 1.5f, hz = (float)P.nz - 1.5f;
    if (!(r.cgx >= 0.5f && r.cgx <= hx && r.cgy >= 0.5f && r.cgy <= hy && r.cgz >= 0.5f && r.cgz <= hz)) return 1.0f;
    const float dx = (uc - P.cx32) * P.ifx32, dy = (vc - P.cy32) * P.ify32;
    float w0 = sR[0] * dx + sR[1] * dy + sR[2], w1 = sR[3] * dx + sR[4] * dy + sR[5], w2 = sR[6] * dx + sR[7] * dy + sR[8];
    const float inv = rsqrtf(w0 * w0 + w1 * w1 + w2 * w2);
    w0 *= inv;
    w1 *= inv;
    w2 *= inv;
    const float dl = fmaxf(fmaxf(fabsf(r.rx - w0), fabsf(r.ry - w1)), fabsf(r.rz - w2));
    // (a non-negative float's bits order as the float; 8 voxels a step)
    const float delta = 8.0f * __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(dl)));
    const int lane = threadIdx.x & 31;
    for (int base = 0;; base += 32) {
        const float j = (float)(base + lane), s = 8.0f * (j + 0.5f);
        const float gx = fmaf(s, w0, r.cgx), gy = fmaf(s, w1, r.cgy), gz = fmaf(s, w2, r.cgz);
        bool open = (j + 1.0f) * delta <= 3.9f && gx >= 0.0f && gx <= hx && gy >= 0.0f && gy <= hy && gz >= 0.0f && gz <= hz;
        if (open) {
            const int bi = box_index(P, (int)gx >> 3, (int)gy >> 3, (int)gz >> 3);
            open = PRISM_IN_RANGE(P, CHK_RENDER_BRICK, bi, P.nbox) && (__ldg(M.boxes + bi) & kBoxOpen) != 0u;
        }
        const uint32_t shut = ~__ballot_sync(0xffffffffu, open);
        if (shut) {
            const float d = 8.0f * (float)(base + __ffs(shut) - 1) * P.vs32;   // all samples before this distance
            return fminf(fmaxf(floorf(d / P.eps32 * (1.0f - 1e-6f)), 1.0f), (float)P.kmax);
        }
    }
}

// What the march of a ray found: the index k of the first sample above tau (0:
// none), its value and cell, and the value of sample k - 1 if it was evaluated.
struct MarchHit {
    int k;
    float f, f_prev;
    bool prev_ok;
    Sample cur;
};

// The march of App. B: samples k = 1, 2, ... up to the first one above tau,
// outside the grid or past kmax (below 2^24: fill_kparams; the index is a
// float, exact there).  The grid bounds are tested only for samples after
// k_safe, which a conservative FP32 bound (one voxel of margin, far above the
// rounding of the bound and of the sample positions) keeps inside the grid.
// A ray evaluates NS samples at once (8 NS gathers in flight); a later one past
// kmax or outside the grid is ignored (sample k's corners are read again), one
// past the hit or in a brick without hits changes nothing.
//
// Without P.skip each ray goes on by itself: the march that the jumps below share
// with the warp took twice as long here (32 frames of 640x480 on a 256^3 map in
// one launch: 8.3 ms, 4.6 ms in this loop).
//
// With P.skip the empty-space index decides which samples are evaluated,
// starting from k0 (beam_start); the hit and its values are those of the march
// over every sample.  Every lane of the warp calls it (active: the lane has a
// ray): the lanes jump until each has a sample to evaluate or has ended, then
// evaluate together, so that a warp waits for its gathers a few times instead of
// whenever one lane reaches a surface.  A ray looks a brick up once, and
// evaluates every sample up to its exit (k_eval).  NS = 2, 3, 4 with 8, 6, 5
// blocks an SM: 60.8, 47.8, 44.5 us for one frame of 640x480 on a clean 256^3
// map, 284, 233, 215 us with noise in every brick (a lookup every NS samples,
// NS = 3: 50 and 256 us).  A ray that grazes a surface jumps a hundred times, a
// brick at a time, and the last warps of a launch wait for such rays alone:
// the jump loop is one short dependent chain, without conversions between
// integers and floats (which take ~20 cycles each) and without branches but
// the lookup's.
// nsamp: samples evaluated, up to the hit; steps: jumps and evaluations; uniq
// (DETAIL): distinct corners of the samples evaluated.
template <bool BF16, bool DETAIL, int PX, int NS = 4>
__device__ __forceinline__ MarchHit march(const KParams& P, const MapPlanes& M, const Ray& r, bool active, float k0,
                                          int& nsamp, int& steps, unsigned int& uniq) {
    const uint32_t px = PX > 0 ? (uint32_t)PX : P.px;
    const uint32_t pxy = PX > 0 ? (uint32_t)(PX * PX) : P.pxy;
    const float hx = (float)P.nx - 0.5f, hy = (float)P.ny - 0.5f, hz = (float)P.nz - 0.5f;
    const float rgx = r.rgx, rgy = r.rgy, rgz = r.rgz, cgx = r.cgx, cgy = r.cgy, cgz = r.cgz;
    const float kmax = (float)P.kmax;
    // k_safe: every sample k <= k_safe stays one voxel inside the grid
    float k_safe = 0.0f;
    if (cgx >= 0.5f && cgx <= hx - 1.0f && cgy >= 0.5f && cgy <= hy - 1.0f && cgz >= 0.5f && cgz <= hz - 1.0f) {
        float ks = kmax;
        const float rg3[3] = {rgx, rgy, rgz}, cg3[3] = {cgx, cgy, cgz}, h3[3] = {hx, hy, hz};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (rg3[a] > 0.0f) ks = fminf(ks, (h3[a] - 1.0f - cg3[a]) / (rg3[a] * P.eps32));
            else if (rg3[a] < 0.0f) ks = fminf(ks, (0.5f - cg3[a]) / (rg3[a] * P.eps32));
        }
        k_safe = ks > 0.0f ? floorf(ks) : 0.0f;
    }
    const float ieps = 1.0f / P.eps32;
    const ExitAxis ax(rgx, cgx, ieps), ay(rgy, cgy, ieps), az(rgz, cgz, ieps);
    const bool skip = P.skip && M.boxes != nullptr;
    MarchHit h;
    h.k = 0;
    h.f = h.f_prev = 0.0f;
    h.prev_ok = false;
    float k = k0;
    float k_eval = 0.0f;            // every sample up to this one is evaluated
    int pix = 0, piy = 0, piz = 0;       // DETAIL: the last evaluated sample's cell,
    bool fresh = true;                   // and whether the next one starts a new run of corners
    // sample k's position; false if the ray has ended
    float gx, gy, gz;
    auto position = [&](float kk) {
        const float d = __fmul_rn(kk, P.eps32);
        gx = __fmaf_rn(d, rgx, cgx);
        gy = __fmaf_rn(d, rgy, cgy);
        gz = __fmaf_rn(d, rgz, cgz);
        return kk <= k_safe || (kk <= kmax && gx >= -0.5f && gx < hx && gy >= -0.5f && gy < hy && gz >= -0.5f && gz < hz);
    };
    bool live = active;
    // samples k .. k + NS - 1 of a ray that has sample k; one that it has not reads
    // sample k's corners again
    auto evaluate = [&]() {
        Sample sm[NS];
        float f[NS];
        bool ok[NS];
        position(k);
        sm[0] = cell_of(px, pxy, gx, gy, gz);
        ok[0] = PRISM_IN_RANGE(P, CHK_RENDER_CORNER, (long long)sm[0].base + pxy + px + 1, P.npad);
        if (!ok[0]) {
            live = false;
            return;
        }
#pragma unroll
        for (int j = 1; j < NS; ++j) {
            ok[j] = position(k + (float)j) && ok[j - 1];
            sm[j] = cell_of(px, pxy, gx, gy, gz);
            ok[j] = ok[j] && PRISM_IN_RANGE(P, CHK_RENDER_CORNER, (long long)sm[j].base + pxy + px + 1, P.npad);
            if (!ok[j]) sm[j] = sm[0];
        }
#pragma unroll
        for (int j = 0; j < NS; ++j)
            f[j] = trilinear<BF16, PX>(M.occ, sm[j].base, px, pxy, sm[j].fx, sm[j].fy, sm[j].fz);
        int hit = -1, last = 0;   // the first one above tau, and the last one the ray has
#pragma unroll
        for (int j = NS - 1; j >= 0; --j)
            if (ok[j] && f[j] > P.tau32) hit = j;
#pragma unroll
        for (int j = 1; j < NS; ++j)
            if (ok[j]) last = j;
        if (DETAIL) {   // consecutive cells share 8 >> (axes changed) corners (steps below one voxel)
#pragma unroll
            for (int j = 0; j < NS; ++j)
                if (ok[j] && (hit < 0 || j <= hit)) {
                    const int ch = (sm[j].ix != pix) + (sm[j].iy != piy) + (sm[j].iz != piz);
                    uniq += fresh ? 8u : 8u - (8u >> ch);
                    pix = sm[j].ix; piy = sm[j].iy; piz = sm[j].iz;
                    fresh = false;
                }
        }
        if (hit >= 0) {
            h.k = (int)k + hit;
            nsamp += hit + 1;
#pragma unroll
            for (int j = 0; j < NS; ++j)
                if (j == hit) {
                    h.cur = sm[j];
                    h.f = f[j];
                    if (j > 0) h.f_prev = f[j > 0 ? j - 1 : 0];
                }
            h.prev_ok = h.prev_ok || hit > 0;
            live = false;
        } else {
            nsamp += last + 1;
            h.f_prev = f[0];
            float step = 1.0f;
#pragma unroll
            for (int j = 1; j < NS; ++j)
                if (ok[j]) {
                    h.f_prev = f[j];
                    step = (float)(j + 1);
                }
            h.prev_ok = true;
            k += step;
        }
    };
    if (!skip) {   // (warp-uniform) every sample, each ray by itself
        while (live) {
            live = position(k);
            if (!live) break;
            ++steps;
            evaluate();
        }
        return h;
    }
    while (__any_sync(0xffffffffu, live)) {
        const float k_in = k;
        bool found = false;
        while (live && !found) {
            live = position(k);
            ++steps;
            if (k <= k_eval) {
                found = true;
                break;
            }
            uint32_t w = 0xffu, brick = 0u, cx = 0u, cy = 0u, cz = 0u;
            if (live) {
                // cell coordinates, at least 0, + kFloorMagicBits, whose low 22 bits are 0
                cx = max(__float_as_uint(__fadd_rd(gx, kFloorMagic)), kFloorMagicBits);
                cy = max(__float_as_uint(__fadd_rd(gy, kFloorMagic)), kFloorMagicBits);
                cz = max(__float_as_uint(__fadd_rd(gz, kFloorMagic)), kFloorMagicBits);
                const int bi = box_index(P, (int)((cx >> 3) & 0x7ffffu), (int)((cy >> 3) & 0x7ffffu),
                                         (int)((cz >> 3) & 0x7ffffu));
                brick = ((cx >> 2) & 1u) | ((cy >> 1) & 2u) | (cz & 4u);
                if (PRISM_IN_RANGE(P, CHK_RENDER_BRICK, bi, P.nbox)) w = __ldg(M.boxes + bi);
            }
            found = (w >> brick) & 1u;
            const uint32_t c = (w >> 8) & 3u, clear = (4u << c) - 1u;   // an empty box of 4 2^c cells around it, or the brick
            const float ef = __uint_as_float((129u + c) << 23);
            const float dm = fminf(fminf(ax.dist(cx, clear, ef), ay.dist(cy, clear, ef)), fminf(az.dist(cz, clear, ef), kmax));
            // the last sample before the exit (dm < 2^22 but for enormous marches)
            const float fl = P.kmax < (1 << 22) ? __fadd_rd(dm, kFloorMagic) - kFloorMagic : floorf(dm);
            if (found) k_eval = fl;
            else k = fmaxf(fl, k) + 1.0f;
        }
        found = found && live;
        if (k != k_in) {
            h.prev_ok = false;
            fresh = true;
        }
        __syncwarp();
        if (found) evaluate();
    }
    return h;
}

}  // namespace render_detail

// The work counters of one 128-thread tile: one atomic a counter and block
// (four a block kept one L2 slice 40 % busy).  Every thread calls it.
template <bool DETAIL>
__device__ __forceinline__ void tile_stats(DevStats* stats, bool active, bool hit, int nsamp, unsigned int uniq) {
    __shared__ unsigned long long s_stat[4][4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned long long s = warp_sum_u64((unsigned long long)nsamp);
    const unsigned long long q = DETAIL ? warp_sum_u64((unsigned long long)uniq) : 0ull;
    const unsigned int hits = __popc(__ballot_sync(0xffffffffu, hit));
    const unsigned int rays = __popc(__ballot_sync(0xffffffffu, active));
    if (lane == 0) {
        s_stat[warp][0] = rays;
        s_stat[warp][1] = s;
        s_stat[warp][2] = hits;
        s_stat[warp][3] = q;
    }
    __syncthreads();
    if (threadIdx.x < (DETAIL ? 4 : 3))   // (the four counters are consecutive)
        atomicAdd(&stats->render_rays + threadIdx.x, s_stat[0][threadIdx.x] + s_stat[1][threadIdx.x] +
                                                         s_stat[2][threadIdx.x] + s_stat[3][threadIdx.x]);
}

// One 16x8-pixel tile (128 threads; warp w covers the 8x4 pixels at
// ((w & 1) 8, (w >> 1) 4) of the tile).  sR / sc: camera-to-world rotation
// and centre in shared memory.  Returns the thread's march steps (0 outside
// the image), the anchor render's tile cost.  The value of a sample k - 1
// that the march did not evaluate is recomputed at the hit.
template <bool BF16, bool DETAIL, int PX>
__device__ __forceinline__ int render_tile(const KParams& P, const float* sR, const float* sc, const MapPlanes& M,
                                            float* __restrict__ depth, float* __restrict__ rgb,
                                            uint8_t* __restrict__ mask, int32_t* __restrict__ hitk,
                                            DevStats* __restrict__ stats, int tile_x, int tile_y) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int u = tile_x * 16 + (warp & 1) * 8 + (lane & 7);
    const int v = tile_y * 8 + (warp >> 1) * 4 + (lane >> 3);
    const bool active = u < P.W && v < P.H;
    const uint32_t px = PX > 0 ? (uint32_t)PX : P.px;
    const uint32_t pxy = PX > 0 ? (uint32_t)(PX * PX) : P.pxy;

    int nsamp = 0, hk = 0, steps = 0;
    unsigned int uniq = 0;   // distinct occupancy corners of this ray (DETAIL only)
    float out_d = 0.0f, out_r = 0.0f, out_g = 0.0f, out_b = 0.0f;
    const render_detail::Ray r = render_detail::ray_of(P, sR, sc, u, v);
    const float k0 = P.skip && M.boxes != nullptr
                       ? render_detail::beam_start(P, M, sR, r, (float)(tile_x * 16 + (warp & 1) * 8) + 3.5f,
                                                   (float)(tile_y * 8 + (warp >> 1) * 4) + 1.5f)
                       : 1.0f;
    const render_detail::MarchHit h = render_detail::march<BF16, DETAIL, PX>(P, M, r, active, k0, nsamp, steps, uniq);
    if (active) {
        const int k = h.k;
        if (k == 1) hk = -1;
        if (k >= 2) {
            hk = k;
            const render_detail::Sample& cur = h.cur;
            float f_prev = h.f_prev;
            // sample k - 1, recomputed exactly (same recipe) instead of carried along
            const float d1 = __fmul_rn((float)(k - 1), P.eps32);
            const render_detail::Sample prev = render_detail::cell_of(px, pxy, __fmaf_rn(d1, r.rgx, r.cgx),
                                        __fmaf_rn(d1, r.rgy, r.cgy), __fmaf_rn(d1, r.rgz, r.cgz));
            if (PRISM_IN_RANGE(P, CHK_RENDER_CORNER, (long long)prev.base + pxy + px + 1, P.npad)) {
                if (!h.prev_ok) f_prev = render_detail::trilinear<BF16, PX>(M.occ, prev.base, px, pxy, prev.fx, prev.fy, prev.fz);
                const float alpha = __fdiv_rn(P.tau32 - f_prev, h.f - f_prev);
                const float dk = __fmul_rn((float)k, P.eps32);
                const float dstar = fmaf(alpha, dk - d1, d1);
                out_d = dstar * r.inv_n;
                float a1 = render_detail::trilinear<BF16, PX>(M.r, cur.base, px, pxy, cur.fx, cur.fy, cur.fz);
                float a0 = render_detail::trilinear<BF16, PX>(M.r, prev.base, px, pxy, prev.fx, prev.fy, prev.fz);
                out_r = fmaf(alpha, a1 - a0, a0);
                a1 = render_detail::trilinear<BF16, PX>(M.g, cur.base, px, pxy, cur.fx, cur.fy, cur.fz);
                a0 = render_detail::trilinear<BF16, PX>(M.g, prev.base, px, pxy, prev.fx, prev.fy, prev.fz);
                out_g = fmaf(alpha, a1 - a0, a0);
                a1 = render_detail::trilinear<BF16, PX>(M.b, cur.base, px, pxy, cur.fx, cur.fy, cur.fz);
                a0 = render_detail::trilinear<BF16, PX>(M.b, prev.base, px, pxy, prev.fx, prev.fy, prev.fz);
                out_b = fmaf(alpha, a1 - a0, a0);
            }
        }
        const int p = v * P.W + u;
        if (depth) depth[p] = out_d;
        if (rgb) { rgb[3 * p] = out_r; rgb[3 * p + 1] = out_g; rgb[3 * p + 2] = out_b; }
        if (mask) mask[p] = (uint8_t)(hk >= 2);
        if (hitk) hitk[p] = hk;
    }
    if (stats) tile_stats<DETAIL>(stats, active, hk >= 2, nsamp, uniq);
    return steps;
}

// The order of an anchor render's tiles, heaviest predicted first.  A ray's
// march length varies by two orders of magnitude across the image (rays
// grazing a surface evaluate a sample at every step of a long run of bricks
// that cannot be skipped); rendered in raster order, the heavy tiles start
// last and their blocks run on after the other SMs have emptied.  The
// prediction is the last anchor render's cost (per tile, the sum over its
// warps of the warp's largest count of march steps, jumps over empty bricks
// included) at the tile each tile's centre ray falls in when seen from the
// last camera -- the ray's direction, then its point at the depth the last
// render saw in that direction (the parallax of the centre's move) --
// maximised over its 3x3 tile neighbourhood; a ray outside the last image
// counts as heaviest.  Tiles go into 64 cost buckets, the buckets are laid out
// heaviest first; within a bucket the order is arbitrary.  The order only
// decides when a tile is rendered, never what it renders.  One block (a
// multiple of 32 threads); key: one word of scratch per tile.
__device__ __forceinline__ void render_plan_block(const KParams& P, const RenderPlanIn& in) {
    constexpr int kBuckets = 64;
    constexpr uint32_t kUnknown = 0xffffffffu;
    __shared__ uint32_t hist[kBuckets], base[kBuckets], s_max;
    const int gx = (P.W + 15) >> 4, gy = (P.H + 7) >> 3, nt = gx * gy;
    if (threadIdx.x < kBuckets) hist[threadIdx.x] = 0u;
    if (threadIdx.x == 0) s_max = 0u;
    // R = R_lastᵀ R_next: the next camera's ray directions in the last camera's
    // frame; dc = R_lastᵀ (c_next - c_last): the next centre there
    float R[9], dc[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
#pragma unroll
        for (int j = 0; j < 3; ++j)
            R[3 * i + j] = in.rot_last[i] * in.c2w[j] + in.rot_last[3 + i] * in.c2w[3 + j] +
                           in.rot_last[6 + i] * in.c2w[6 + j];
        dc[i] = in.rot_last[i] * (in.c2w[9] - in.rot_last[9]) + in.rot_last[3 + i] * (in.c2w[10] - in.rot_last[10]) +
                in.rot_last[6 + i] * (in.c2w[11] - in.rot_last[11]);
    }
    __syncthreads();
    uint32_t lmax = 0u;
    for (int t = threadIdx.x; t < nt; t += blockDim.x) {
        const float dx = ((float)((t % gx) * 16 + 8) - P.cx32) * P.ifx32;
        const float dy = ((float)((t / gx) * 8 + 4) - P.cy32) * P.ify32;
        const float ex = R[0] * dx + R[1] * dy + R[2], ey = R[3] * dx + R[4] * dy + R[5];
        const float ez = R[6] * dx + R[7] * dy + R[8];
        uint32_t e = kUnknown;
        if (ez > 1e-6f) {
            float u = P.fx32 * ex / ez + P.cx32, v = P.fy32 * ey / ez + P.cy32;
            if (in.depth_last && u >= 0.0f && u < (float)P.W && v >= 0.0f && v < (float)P.H) {
                // parallax: the ray's point at the depth the last render saw in that
                // direction, projected into the last camera from the next centre
                const float z0 = in.depth_last[min((int)v, P.H - 1) * P.W + min((int)u, P.W - 1)];
                const float sz = (z0 - dc[2]) / ez;
                if (z0 > 0.0f && sz > 0.0f) {
                    const float px = dc[0] + sz * ex, py = dc[1] + sz * ey, pz = dc[2] + sz * ez;
                    if (pz > 1e-6f) {
                        u = P.fx32 * px / pz + P.cx32;
                        v = P.fy32 * py / pz + P.cy32;
                    }
                }
            }
            if (u >= 0.0f && u < (float)P.W && v >= 0.0f && v < (float)P.H) {
                const int tx = min((int)u >> 4, gx - 1), ty = min((int)v >> 3, gy - 1);
                const int x0 = max(tx - 1, 0), x2 = min(tx + 1, gx - 1);
                const int y0 = max(ty - 1, 0), y2 = min(ty + 1, gy - 1);
                const uint32_t* r0 = in.cost + y0 * gx;
                const uint32_t* r1 = in.cost + ty * gx;
                const uint32_t* r2 = in.cost + y2 * gx;
                e = max(max(max(r0[x0], r0[tx]), max(r0[x2], r1[x0])), max(max(r1[tx], r1[x2]), max(r2[x0], r2[tx])));
                e = max(e, r2[x2]);
                lmax = max(lmax, e);
            }
        }
        in.key[t] = e;
    }
    lmax = __reduce_max_sync(0xffffffffu, lmax);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_max, lmax);
    __syncthreads();
    const unsigned long long mx = s_max > 0u ? s_max : 1u;
    for (int t = threadIdx.x; t < nt; t += blockDim.x) {   // the same thread wrote key[t] above
        const uint32_t e = in.key[t];
        const uint32_t k = e == kUnknown ? kBuckets - 1 : (uint32_t)((unsigned long long)e * (kBuckets - 1) / mx);
        in.key[t] = k;
        atomicAdd(&hist[k], 1u);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t run = 0u;
        for (int k = kBuckets - 1; k >= 0; --k) {
            base[k] = run;
            run += hist[k];
        }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nt; t += blockDim.x) {
        const uint32_t pos = atomicAdd(&base[in.key[t]], 1u);
        if (PRISM_IN_RANGE(P, CHK_PLAN, pos, nt)) in.order[pos] = t;
    }
}

__device__ __forceinline__ void depth_mask_px(const KParams& P, const float* __restrict__ depth,
                                              uint8_t* __restrict__ mask, int p) {
    mask[p] = (uint8_t)depth_valid(P, depth, p % P.W, p / P.W);
}

// Anchor packing (App. E.3, reading R18): per pixel
//   a0 = (n_x, n_y, n_z, z)  with z = 0 where the normal is invalid,
//   a1 = (r, g, b, 1 if the depth is valid else 0).
// n = normalize((P(u+1,v) - P(u-1,v)) x (P(u,v+1) - P(u,v-1))), facing the camera.
// anchor_pack_core takes the pixel's depth dc and its neighbours' (dr: u + 1,
// dl: u - 1, dd: v + 1, du: v - 1), its depth validity mc and ok = it and its
// four neighbours are valid inside the image border.
__device__ __forceinline__ void anchor_pack_core(const KParams& P, int u, int v, float dc, float dr, float dl,
                                                 float dd, float du, bool mc, bool ok,
                                                 const float* __restrict__ rgb, float4* __restrict__ a0,
                                                 float4* __restrict__ a1, int p) {
    float n0 = 0.0f, n1 = 0.0f, n2 = 0.0f;
    if (ok) {
        float a[3], b[3], c[3], d[3], pc[3];
        backproject_rn(P, u + 1, v, dr, a);
        backproject_rn(P, u - 1, v, dl, b);
        backproject_rn(P, u, v + 1, dd, c);
        backproject_rn(P, u, v - 1, du, d);
        backproject_rn(P, u, v, dc, pc);
        float e1[3], e2[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) { e1[i] = __fsub_rn(a[i], b[i]); e2[i] = __fsub_rn(c[i], d[i]); }
        float c0 = __fsub_rn(__fmul_rn(e1[1], e2[2]), __fmul_rn(e1[2], e2[1]));
        float c1 = __fsub_rn(__fmul_rn(e1[2], e2[0]), __fmul_rn(e1[0], e2[2]));
        float c2 = __fsub_rn(__fmul_rn(e1[0], e2[1]), __fmul_rn(e1[1], e2[0]));
        float nn = __fmaf_rn(c0, c0, __fmaf_rn(c1, c1, __fmul_rn(c2, c2)));
        if (!(nn > 0.0f) || !isfinite(nn)) {
            ok = false;
        } else {
            float inv = __fdiv_rn(1.0f, __fsqrt_rn(nn));
            n0 = __fmul_rn(c0, inv); n1 = __fmul_rn(c1, inv); n2 = __fmul_rn(c2, inv);
            float dp = __fmaf_rn(n0, pc[0], __fmaf_rn(n1, pc[1], __fmul_rn(n2, pc[2])));
            if (dp > 0.0f) { n0 = -n0; n1 = -n1; n2 = -n2; }
        }
    }
    if (!ok) n0 = n1 = n2 = 0.0f;
    a0[p] = make_float4(n0, n1, n2, ok ? dc : 0.0f);
    a1[p] = make_float4(rgb[3 * p], rgb[3 * p + 1], rgb[3 * p + 2], mc ? 1.0f : 0.0f);
}

// One 32x8-pixel tile on a block of 256 threads: the depths of the tile and
// a 2-pixel halo, then the validity of the tile and a 1-pixel halo, go
// through shared memory (one global read of each depth), with the
// comparisons of depth_valid.
constexpr int kPackTW = 32, kPackTH = 8;

__device__ __forceinline__ void anchor_pack_tile(const KParams& P, const float* __restrict__ depth,
                                                 const float* __restrict__ rgb, float4* __restrict__ a0,
                                                 float4* __restrict__ a1, int tile_x, int tile_y) {
    constexpr int DW = kPackTW + 4, DH = kPackTH + 4, VW = kPackTW + 2, VH = kPackTH + 2;
    __shared__ float sd[DH][DW];
    __shared__ uint8_t sv[VH][VW];
    const int W = P.W, H = P.H, x0 = tile_x * kPackTW, y0 = tile_y * kPackTH, t = threadIdx.x;
    for (int e = t; e < DW * DH; e += blockDim.x) {
        const int r = e / DW, c = e % DW, u = x0 - 2 + c, v = y0 - 2 + r;
        sd[r][c] = (u >= 0 && u < W && v >= 0 && v < H) ? depth[v * W + u] : 0.0f;
    }
    __syncthreads();
    for (int e = t; e < VW * VH; e += blockDim.x) {
        const int r = e / VW, c = e % VW, u = x0 - 1 + c, v = y0 - 1 + r;
        bool ok = false;
        if (u >= 0 && u < W && v >= 0 && v < H) {   // depth_valid on the tile
            const float d = sd[r + 1][c + 1];
            ok = (d > 0.0f) && isfinite(d);
            if (ok && u > 0) ok = fabsf(__fsub_rn(d, sd[r + 1][c])) <= P.disc32;
            if (ok && u < W - 1) ok = fabsf(__fsub_rn(d, sd[r + 1][c + 2])) <= P.disc32;
            if (ok && v > 0) ok = fabsf(__fsub_rn(d, sd[r][c + 1])) <= P.disc32;
            if (ok && v < H - 1) ok = fabsf(__fsub_rn(d, sd[r + 2][c + 1])) <= P.disc32;
        }
        sv[r][c] = (uint8_t)ok;
    }
    __syncthreads();
    const int tx = t % kPackTW, ty = t / kPackTW, u = x0 + tx, v = y0 + ty;
    if (ty < kPackTH && u < W && v < H) {
        const int r = ty + 1, c = tx + 1;   // in sv; in sd: r + 1, c + 1
        const bool mc = sv[r][c] != 0;
        const bool ok = u >= 1 && u <= W - 2 && v >= 1 && v <= H - 2 && mc && sv[r][c - 1] && sv[r][c + 1] &&
                        sv[r - 1][c] && sv[r + 1][c];
        const float dc = sd[r + 1][c + 1];
        float dr = 0.0f, dl = 0.0f, dd = 0.0f, du = 0.0f;
        if (ok) {
            dr = sd[r + 1][c + 2];
            dl = sd[r + 1][c];
            dd = sd[r + 2][c + 1];
            du = sd[r][c + 1];
        }
        anchor_pack_core(P, u, v, dc, dr, dl, dd, du, mc, ok, rgb, a0, a1, v * W + u);
    }
}

}  // namespace prism
