// mapping.cu — gradient-descent mapping, the alternative to the closed-form
// map update that the paper compares against (Sec. 4.4, Fig. sdfvsvi): a
// rendering loss over frames with known poses, carried to the map means by
// the render adjoint (render_bwd.cu), and plain descent steps on the means.
#include "adjoint_dev.cuh"
#include "kernels.h"
#include "prism_dev.cuh"

namespace prism {

namespace {

// The loss of one rendered frame against its observation (obs_d, obs_c):
// where the render hits and the observed depth is valid (finite, > 0),
// (d - D)^2 / (2 sd^2) + |c - C|^2 / (2 sc^2), in FP64 (a hit's few FP64
// instructions wait beside its gathers: pairs of floats were no faster, 178 us a
// step of eight frames of 320x240 against 177).
struct FrameLoss {
    static constexpr bool kImage = true;
    const float* obs_d;
    const float* obs_c;
    float inv_sd2, inv_sc2;
    double half_inv_sd2, half_inv_sc2;
    double* loss;
    float D;
    double l;   // this thread's loss
    __device__ __forceinline__ bool want(int p) {
        D = obs_d[p];
        return true;
    }
    // (every ray is marched: the render's counters count the rays without a depth too)
    __device__ __forceinline__ bool get(int p, float d, const float* c, float& gd, float gc[3]) {
        if (!(isfinite(D) && D > 0.0f)) return false;
        const float r = d - D;
        gd = r * inv_sd2;
        double lc = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float rc = c[k] - obs_c[3 * p + k];
            gc[k] = rc * inv_sc2;
            lc = fma((double)rc, (double)rc, lc);
        }
        l = fma((double)r * (double)r, half_inv_sd2, lc * half_inv_sc2);
        return gd != 0.0f || gc[0] != 0.0f || gc[1] != 0.0f || gc[2] != 0.0f;
    }
};

}  // namespace

// The FP32 camera-to-world matrices of a batch of poses, one warp each.
struct DescentPoses {
    double p[kDescentBatch][7];
};
__global__ void k_descent_mats(const __grid_constant__ DescentPoses poses, float* __restrict__ mats) {
    pdl_enter();
    warp_mats_c2w(poses.p[blockIdx.x], mats + 12 * blockIdx.x);
}

// Render, loss and adjoint of a batch of frames in one pass, grid z = frame:
// each ray is marched once, and the image stays in registers.  One launch a
// batch instead of four a frame (matrices, render, loss, adjoint, the image
// written and read between them): 126 us for eight frames of 320x240 on a
// 128^3 map, against 520 us.
template <bool BF16, bool DETAIL>
__global__ void __launch_bounds__(128) k_descent_frames(KParams P, const float* __restrict__ mats, MapPlanes M,
                                                        FrameLoss frame, float* __restrict__ g_occ,
                                                        float* __restrict__ g_rgb, DevStats* __restrict__ stats) {
    pdl_enter();
    __shared__ float sR[9], sc[3];
    __shared__ double s_l[4];
    const size_t f = blockIdx.z, npix = (size_t)P.W * P.H;
    if (threadIdx.x < 12) {
        const float v = mats[12 * f + threadIdx.x];
        if (threadIdx.x < 9) sR[threadIdx.x] = v;
        else sc[threadIdx.x - 9] = v;
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int u = blockIdx.x * 16 + (warp & 1) * 8 + (lane & 7), v = blockIdx.y * 8 + (warp >> 1) * 4 + (lane >> 3);
    frame.obs_d += f * npix;
    frame.obs_c += 3 * f * npix;
    frame.l = 0.0;
    float gpose[6] = {0, 0, 0, 0, 0, 0};   // (not used: known poses)
    int nsamp = 0;
    unsigned int uniq = 0;
    const int k = adjoint_tile<BF16, DETAIL, 0>(P, sR, sc, M, frame, g_occ, g_rgb, gpose, nsamp, uniq, blockIdx.x, blockIdx.y);
    double l = frame.l;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) s_l[warp] = l;
    if (stats) tile_stats<DETAIL>(stats, u < P.W && v < P.H, k >= 2, nsamp, uniq);
    __syncthreads();
    if (threadIdx.x == 0) {
        l = (s_l[0] + s_l[1]) + (s_l[2] + s_l[3]);
        if (l != 0.0) atomicAdd(frame.loss, l);
    }
}

namespace {

// A sum of squares of FP32 values, kept as an unevaluated sum of three floats
// a + b + c: a square is h + l exactly (its rounding error by an FMA), and every
// addition into a and b keeps its rounding error (Knuth's two-sum); only c's
// additions round.  With b and c folded upwards once a row the sum is good to 1e-16
// (against exact sums of 3 to 4,000 squares; FP64 additions: 1e-16 to 1e-14).  It takes
// two dozen FP32 instructions a value where an FP64 conversion and FMA take 16
// cycles each on an SM: a descent step on 128^3 voxels 86 us against 110, on 256^3
// 430 against 536 (one and two frames).  The floats hold the squares of 2^-50
// (below it l would underflow) to 1e14 (3e10 of them stay finite); `rest` sums the
// others in FP64.
struct SquareSum {
    float a = 0.0f, b = 0.0f, c = 0.0f;
    double rest = 0.0;
    // s = s + x with the rounding error left in x
    static __device__ __forceinline__ void two_sum(float& s, float& x) {
        const float t = s + x, z = t - s;
        x = (s - (t - z)) + (x - z);
        s = t;
    }
    __device__ __forceinline__ void add(float h, float l, float m) {
        two_sum(a, h);
        two_sum(b, h);
        two_sum(b, l);
        c += (h + l) + m;
    }
    __device__ __forceinline__ void square(float r) {
        const float x = fabsf(r);
        if (x <= 1e14f && (x >= 0x1p-50f || x == 0.0f)) {
            const float h = r * r;
            add(h, fmaf(r, r, -h), 0.0f);
        } else {
            rest = fma((double)r, (double)r, rest);
        }
    }
    __device__ __forceinline__ void fold() {
        two_sum(a, b);
        two_sum(b, c);
    }
    // the floats summed over the N lanes that differ in the lowest bits
    template <int N>
    __device__ __forceinline__ void over_lanes() {
#pragma unroll
        for (int o = 1; o < N; o <<= 1)
            add(__shfl_xor_sync(0xffffffffu, a, o), __shfl_xor_sync(0xffffffffu, b, o), __shfl_xor_sync(0xffffffffu, c, o));
    }
    __device__ __forceinline__ double value() const { return (double)a + ((double)b + (double)c); }
    // this thread's rest, times scale, to *loss (rare)
    __device__ __forceinline__ void add_rest(double scale, double* loss) const {
        if (__double_as_longlong(rest)) atomicAdd(loss, rest * scale);
    }
};

}  // namespace

// The descent step on every padded element (ghosts included, each from the
// voxel it clamps to, as the map load fills them):
//   mu <- mu - lr (g + (mu - mu0) / prior_var)
// for occupancy (g_occ, lr_occ, mu0_occ) and the three colour planes (g_rgb,
// lr_rgb, mu0_rgb).  The prior term of the loss, sum (mu - mu0)^2 /
// (2 prior_var) over the voxels before the step, is added to *loss.  One warp
// per padded row, so that the row's coordinates are worked out once: 34 us for
// 128^3 voxels, 71 us with a division chain an element and the loss in FP64.
template <bool BF16>
__global__ void __launch_bounds__(256) k_map_step(KParams P, MapPlanes M, const float* __restrict__ g_occ,
                                                  const float* __restrict__ g_rgb, float lr_occ, float lr_rgb,
                                                  float mu0_occ, float mu0_rgb, float inv_v0, double half_inv_v0,
                                                  double* loss) {
    pdl_enter();
    __shared__ float part[8][3];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t rows = P.npad / P.px;
    SquareSum l;
    for (uint32_t row = blockIdx.x * 8 + warp; row < rows; row += gridDim.x * 8) {
        const int gy = (int)(row % P.py) - 1, gz = (int)(row / P.py) - 1;
        const int y = min(max(gy, 0), P.ny - 1), z = min(max(gz, 0), P.nz - 1);
        const bool in_row = gy == y && gz == z;
        const size_t vox = ((size_t)z * P.ny + y) * P.nx;
        for (uint32_t e = lane; e < P.px; e += 32) {
            const int gx = (int)e - 1, x = min(max(gx, 0), P.nx - 1);
            const bool interior = in_row && gx == x;
            const size_t i = vox + x;
            const uint32_t q = row * P.px + e;
            {
                const float m = map_load_rw<BF16>(M.occ, q);
                const float dm = m - mu0_occ;
                if (interior) l.square(dm);
                map_store<BF16>(M.occ, q, m - lr_occ * (g_occ[i] + dm * inv_v0));
            }
            void* planes[3] = {M.r, M.g, M.b};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float m = map_load_rw<BF16>(planes[c], q);
                const float dm = m - mu0_rgb;
                if (interior) l.square(dm);
                map_store<BF16>(planes[c], q, m - lr_rgb * (g_rgb[3 * i + c] + dm * inv_v0));
            }
        }
        l.fold();
    }
    __syncwarp();
    l.add_rest(half_inv_v0, loss);
    l.over_lanes<32>();
    if (lane == 0) {
        part[warp][0] = l.a;
        part[warp][1] = l.b;
        part[warp][2] = l.c;
    }
    __syncthreads();
    if (warp == 0) {
        l.a = part[lane & 7][0];
        l.b = part[lane & 7][1];
        l.c = part[lane & 7][2];
        l.over_lanes<8>();
        if (lane == 0) atomicAdd(loss, l.value() * half_inv_v0);
    }
}

cudaError_t launch_descent_frames(const KParams& P, const double* poses, int frames, const MapPlanes& M,
                                  const float* obs_d, const float* obs_c, double sd, double sc, float* mats,
                                  float* g_occ, float* g_rgb, double* loss, DevStats* stats, bool detail, cudaStream_t s) {
    if (frames < 1 || frames > kDescentBatch) return cudaErrorInvalidValue;
    DescentPoses dp{};
    for (int j = 0; j < frames; ++j)
        for (int a = 0; a < 7; ++a) dp.p[j][a] = poses[7 * j + a];
    cudaError_t e = launch_pdl(k_descent_mats, frames, 32, s, dp, mats);
    if (e != cudaSuccess) return e;
    FrameLoss f{};
    f.obs_d = obs_d;
    f.obs_c = obs_c;
    f.inv_sd2 = (float)(1.0 / (sd * sd));
    f.inv_sc2 = (float)(1.0 / (sc * sc));
    f.half_inv_sd2 = 0.5 / (sd * sd);
    f.half_inv_sc2 = 0.5 / (sc * sc);
    f.loss = loss;
    const dim3 grid((P.W + 15) / 16, (P.H + 7) / 8, frames);
    auto go = [&](auto kern) { return launch_pdl(kern, grid, 128, s, P, (const float*)mats, M, f, g_occ, g_rgb, stats); };
    if (P.bf16) return detail ? go(k_descent_frames<true, true>) : go(k_descent_frames<true, false>);
    return detail ? go(k_descent_frames<false, true>) : go(k_descent_frames<false, false>);
}

cudaError_t launch_map_step(const KParams& P, const MapPlanes& M, const float* g_occ, const float* g_rgb,
                            double lr_occ, double lr_rgb, double mu0_occ, double mu0_rgb, double prior_var,
                            double* loss, cudaStream_t s) {
    const uint32_t need = (P.npad / P.px + 7) / 8, grid = need > 152u * 8u ? 152u * 8u : need;
    const float inv_v0 = (float)(1.0 / prior_var);
    auto go = [&](auto kern) {
        return launch_pdl(kern, grid, 256, s, P, M, g_occ, g_rgb, (float)lr_occ, (float)lr_rgb, (float)mu0_occ,
                          (float)mu0_rgb, inv_v0, 0.5 / prior_var, loss);
    };
    return P.bf16 ? go(k_map_step<true>) : go(k_map_step<false>);
}

}  // namespace prism
