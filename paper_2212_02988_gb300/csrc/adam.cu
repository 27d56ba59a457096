// adam.cu — the paper's pose optimiser (App. F.2, "Pose optimisation"): Adam
// with its momentum disabled, on the objective of App. E.3
// (Eq. pointtoplanelaplace), as an alternative to the Gauss-Newton passes.
//
// One block runs every step: the steps are sequential, and a step is a chain of
// latencies (FP64 instructions at ~64-105 cycles, one round of gathers).  So a
// step holds only what the next one waits for: warp 0 derives the iterate's
// FP32 matrices into the anchor camera as the Gauss-Newton passes do
// (warp_iterate_mats: xi are tangent coordinates at the prior mean), and beside
// it warp 1 the tangent map C = diag(Ra^T, Ra^T J_l(xi_theta)), warp 2 L xi (L =
// prior pose precision) and warp 3 the step's 1 / (1 - beta2^s).  Thread
// k < pixels draws pixel floor(n u), u the high 32 bits of SplitMix64 output
// (n_localised steps + s - 1) pixels + k from `seed` over 2^32; the draws do not
// depend on the iterate, so the observation of step s + 1 is loaded during
// step s.  The pixels are evaluated with the localisation passes' device code
// (the L1 subgradient sign(r) J / b of their kept residuals); a fixed-order block
// sum gives the anchor-frame gradient g'.  Warp 0 then forms the tangent
// gradient g = (n_pixels / pixels) C^T g' + L xi (the data term estimates the
// full-image objective) and takes the Adam step, one component a lane:
// v = beta2 v + (1 - beta2) g^2, v_hat = v / (1 - beta2^s),
// xi -= lr g / (sqrt(v_hat) + eps), lr = lr_t on translation, lr_r on rotation.
// A pass over 200 of 320x240 pixels takes 3.7 us a step, 1000 steps in all;
// 5.2 us when warp 0 alone derived C and the matrices through the pose, and the
// drawn pixel was loaded after them.
// The unstated constants (beta2, eps) take Adam's defaults in the caller's
// configuration.
#include "kernels.h"
#include "linalg64.cuh"
#include "prism_dev.cuh"
#include "track_dev.cuh"

namespace prism {

namespace {

// Output i of SplitMix64 started at state `seed` (Steele, Lea and Flood 2014:
// the golden gamma increment and the variant-13 finaliser).
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long seed, unsigned long long i) {
    unsigned long long z = seed + (i + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// The pose of xi on every lane of the calling warp: t = pt + xi_t,
// q = normalise(Exp(xi_theta) (x) pq).
__device__ __forceinline__ void warp_pose_of(const double* xi, const double* pq, const double* pt, double pose[7]) {
    const int lane = threadIdx.x & 31;
    const double qn = warp_quat_exp_mul(xi + 3, pq);
    pose[3] = __shfl_sync(0xffffffffu, qn, 0);
    pose[4] = __shfl_sync(0xffffffffu, qn, 1);
    pose[5] = __shfl_sync(0xffffffffu, qn, 2);
    pose[6] = __shfl_sync(0xffffffffu, qn, 3);
    const int ta = lane < 3 ? lane : 0;
    const double tv = pt[ta] + xi[ta];
    pose[0] = __shfl_sync(0xffffffffu, tv, 0);
    pose[1] = __shfl_sync(0xffffffffu, tv, 1);
    pose[2] = __shfl_sync(0xffffffffu, tv, 2);
}

constexpr int kAdamThreads = 256;

__global__ void __launch_bounds__(kAdamThreads, 1)
    k_adam(KParams P, const float* __restrict__ od, const float* __restrict__ orgb, const uint8_t* __restrict__ om,
           const float4* __restrict__ a0, const float4* __restrict__ a1, DevState* dev, AdamArgs A) {
    pdl_enter();
    constexpr int N = NV<TRACK_ADAM>::value;   // g' (6), cost, count
    static_assert(N == 8, "the block sum below takes eight values");
    __shared__ float sMb[12];
    __shared__ double s_xi[6], s_C1[9], s_Ra[9], s_Lx[6], s_anchor[7], s_pq[4], s_pt[3], s_prec[36], s_q0[4], s_b0[3];
    __shared__ double s_bias;
    __shared__ float swarp[kAdamThreads / 32][N];
    __shared__ unsigned long long s_c0;
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    if (tid < 7) s_anchor[tid] = dev->anchor_pose[tid];
    else if (tid < 11) s_pq[tid - 7] = dev->pq[tid - 7];
    else if (tid < 14) s_pt[tid - 11] = dev->pt[tid - 11];
    else if (tid < 20) s_xi[tid - 14] = 0.0;
    else if (tid >= 32 && tid < 68) s_prec[tid - 32] = dev->prec_pp[tid - 32];
    else if (tid >= 96 && tid < 105) s_Ra[tid - 96] = dev->gn_Ci[tid - 96];
    else if (tid >= 128 && tid < 132) s_q0[tid - 128] = dev->gn_q0[tid - 128];
    else if (tid >= 132 && tid < 135) s_b0[tid - 132] = dev->gn_b0[tid - 132];
    if (tid == 0) s_c0 = (unsigned long long)dev->n_localised * (unsigned long long)A.steps * (unsigned long long)A.pixels;
    __syncthreads();
    const float* sM = sMb;
    const float* sb = sMb + 9;
    const int W = P.W, Hh = P.H, NP = W * Hh;
    const float fW1 = (float)(W - 1), fH1 = (float)(Hh - 1), fW2 = (float)(W - 2), fH2 = (float)(Hh - 2);
    const EvalConst kc{1.0f / P.b_geo32, 1.0f / P.b_rgb32};
    const double scale = (double)NP / (double)A.pixels;
    auto draw = [&](int s) {   // this thread's pixel of step s (1, 2, ...)
        const unsigned long long u = splitmix64(A.seed, s_c0 + (unsigned long long)(s - 1) * A.pixels + tid);
        return (int)(((u >> 32) * (unsigned long long)NP) >> 32);
    };
    const bool draws = tid < A.pixels;
    int p = draws ? draw(1) : 0;
    TrackObs obs = track_observe<false>(P, od, orgb, om, nullptr, p, W);
    double v2 = 0.0, b2t = 1.0;   // warp 0, lane i < 6: second moment of component i; warp 3: beta2^s
    const int i6 = lane < 6 ? lane : 0, bi = i6 / 3, ii = i6 % 3;   // warp 0: this lane's component
    const double lr = lane < 3 ? A.lr_t : A.lr_r;
    for (int s = 1; s <= A.steps; ++s) {
        if (warp == 0) {
            double me, be;
            warp_iterate_mats(s_Ra, s_xi, s_q0, s_b0, me, be);
            if (lane < 9) sMb[lane] = (float)me;
            else if (lane < 12) sMb[lane] = (float)be;
        } else if (warp == 1) {   // C1 = Ra^T J_l(xi_theta)
            const int e = lane < 9 ? lane : 0, i = e / 3, j = e % 3;
            const double jl = so3_exp_jl_entry(s_xi + 3, false, i, j);
            const double c = fdot3(s_Ra[i], __shfl_sync(0xffffffffu, jl, j), s_Ra[3 + i], __shfl_sync(0xffffffffu, jl, 3 + j),
                                   s_Ra[6 + i], __shfl_sync(0xffffffffu, jl, 6 + j));
            if (lane < 9) s_C1[lane] = c;
        } else if (warp == 2) {
            double lx = 0.0;
#pragma unroll
            for (int k = 0; k < 6; ++k) lx = fma(s_prec[6 * i6 + k], s_xi[k], lx);
            if (lane < 6) s_Lx[lane] = lx;
        } else if (warp == 3) {
            b2t *= A.beta2;
            const double r = 1.0 / (1.0 - b2t);
            if (lane == 0) s_bias = r;
        }
        __syncthreads();
        float acc[N];
#pragma unroll
        for (int v = 0; v < N; ++v) acc[v] = 0.0f;
        if (draws) {
            TrackPix q;
            track_project(P, sM, sb, obs, a0, a1, p, W, fW1, fH1, fW2, fH2, q);
            if (s < A.steps) {   // the next step's pixel, in flight beside the gathers
                p = draw(s + 1);
                obs = track_observe<false>(P, od, orgb, om, nullptr, p, W);
            }
            track_eval<TRACK_ADAM>(P, kc, sb, q, acc);
        }
        __syncwarp();
        // fixed-order block sum: a shuffle tree per warp (the eight values' trees
        // share their shuffles: value k ends in the lanes with l >> 2 == k), then
        // warps 0, 1, ...
#pragma unroll
        for (int w = 4, o = 16; w >= 1; w >>= 1, o >>= 1) {
            const bool upper = (lane & o) != 0;
#pragma unroll
            for (int v = 0; v < w; ++v) {
                const float send = upper ? acc[v] : acc[v + w], keep = upper ? acc[v + w] : acc[v];
                acc[v] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
        acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 2);
        acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
        if ((lane & 3) == 0) swarp[warp][lane >> 2] = acc[0];
        __syncthreads();
        if (warp == 0) {
            float sv = swarp[0][i6];
#pragma unroll
            for (int w = 1; w < kAdamThreads / 32; ++w) sv += swarp[w][i6];
            // lane i < 6: g_i = scale (C^T g')_i + (L xi)_i, then the Adam step
            const double gd = (double)sv;
            const double g0 = __shfl_sync(0xffffffffu, gd, 3 * bi), g1 = __shfl_sync(0xffffffffu, gd, 3 * bi + 1),
                         g2 = __shfl_sync(0xffffffffu, gd, 3 * bi + 2);
            // C^T's row: of C0 = Ra^T (entry (ii, k) of Ra), or of C1
            const double* C = bi ? s_C1 + ii : s_Ra + 3 * ii;
            const int sC = bi ? 3 : 1;
            const double mg = fdot3(C[0], g0, C[sC], g1, C[2 * sC], g2);
            const double g = scale * mg + s_Lx[i6];
            v2 = A.beta2 * v2 + (1.0 - A.beta2) * g * g;
            const double d = sqrt(v2 * s_bias) + A.eps, lg = lr * g;
            // (one FP64 reciprocal step from an FP32 seed; the division for what it does not take)
            const double step = __all_sync(0xffffffffu, pivot_ok(d)) ? lg * rcp64(d) : lg / d;
            const double xn = s_xi[i6] - step;
            __syncwarp();
            if (lane < 6) s_xi[lane] = xn;
        }
        __syncthreads();
    }
    if (warp == 0) {   // the optimum's pose and matrices for the Laplace pass
        double pose[7];
        warp_pose_of(s_xi, s_pq, s_pt, pose);
        warp_mats_rel(pose, s_anchor, dev->rel);
        if (lane < 6) dev->xi[lane] = s_xi[lane];
        if (lane < 7) dev->cur_pose[lane] = pose[lane];
    }
}

}  // namespace

cudaError_t launch_adam(const KParams& P, const float* o_depth, const float* o_rgb, const uint8_t* o_mask,
                        const float4* a0, const float4* a1, DevState* dev, const AdamArgs& A, cudaStream_t s) {
    if (A.pixels < 1 || A.pixels > kAdamThreads || A.steps < 1) return cudaErrorInvalidValue;
    return launch_pdl(k_adam, 1, kAdamThreads, s, P, o_depth, o_rgb, o_mask, a0, a1, dev, A);
}

}  // namespace prism
