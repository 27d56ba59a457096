// render_bwd.cu — adjoint of the render of App. B: gradients of
// L = sum gD * depth + sum gC . rgb for given images gD, gC; the device body is
// in adjoint_dev.cuh.  The pose gradient is reduced per block and added to
// DevState::grad_pose in FP64.
#include "adjoint_dev.cuh"
#include "kernels.h"
#include "prism_dev.cuh"

namespace prism {

namespace {

// The gradient images (either may be null: zero).  A ray whose gradients are
// all zero is not marched.
struct GivenGradients {
    static constexpr bool kImage = false;
    const float* gD;
    const float* gC;
    float gd, c0, c1, c2;
    __device__ __forceinline__ bool want(int p) {
        gd = gD ? gD[p] : 0.0f;
        c0 = gC ? gC[3 * p] : 0.0f;
        c1 = gC ? gC[3 * p + 1] : 0.0f;
        c2 = gC ? gC[3 * p + 2] : 0.0f;
        return gd != 0.0f || c0 != 0.0f || c1 != 0.0f || c2 != 0.0f;
    }
    __device__ __forceinline__ bool get(int, float, const float*, float& d, float c[3]) const {
        d = gd;
        c[0] = c0;
        c[1] = c1;
        c[2] = c2;
        return true;   // (want)
    }
};

}  // namespace

template <bool BF16>
__global__ void __launch_bounds__(128) k_render_bwd(KParams P, const float* __restrict__ mats, MapPlanes M,
                                                    const float* __restrict__ gD, const float* __restrict__ gC,
                                                    float* __restrict__ g_occ, float* __restrict__ g_rgb,
                                                    DevState* __restrict__ dev) {
    pdl_enter();
    __shared__ float sR[9], sc[3];
    __shared__ float sred[4][6];
    if (threadIdx.x < 12) {
        if (threadIdx.x < 9) sR[threadIdx.x] = mats[threadIdx.x];
        else sc[threadIdx.x - 9] = mats[threadIdx.x];
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float gpose[6] = {0, 0, 0, 0, 0, 0};
    GivenGradients grads{gD, gC, 0.0f, 0.0f, 0.0f, 0.0f};
    int nsamp = 0;
    unsigned int uniq = 0;
    adjoint_tile<BF16, false, 0>(P, sR, sc, M, grads, g_occ, g_rgb, gpose, nsamp, uniq, blockIdx.x, blockIdx.y);
    for (int i = 0; i < 6; ++i) {
        const float sum = warp_sum(gpose[i]);
        if (lane == 0) sred[warp][i] = sum;
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        const double s = (double)sred[0][threadIdx.x] + sred[1][threadIdx.x] + sred[2][threadIdx.x] +
                         sred[3][threadIdx.x];
        if (s != 0.0) atomicAdd(&dev->grad_pose[threadIdx.x], s);
    }
}

cudaError_t launch_render_bwd(const KParams& P, const float* mats, const MapPlanes& M, const float* grad_depth,
                              const float* grad_rgb, float* grad_occ, float* grad_rgb_map, DevState* dev,
                              cudaStream_t s) {
    dim3 grid((P.W + 15) / 16, (P.H + 7) / 8), block(128);
    if (P.bf16)
        launch_pdl(k_render_bwd<true>, grid, block, s, P, mats, M, grad_depth, grad_rgb, grad_occ, grad_rgb_map, dev);
    else
        launch_pdl(k_render_bwd<false>, grid, block, s, P, mats, M, grad_depth, grad_rgb, grad_occ, grad_rgb_map, dev);
    return cudaGetLastError();
}

}  // namespace prism
