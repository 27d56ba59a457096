// state.cu — single-stream launches of the prediction and of the pose
// matrices; the device bodies are in state_dev.cuh.
#include "state_dev.cuh"

namespace prism {

__global__ void __launch_bounds__(256) k_predict(KParams P, DevState* dev, const double* __restrict__ imu, int n,
                                                 double dt) {
    pdl_enter();
    predict_block<PREP_NONE>(P, dev, imu, n, dt);
}

// The prediction and the Gauss-Newton start matrices of the new prior against
// the state mean's camera.
__global__ void __launch_bounds__(256) k_predict_prep(KParams P, DevState* dev, const double* __restrict__ imu,
                                                      int n, double dt) {
    pdl_enter();
    predict_block<PREP_REL_NEXT>(P, dev, imu, n, dt);
}

__global__ void k_prep(DevState* dev, int kind, PoseArg pose) {
    pdl_enter();
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);   // (warp-uniform to the compiler)
    if (warp == 0) prep_mats_warp(dev, kind, pose);
    else if (kind == PREP_REL) prep_vector_warp(dev);
}

// A new state and its FP32 matrices; everything else of the device state but the
// anchor's pose is cleared.  The state arrives as a kernel argument, so the call
// neither waits for the stream nor copies: with the anchor's pose read back and
// the struct written from the host (two copies and a wait, then k_prep) a
// mapping loop over known poses idled for ~30 us a frame (16 frames of 251x189
// into a 200^3 map, with the map's read-out and a view: 1026 -> 577 us).
__global__ void __launch_bounds__(256) k_set_state(DevState* dev, const __grid_constant__ StateArg state) {
    pdl_enter();
    constexpr int kHead = offsetof(StateArg, n_localised) / 8, kAnchor = offsetof(DevState, anchor_pose) / 8;
    static_assert(kHead == offsetof(DevState, pt) / 8 && sizeof(DevState) % 8 == 0, "the same head, whole words");
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    double* words = reinterpret_cast<double*>(dev);
    for (int e = tid; e < (int)(sizeof(DevState) / 8); e += blockDim.x)
        if (e < kAnchor || e >= kAnchor + 7) words[e] = e < kHead ? reinterpret_cast<const double*>(&state)[e] : 0.0;
    __syncthreads();
    if (tid == 0) dev->n_localised = state.n_localised;
    if (warp == 0) prep_mats_warp(dev, PREP_STATE, PoseArg{});
}

cudaError_t launch_set_state(DevState* dev, const StateArg& state, cudaStream_t s) {
    return launch_pdl(k_set_state, 1, 256, s, dev, state);
}

cudaError_t launch_prep(DevState* dev, int kind, const PoseArg& pose, cudaStream_t s, bool pdl) {
    if (pdl) return launch_pdl(k_prep, 1, 64, s, dev, kind, pose);
    k_prep<<<1, 64, 0, s>>>(dev, kind, pose);
    return cudaGetLastError();
}

cudaError_t launch_predict(const KParams& P, DevState* dev, const double* imu, int n, double dt, cudaStream_t s,
                           bool pdl) {
    if (pdl) return launch_pdl(k_predict, 1, 256, s, P, dev, imu, n, dt);
    k_predict<<<1, 256, 0, s>>>(P, dev, imu, n, dt);
    return cudaGetLastError();
}

cudaError_t launch_predict_prep(const KParams& P, DevState* dev, const double* imu, int n, double dt,
                                cudaStream_t s) {
    k_predict_prep<<<1, 256, 0, s>>>(P, dev, imu, n, dt);
    return cudaGetLastError();
}

}  // namespace prism
