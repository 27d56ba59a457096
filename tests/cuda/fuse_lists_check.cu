// The lists of the map update (fuse_dev.cuh, mapio.cu) with counters that do not
// start at zero.  argv[1]: where they start.  Prints the tiles appended in the
// list, the words changed past its end, and the tiles that launch_brick_flags
// took from past it.  Every buffer here is three lists long, so that a write or
// read past a list stays inside it.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "fuse_dev.cuh"
#include "mapio.cu"

using namespace prism;

__global__ void __launch_bounds__(256) k_lists(KParams P, const float* w2c, int* list, int* cells, unsigned int* ctr) {
    __shared__ float sM[9], sb[3];
    load_w2c(w2c, sM, sb);
    __syncthreads();
    cull_tiles(P, sM, sb, blockIdx.x * blockDim.x + threadIdx.x, false, list, cells, ctr);
}

int main(int, char** argv) {
    const unsigned int start = (unsigned int)std::atoi(argv[1]);
    KParams P{};
    P.nx = P.ny = P.nz = 64;
    P.nbx = P.nby = P.nbz = 8;
    P.px = P.py = 66;
    P.pxy = 66 * 66;
    P.npad = 66 * 66 * 66;
    P.W = 80;
    P.H = 60;
    P.skip = 1;
    P.vs32 = 0.0625f;
    P.o32[0] = P.o32[1] = -2.0f;
    P.o32[2] = 1.0f;
    P.fx32 = P.fy32 = 70.0f;
    P.cx32 = 39.5f;
    P.cy32 = 29.5f;
    const int n = 512, words = 3 * n;
    const float w2c[12] = {1, 0, 0, 0, 1, 0, 0, 0, 1, 0, 0, 0};
    float *d_w2c, *occ;
    int* lists;
    unsigned int* ctr;
    uint8_t* bricks;
    if (cudaMalloc(&d_w2c, sizeof(w2c)) || cudaMalloc(&lists, 2 * words * sizeof(int)) || cudaMalloc(&ctr, 2 * sizeof(int)) ||
        cudaMalloc(&occ, P.npad * sizeof(float)) || cudaMalloc(&bricks, n))
        return 2;
    std::vector<int> h(2 * words, -7);
    const unsigned int c0[2] = {start, start};
    cudaMemcpy(d_w2c, w2c, sizeof(w2c), cudaMemcpyHostToDevice);
    cudaMemcpy(lists, h.data(), 2 * words * sizeof(int), cudaMemcpyHostToDevice);
    cudaMemcpy(ctr, c0, sizeof(c0), cudaMemcpyHostToDevice);
    k_lists<<<2, 256>>>(P, d_w2c, lists, lists + words, ctr);
    if (cudaDeviceSynchronize()) return 3;
    cudaMemcpy(h.data(), lists, 2 * words * sizeof(int), cudaMemcpyDeviceToHost);
    int in = 0, past = 0;
    for (int i = 0; i < 2 * words; ++i)
        if (h[i] != -7) (i % words < n ? in : past) += 1;
    // a list of tile 5, followed by tile 9, with a count of 2 n
    std::vector<int> l(words, 9);
    for (int i = 0; i < n; ++i) l[i] = 5;
    const unsigned int c1 = 2 * n;
    cudaMemcpy(lists, l.data(), words * sizeof(int), cudaMemcpyHostToDevice);
    cudaMemcpy(ctr, &c1, sizeof(c1), cudaMemcpyHostToDevice);
    cudaMemset(occ, 0, P.npad * sizeof(float));
    cudaMemset(bricks, 0xaa, n);
    MapPlanes M{};
    M.occ = occ;
    M.bricks = bricks;
    if (launch_brick_flags(P, M, lists, ctr, 0) || cudaDeviceSynchronize()) return 4;
    std::vector<uint8_t> b(n);
    cudaMemcpy(b.data(), bricks, n, cudaMemcpyDeviceToHost);
    std::printf("%d %d %d %d\n", in, past, (int)(b[5] != 0xaa), (int)(b[9] != 0xaa));
    return 0;
}
