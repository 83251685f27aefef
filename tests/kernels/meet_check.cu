// Test harness of the bounded meeting: `blocks` blocks of a cooperative launch meet `rounds` times;
// in round `miss` the target is one arrival more than there are blocks, so that the wait runs out.
#include <cuda_runtime.h>

#include "m2m_meet.cuh"

using namespace m2m;

static __global__ void k_meet(Meet *g, int rounds, int miss, unsigned limit, int *passed)
{
    __shared__ bool ok;
    unsigned meetings = 0;
    int n = 0;
    for (int r = 0; r < rounds; ++r) {
        meetings += gridDim.x;
        if (!meet(g, meetings + (r == miss ? 1u : 0u), &ok, limit)) break;
        ++n;
    }
    if (threadIdx.x == 0) passed[blockIdx.x] = n;
}

// passed: per block, the meetings that came about; failed: the scratch's flag.
extern "C" int meet_check(int blocks, int rounds, int miss, unsigned limit, int *passed, unsigned *failed)
{
    Meet *g = nullptr;
    int *d = nullptr;
    if (cudaMalloc(&g, sizeof(Meet)) != cudaSuccess || cudaMalloc(&d, sizeof(int) * blocks) != cudaSuccess) return 1;
    cudaMemset(g, 0, sizeof(Meet));
    cudaMemset(d, 0, sizeof(int) * blocks);
    void *args[] = {&g, &rounds, &miss, &limit, &d};
    cudaError_t e = cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(k_meet), dim3(blocks), dim3(64), args, 0, nullptr);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    Meet h;
    if (e == cudaSuccess) e = cudaMemcpy(&h, g, sizeof h, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(passed, d, sizeof(int) * blocks, cudaMemcpyDeviceToHost);
    *failed = h.failed;
    cudaFree(g);
    cudaFree(d);
    return e == cudaSuccess ? 0 : 2;
}
