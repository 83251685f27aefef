// The meeting of the blocks of a cooperative launch, with a limit on every wait.
#pragma once

namespace m2m {

constexpr unsigned kPollLimit = 1u << 24;  // about ten seconds of polling

// Scratch of the meetings; all zero between launches.
struct Meet {
    unsigned arrived, done, failed, pad;
    double wcheck[3];
};

// Every block arrives and waits for `target` arrivals. Returns false after the poll limit or
// once another block has given up.
__device__ inline bool meet(Meet *g, unsigned target, bool *ok, unsigned limit = kPollLimit)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&g->arrived, 1u);
        unsigned polls = 0, v;
        bool good = true;
        do {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&g->arrived) : "memory");
            if (v < target && (++polls & 1023u) == 0) {
                unsigned f;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(f) : "l"(&g->failed) : "memory");
                if (f || polls >= limit) good = false;
            }
        } while (v < target && good);
        if (!good) atomicExch(&g->failed, 1u);
        *ok = good;
    }
    __syncthreads();
    return *ok;
}

}  // namespace m2m
