// Test harness of the integer FP64 functions: evaluates them on the device or on the host at
// given points, and gives each result's error in units of its last place against long double.
#include <cuda_runtime.h>

#include <cmath>
#include <vector>

#include "fp64_int.cuh"

using namespace m2m;

enum { kSqrt, kRsqrt, kDiv, kMul, kExp, kExpMhalf, kLog, kHernquist, kNfwMu };

__host__ __device__ static double eval(int fn, double a, double b, double c, const u64 *et, const u64 *ln)
{
    Big r, ir;
    switch (fn) {
    case kSqrt: return sqrt_int(a);
    case kRsqrt:
        big_rsqrt(big_of(a), ir, r);
        return big_double(ir);
    case kDiv: return div_int(a, b);
    case kMul: return mul_int(a, b);
    case kExp: return exp_int(a, et);
    case kExpMhalf: return exp_mhalf(a, et);
    case kLog: return log_int(a, ln);
    case kHernquist:  // G M = b, a = c at r^2 = a
        big_rsqrt(big_of(a), ir, r);
        return big_double(hernquist_big(b, c, r, ir));
    default: return big_double(nfw_mu_big(b, big_of(a), ln));  // r = a, r_s = b
    }
}

static long double reference(int fn, long double a, long double b, long double c)
{
    switch (fn) {
    case kSqrt: return sqrtl(a);
    case kRsqrt: return 1.0L / sqrtl(a);
    case kDiv: return a / b;
    case kMul: return a * b;
    case kExp: return expl(a);
    case kExpMhalf: return expl(-0.5L * a);
    case kLog: return logl(a);
    case kHernquist: {
        const long double r = sqrtl(a);
        return b / ((r + c) * (r + c) * r);
    }
    default: {
        const long double q = a / b;
        if (q > 0.05L) return log1pl(q) - q / (1.0L + q);
        long double s = 0.0L, p = q;
        for (int k = 2; k < 40; ++k) {
            p *= q;
            s += (k % 2 ? -p : p) * (k - 1) / k;
        }
        return s;
    }
    }
}

static __global__ void k_eval(int fn, const double *x, long long n, const u64 *tab, double *out)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        out[i] = eval(fn, x[i], x[n + i], x[2 * n + i], tab, tab + kExpEntries);
}

// x: three arguments of n points each, one after the other; y: the results; err (or null): in ulp.
extern "C" int int_check(int fn, int device, const double *x, long long n, double *y, double *err)
{
    std::vector<u64> tab(kExpEntries + 2 * kLnEntries);
    exp_table(tab.data());
    ln_table(tab.data() + kExpEntries);
    if (device) {
        double *d = nullptr;
        u64 *t = nullptr;
        if (cudaMalloc(&d, sizeof(double) * 4 * n) != cudaSuccess || cudaMalloc(&t, sizeof(u64) * tab.size()) != cudaSuccess)
            return 1;
        cudaMemcpy(d, x, sizeof(double) * 3 * n, cudaMemcpyHostToDevice);
        cudaMemcpy(t, tab.data(), sizeof(u64) * tab.size(), cudaMemcpyHostToDevice);
        k_eval<<<304, 256>>>(fn, d, n, t, d + 3 * n);
        cudaMemcpy(y, d + 3 * n, sizeof(double) * n, cudaMemcpyDeviceToHost);
        const cudaError_t e = cudaDeviceSynchronize();
        cudaFree(d);
        cudaFree(t);
        if (e != cudaSuccess) return 2;
    } else {
        for (long long i = 0; i < n; ++i) y[i] = eval(fn, x[i], x[n + i], x[2 * n + i], tab.data(), tab.data() + kExpEntries);
    }
    for (long long i = 0; err && i < n; ++i) {
        const long double r = reference(fn, x[i], x[n + i], x[2 * n + i]);
        int e;
        frexpl(r, &e);
        err[i] = double(fabsl((long double)y[i] - r) / ldexpl(1.0L, e - 53));
    }
    return 0;
}

// seed_bits of a float.
extern "C" unsigned long long int_seed_bits(float y) { return seed_bits(y); }

// Every 24-bit lead of a significand, with the bits below all zero and all one: the largest
// |a (1/a) - 1| 2^60 and |a (a^-1/2)^2 - 1| 2^60 of the reciprocal and, for both parities of the
// exponent, of the inverse root.
static __global__ void k_leads(unsigned long long *out)
{
    unsigned long long worst[2] = {0, 0};
    const unsigned stride = gridDim.x * blockDim.x;
    for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < (1u << 24); q += stride) {
        const u64 m = (1ull << 63) | (u64(q >> 1) << 40) | ((q & 1) ? (1ull << 40) - 1 : 0);
        const Big z = big_rcp(Big{m, 0});  // in (1/2, 1]: m (scale 2^63) times m_z (scale 2^64)
        i64 d = i64(mulhi_u(m, z.m) - (1ull << 63));
        u64 v = u64(d < 0 ? -d : d) >> 3;
        if (v > worst[0]) worst[0] = v;
        for (int odd = 0; odd < 2; ++odd) {
            Big r, ir;
            big_rsqrt(Big{m, odd}, ir, r);  // value (1 + odd) m 2^-63 = v; ir in [1/2, 1] at scale 2^64
            const u64 s = mulhi_u(ir.m, ir.m);           // scale 2^64
            const u64 p = mulhi_u(odd ? m : m >> 1, s);  // v s at scale 2^62
            d = i64(p - (1ull << 62));
            v = u64(d < 0 ? -d : d) >> 2;
            if (v > worst[1]) worst[1] = v;
        }
    }
    atomicMax(out, worst[0]);
    atomicMax(out + 1, worst[1]);
}

extern "C" int int_leads(unsigned long long *out)
{
    unsigned long long *d = nullptr;
    if (cudaMalloc(&d, 16) != cudaSuccess) return 1;
    cudaMemset(d, 0, 16);
    k_leads<<<608, 256>>>(d);
    cudaMemcpy(out, d, 16, cudaMemcpyDeviceToHost);
    const cudaError_t e = cudaDeviceSynchronize();
    cudaFree(d);
    return e == cudaSuccess ? 0 : 2;
}
