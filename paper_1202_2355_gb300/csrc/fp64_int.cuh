// FP64 functions of the step on the integer pipe.
//
// An SM of this part issues an FP64 instruction for a warp every 16 cycles and 64 others
// meanwhile, so the FP64 pipe bounds the FP64 step and a function on 64-bit integers is cheap
// beside it: the library square root and division (10 FP64 instructions each), an exponential
// (12) and a logarithm (25) become 30 to 60 integer instructions. They work on the significand
// as a 64-bit fixed-point number (products keep the high 64 of 128 bits), so they carry 8 to 10
// more bits than FP64 and round once at the end. Worst errors, in ulp, against long double: square
// root and inverse root 0.516, quotient 0.51, exponential 0.51, product 0.501, the Hernquist
// factor (four of these) 0.54. Sums of fixed-point terms are bounded absolutely instead: the
// logarithm 2^-60 for 1/2 <= x < 2 (and 0.9 ulp beyond), the NFW mass factor 12 2^-62 for r/r_s up to 1
// above its series (some 300 ulp where the series ends, at mu = 2^-15; ln(1+q) - q/(1+q) in FP64 is off
// by 120 to 1,500 there), 2 ulp elsewhere. Seeds come from the hardware approximations in FP32
// (relative error below 2^-21); a seed's residual e is formed exactly and the series
// (1 - e)^(-1/2) = 1 + e/2 + 3 e^2/8 + ... or 1/(1 - e) = 1 + e + e^2 + ... ends the root.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

namespace m2m {

typedef unsigned long long u64;
typedef long long i64;

__host__ __device__ __forceinline__ u64 mulhi_u(u64 a, u64 b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return u64((static_cast<unsigned __int128>(a) * b) >> 64);
#endif
}
__host__ __device__ __forceinline__ i64 mulhi_s(i64 a, i64 b)
{
#ifdef __CUDA_ARCH__
    return __mul64hi(a, b);
#else
    return i64((static_cast<__int128>(a) * b) >> 64);
#endif
}
__host__ __device__ __forceinline__ int mulhi_s32(int a, int b)
{
#ifdef __CUDA_ARCH__
    return __mulhi(a, b);
#else
    return int((i64(a) * b) >> 32);
#endif
}
// The bits of a double and back, opaque to the compiler's front end: it would turn integer tests
// of them into FP64 comparisons and sign changes into FP64 arithmetic.
__host__ __device__ __forceinline__ i64 bits_of(double x)
{
#ifdef __CUDA_ARCH__
    i64 b;
    asm("mov.b64 %0, %1;" : "=l"(b) : "d"(x));
    return b;
#else
    i64 b;
    std::memcpy(&b, &x, 8);
    return b;
#endif
}
__host__ __device__ __forceinline__ double of_bits(i64 b)
{
#ifdef __CUDA_ARCH__
    double x;
    asm("mov.b64 %0, %1;" : "=d"(x) : "l"(b));
    return x;
#else
    double x;
    std::memcpy(&x, &b, 8);
    return x;
#endif
}
__host__ __device__ __forceinline__ float of_bits32(unsigned b)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float x;
    std::memcpy(&x, &b, 4);
    return x;
#endif
}
__host__ __device__ __forceinline__ unsigned bits_of32(float x)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    unsigned b;
    std::memcpy(&b, &x, 4);
    return b;
#endif
}
__host__ __device__ __forceinline__ float seed_rsqrt(float x)
{
#ifdef __CUDA_ARCH__
    return rsqrtf(x);
#else
    return 1.f / std::sqrt(x);
#endif
}
__host__ __device__ __forceinline__ float seed_rcp(float x)
{
#ifdef __CUDA_ARCH__
    return __fdividef(1.f, x);
#else
    return 1.f / x;
#endif
}

// The FP64 product of factors out of mul_int's range. Not inlined: the compiler would compute one
// FP64 instruction ahead of the test and select (it looks cheap, and is 16 cycles of the pipe).
#ifdef __CUDACC__
static __device__ __noinline__ double mul_far(double a, double b) { return a * b; }
#endif

// A positive number m 2^(e - 63) with the top bit of m set.
struct Big {
    u64 m;
    int e;
};

// Whether x is positive, normal and of moderate exponent (2^-200 .. 2^200): the range in
// which the functions below need no special cases. Anything else (0, subnormal, infinite, NaN)
// goes to the library.
__host__ __device__ __forceinline__ bool big_range(double x)
{
    const unsigned hi = unsigned(u64(bits_of(x)) >> 32);
    return hi - (unsigned(1023 - 200) << 20) < (400u << 20);
}

// x positive and normal.
__host__ __device__ __forceinline__ Big big_of(double x)
{
    const u64 b = u64(bits_of(x));
    return Big{(b << 11) | (1ull << 63), int(b >> 52) - 1023};
}

// Rounded to the nearest double; a result of exponent below -1022 is not formed here.
__host__ __device__ __forceinline__ double big_double(const Big &a)
{
    const u64 r = (a.m >> 11) + ((a.m >> 10) & 1);  // 2^52 .. 2^53; the carry moves the exponent on
    return of_bits(i64(r + (u64(i64(a.e + 1022)) << 52)));
}

// The leading 24 bits of a significand as a float in [1, 2).
__host__ __device__ __forceinline__ float big_lead(u64 m) { return of_bits32(0x3f800000u | (unsigned(m >> 40) & 0x7fffffu)); }

// The seed as its 24 bits, in [1/2, 1): the hardware approximations may give 1, or a value below
// 1/2 for an argument next to 2, whose significand would be read as nearly 1.
__host__ __device__ __forceinline__ u64 seed_bits(float y)
{
    y = y < 0.99999994f ? y : 0.99999994f;
    return (bits_of32(y > 0.5f ? y : 0.5f) & 0x7fffffu) | 0x800000u;
}

// A root in [1/2, 1] at scale 2^64 that its rounding may have carried a few units over either
// end: back inside.
__host__ __device__ __forceinline__ u64 root_clamp(u64 y)
{
    return (y >> 63) ? y : ((y >> 62) ? (1ull << 63) : ~0ull);
}

// a^(-1/2) and a^(1/2) to about 2^-59 relative.
__host__ __device__ __forceinline__ void big_rsqrt(const Big &a, Big &inv, Big &root)
{
    const int odd = a.e & 1, half = a.e >> 1;  // a = v 4^half, 1 <= v < 4
    const u64 v = odd ? a.m : a.m >> 1;        // scale 2^62
    const float vf = of_bits32(bits_of32(big_lead(a.m)) + (unsigned(odd) << 23));
    const u64 y0 = seed_bits(seed_rsqrt(vf));                 // scale 2^24
    const i64 e = i64((1ull << 62) - mulhi_u(v, (y0 * y0) << 16));  // 1 - v y0^2, scale 2^62
    const int eh = int(e >> 12);                              // scale 2^50
    const u64 e2 = u64(i64(eh) * eh);                         // scale 2^100
    const i64 c = e + i64((3 * e2) >> 40);                    // e/2 + 3 e^2/8, scale 2^63
    const u64 y = root_clamp((y0 << 40) + u64((i64(y0) * (c >> 4)) >> 19));  // scale 2^64
    inv = Big{y, -1 - half};
    u64 r = mulhi_u(v, y);  // scale 2^62
    if (r < (1ull << 62)) r = 1ull << 62;
    root = Big{r << 1, half};
}

// 1 / a to about 2^-60 relative.
__host__ __device__ __forceinline__ Big big_rcp(const Big &a)
{
    const u64 z0 = seed_bits(seed_rcp(big_lead(a.m)));  // scale 2^24
    const i64 e = i64((1ull << 63) - mulhi_u(a.m, z0 << 40));  // 1 - a z0, scale 2^63
    const int eh = int(e >> 14);                        // scale 2^49
    const i64 c = e + i64(u64(i64(eh) * eh) >> 35);     // e + e^2, scale 2^63
    return Big{root_clamp((z0 << 40) + u64((i64(z0) * (c >> 3)) >> 20)), -1 - a.e};
}

__host__ __device__ __forceinline__ Big big_add(const Big &a, const Big &b)
{
    const int d = a.e - b.e;
    const u64 mb = d >= 0 ? a.m : b.m, ms = d >= 0 ? b.m : a.m;
    const int eb = d >= 0 ? a.e : b.e, sh = 1 + (d >= 0 ? d : -d);
    const u64 s = (mb >> 1) + (sh < 64 ? ms >> sh : 0);
    return (s >> 63) ? Big{s, eb + 1} : Big{s << 1, eb};
}

// Product of two significands read as fractions in [1/2, 1): the exponent of the result is
// that of the product if its top bit is set (see big_norm).
__host__ __device__ __forceinline__ Big big_mul_raw(const Big &a, const Big &b) { return Big{mulhi_u(a.m, b.m), a.e + b.e + 1}; }

__host__ __device__ __forceinline__ int big_clz(u64 v)
{
#ifdef __CUDA_ARCH__
    return __clzll(i64(v));
#else
    return __builtin_clzll(v);
#endif
}

// Up to three leading zeros shifted out.
__host__ __device__ __forceinline__ Big big_norm(Big a)
{
    if (!(a.m >> 62)) {
        a.m <<= 2;
        a.e -= 2;
    }
    if (!(a.m >> 63)) {
        a.m <<= 1;
        a.e -= 1;
    }
    return a;
}

// a b: the high half of the product of the significands, rounded to nearest; zeros, subnormal or
// non-finite factors and results near the ends of the range take the FP64 instruction.
__host__ __device__ __forceinline__ double mul_int(double a, double b)
{
    const u64 x = u64(bits_of(a)), y = u64(bits_of(b));
    const unsigned ex = unsigned(x >> 52) & 0x7ffu, ey = unsigned(y >> 52) & 0x7ffu, e = ex + ey;
    // ex, ey >= 1 and e - 1023 within 1 .. 2045: both normal, the product too
    if (ex - 1u >= 2046u || ey - 1u >= 2046u || e - 1024u >= 2044u) {
#ifdef __CUDA_ARCH__
        return mul_far(a, b);
#else
        return a * b;
#endif
    }
    const u64 m = mulhi_u((x << 11) | (1ull << 63), ((y << 11) | (1ull << 63)));
    const unsigned up = unsigned(m >> 63);
    const u64 n = up ? m : m << 1;  // the bit shifted in is below the rounding
    const u64 r = (n >> 11) + ((n >> 10) & 1);
    return of_bits(i64((r + (u64(e - 1023u - 1u + up) << 52)) | ((x ^ y) & (1ull << 63))));
}

// ---------------------------------------------------------------- exp
//
// x = N ln2/256 + r, N = 256 e + j, |r| < ln2/512 (1 + 2^-4); exp(x) = 2^e 2^(j/256) (1 + p(r)),
// p = r + r^2 (1/2 + r (1/6 + r (1/24 + r/120))), truncation r^6/720 < 2^-65. r is exact to
// 2^-71: x 2^71 and N ln2/256 2^71 are taken modulo 2^64, their difference fits. The table holds
// 2^(j/256) at scale 2^62. Valid for -707 < x < 709.

constexpr int kExpEntries = 256;

inline void exp_table(u64 t[kExpEntries])
{
    for (int j = 0; j < kExpEntries; ++j)
        t[j] = u64(std::exp2((long double)j / kExpEntries) * (long double)(1ull << 62) + 0.5L);
}

// exp(x) of |x| < 709 as a Big.
__host__ __device__ __forceinline__ Big exp_big(double x, const u64 *t)
{
    constexpr u64 kL = 6393154322601327829ull;   // ln2/256 at scale 2^71, integer part
    constexpr unsigned kLlo = 0xe4f1d9ccu;       // its next 32 bits
    const i64 b = bits_of(x);
    const int ex = int(u64(b) >> 52 & 0x7ff) - 1023;
    // x in FP32 (truncated): enough for N
    const unsigned fb = unsigned(u64(b) >> 29);  // sign and exponent of FP64 drop off the top
    const unsigned xe = unsigned(ex + 127);
    const float xf = ex > -100 ? of_bits32((b < 0 ? 0x80000000u : 0u) | (xe << 23) | (fb & 0x7fffffu)) : 0.f;
#ifdef __CUDA_ARCH__
    const float tf = fmaf(xf, 369.3299304675746f, 12582912.f);
#else
    const float tf = std::fma(xf, 369.3299304675746f, 12582912.f);
#endif
    const int N = int(bits_of32(tf)) - 0x4b400000;
    const u64 m = (u64(b) & 0xfffffffffffffull) | (1ull << 52);
    const int sh = ex + 19;  // m 2^(ex - 52) at scale 2^71
    u64 X = sh >= 0 ? m << sh : (sh > -64 ? m >> -sh : 0);
    if (b < 0) X = 0 - X;
    const i64 R = i64(X - u64(i64(N)) * kL) - ((i64(N) * i64(kLlo)) >> 32);
    const int r = int(R >> 31);                             // scale 2^40
    const int t1 = 178956971 + (mulhi_s32(r, 35791394) >> 8);  // 1/24 + r/120, scale 2^32
    const int s = 715827883 + (mulhi_s32(r, t1) >> 8);         // 1/6 + ..
    const i64 q = (1ll << 62) + ((i64(r) * s) >> 9);           // 1/2 + .., scale 2^63
    const i64 r2 = mulhi_s(R, R);                              // scale 2^78
    const i64 P = R + (mulhi_s(r2, q) >> 6);                   // scale 2^71
    const i64 T = i64(t[N & 255]);                             // scale 2^62
    const u64 y = (u64(T) << 1) + u64(mulhi_s(T, P) >> 6);     // scale 2^63
    const int e = N >> 8;
    return (y >> 63) ? Big{y, e} : Big{y << 1, e - 1};
}

// exp(x) in FP64: 0 below -707 (results under ~1e-307), +inf above 709, NaN propagates.
__host__ __device__ __forceinline__ double exp_int(double x, const u64 *t)
{
    const i64 b = bits_of(x), p = b & 0x7fffffffffffffffll;
    if (p >= 0x4086180000000000ll) {  // |x| >= 707, or NaN
        if (p > 0x7ff0000000000000ll) return x;
        if (b < 0) return 0.0;
        if (p > 0x4086280000000000ll) return of_bits(0x7ff0000000000000ll);  // 709
    }
    return big_double(exp_big(x, t));
}

// exp(-t/2) for t >= 0 (the halving is one step of the exponent); NaN of either sign stays NaN.
__host__ __device__ __forceinline__ double exp_mhalf(double t, const u64 *tab)
{
    const i64 b = bits_of(t);
    const double x = b > (64ll << 52) ? of_bits((b - (1ll << 52)) | i64(1ull << 63)) : 0.0;  // t < 2^-959 gives 1
    const bool far = (b & 0x7fffffffffffffffll) >= (2047ll << 52);
    return exp_int(far ? of_bits(b | i64(1ull << 63)) : x, tab);  // inf and NaN: negated
}

// ---------------------------------------------------------------- force factors

// G M / ((r + a)^2 r) of the Hernquist potential at r^2 = r2. r2, a, gm in big_range.
__host__ __device__ __forceinline__ Big hernquist_big(double gm, double a, const Big &r, const Big &ir)
{
    const Big z = big_rcp(big_add(r, big_of(a)));
    return big_norm(big_mul_raw(big_mul_raw(big_mul_raw(z, z), ir), big_of(gm)));
}

// ln on 128 intervals of [1, 2): entry j holds c = 1/(1 + (j + 1/2)/128) rounded to 2^-30 (scale
// 2^63), then -ln c at scale 2^62.
constexpr int kLnEntries = 128;

inline void ln_table(u64 t[2 * kLnEntries])
{
    for (int j = 0; j < kLnEntries; ++j) {
        const u64 c = u64(std::floor((long double)(1ull << 30) / (1.0L + (j + 0.5L) / kLnEntries) + 0.5L));
        t[2 * j] = c << 33;
        t[2 * j + 1] = u64(-std::log((long double)c / (long double)(1ull << 30)) * (long double)(1ull << 62) + 0.5L);
    }
}

// ln of m 2^-63 in [1, 2) at scale 2^62: -ln c + ln(1 + z), z = m c - 1, |z| < 2^-8 (1 + 2^-7),
// by the series to z^7 (truncation below 2^-66).
__host__ __device__ __forceinline__ i64 ln_frac(u64 m, const u64 *t)
{
    const int j = int(m >> 56) & 127;
    const i64 z = i64(mulhi_u(m, t[2 * j])) - (1ll << 62);         // scale 2^62
    const int zs = int(z >> 24);                                   // scale 2^38
    const int g3 = 858993459 + (mulhi_s32(zs, -715827883 + (mulhi_s32(zs, 613566757) >> 6)) >> 6);  // 1/5 - z/6 + z^2/7
    const int g2 = -1073741824 + (mulhi_s32(zs, g3) >> 6);         // -1/4 + .., scale 2^32
    const i64 h = 1537228672809129301ll + ((i64(zs) * g2) >> 8);   // 1/3 + .., scale 2^62
    const i64 g = -(1ll << 62) + (mulhi_s(z, h) << 3);             // -1/2 + .., scale 2^63
    const i64 z2 = mulhi_s(z << 6, z << 6);                        // scale 2^72
    return i64(t[2 * j + 1]) + z + (mulhi_s(z2, g) >> 9);
}

// The NFW terms at q = r/r_s: mu = ln(1+q) - q/(1+q) and, if l1 is not null, ln(1+q). With
// t = r/(r + r_s) = q/(1+q) and u = 1 - t = r_s/(r + r_s): mu = -ln u - t, both terms in fixed point
// (2^-62 while u > 1/2, 2^-56 beyond); below t = 2^-7, where they cancel, the series
// t^2 (1/2 + t/3 + t^2/4 + ..). ln(1+q) = mu + t.
__host__ __device__ __forceinline__ Big nfw_mu_big(double rs, const Big &r, const u64 *tab, Big *l1 = nullptr)
{
    const Big B = big_of(rs);
    const Big w = big_rcp(big_add(r, B));
    const Big t = big_norm(big_mul_raw(r, w)), u = big_norm(big_mul_raw(B, w));
    Big mu;
    if (t.e < -7) {
        const double x = big_double(t);
        double s = 1.0 / 9.0;
        s = fma(x, s, 1.0 / 8.0);
        s = fma(x, s, 1.0 / 7.0);
        s = fma(x, s, 1.0 / 6.0);
        s = fma(x, s, 1.0 / 5.0);
        s = fma(x, s, 1.0 / 4.0);
        s = fma(x, s, 1.0 / 3.0);
        s = fma(x, s, 0.5);
        mu = big_norm(big_mul_raw(big_mul_raw(t, t), big_of(s)));
    } else {
        const i64 ln = ln_frac(u.m, tab);
        i64 v;
        int sc;
        if (u.e >= -1) {  // -ln u = ln 2 - ln(2 u)
            v = 3196577161300663915ll - ln - i64(t.m >> (1 - t.e));  // scale 2^62: t = m 2^(e - 63)
            sc = 62;
        } else {
            v = i64(-u.e) * 49946518145322874ll - (ln >> 6) - i64(t.m >> (7 - t.e));  // scale 2^56
            sc = 56;
        }
        const int lz = big_clz(u64(v));
        mu = Big{u64(v) << lz, 63 - lz - sc};
    }
    if (l1) *l1 = big_add(t, mu);
    return mu;
}

// G M_s mu(r/r_s) / r^3 of the NFW halo.
__host__ __device__ __forceinline__ Big nfw_big(double gms, double rs, const Big &r, const Big &ir, const u64 *tab)
{
    return big_norm(big_mul_raw(big_norm(big_mul_raw(big_mul_raw(big_mul_raw(ir, ir), ir), big_of(gms))),
                                nfw_mu_big(rs, r, tab)));
}

// ---------------------------------------------------------------- plain functions
//
// FP64 square root, quotient and logarithm on the integer pipe for the arguments of the prior
// binning (the library's for anything out of range).

__host__ __device__ __forceinline__ double sqrt_int(double x)
{
    if (!big_range(x)) return sqrt(x);
    Big r, ir;
    big_rsqrt(big_of(x), ir, r);
    return big_double(r);
}

// a / b for b > 0
__host__ __device__ __forceinline__ double div_int(double a, double b)
{
    const double p = of_bits(bits_of(a) & 0x7fffffffffffffffll);
    if (!big_range(p) || !big_range(b)) return a / b;
    const double q = big_double(big_norm(big_mul_raw(big_rcp(big_of(b)), big_of(p))));
    return of_bits(bits_of(q) | (bits_of(a) & i64(1ull << 63)));
}

// ln x: within 2^-60 of it for 1/2 <= x < 2, and 0.9 ulp beyond.
__host__ __device__ __forceinline__ double log_int(double x, const u64 *tab)
{
    if (!big_range(x)) return log(x);
    const Big b = big_of(x);
    const i64 ln = ln_frac(b.m, tab);
    const bool near1 = b.e == 0 || b.e == -1;
    i64 v = near1 ? (b.e ? ln - 3196577161300663915ll : ln) : i64(b.e) * 24973259072661437ll + (ln >> 7);  // 2^62, 2^55
    if (v == 0) return 0.0;
    const bool neg = v < 0;
    if (neg) v = -v;
    const int lz = big_clz(u64(v));
    const double r = big_double(Big{u64(v) << lz, 63 - lz - (near1 ? 62 : 55)});
    return neg ? -r : r;
}

}  // namespace m2m
