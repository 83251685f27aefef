// Device side of the M2M step: model description, per-particle arithmetic and
// the step kernel. Templated on the state type T: double (FP64 mode) or float
// (mixed mode: FP32 state, push and kernel values; exact integer bin sums).
//
// Method (arXiv 1202.2355): leap-frog push (Sec. 4.1), observables
// y_j = sum_i w_i K_j(z_i) (eq. obs) with the Gauss-Hermite kernels of
// eq. lumghn, temporal smoothing (eq. myts), residuals (eqs. delta, chi),
// (E, x) moving priors (Sec. 2.3.1) and the force of change (eq. modFOC) with
// the entropy of eq. S+ (moving priors) or eq. entropy (global).
#pragma once

#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>

#include "fp64_exp.cuh"
#include "fp64_int.cuh"

namespace m2m {

constexpr int kMaxGroups = 4;
constexpr int kMaxKinds = 16;
constexpr int kKindMass = 0;
constexpr int kKindV2 = 1;
constexpr int kKindV1 = 2;  // internal: first moment, used only to build targets
constexpr int kKindGH0 = 10;
constexpr int kKindAlm0 = 100;  // a_lm on shells: kKindAlm0 + l (l + 1) + m

enum : unsigned { kErrNonFinite = 1u, kErrNegWeight = 2u, kErrOverflow = 4u, kErrIndex = 8u, kErrTimeout = 16u };

struct GroupDesc {
    int geometry;   // 0 annuli, 1 pixels, 2 shells (3-D radial grid of the a_lm, eq. alm)
    int n_ap;
    int n_kinds;
    int obs_off;    // first observable index of the group
    int ap_off;     // first aperture index (into Vp / 1/sp arrays)
    int edge_off;   // first edge (annuli)
    int max_gh;     // highest Gauss-Hermite order used, -1 if none
    int has_v2;     // the group deposits v_los^2 (range-checked against v2max)
    int nx, ny;
    int kinds[kMaxKinds];
    double xlo, ylo, xw, yw;  // pixel box origin and widths (xhi - xlo, yhi - ylo)
    // FP32 versions: pixel origin and nx/xw, ny/yw; annulus lookup: bucket
    // b = floor((log2 R^2 - l0) lscale) -> first candidate annulus lut[lut_off + b]
    float xlo_f, ylo_f, ixw, iyw;
    int lut_off, lut_n;
    float l0, lscale;
    float e0sq_f, ensq_f;     // squared first and last edge (FP32 annuli)
    int lut_identity;         // edges uniform in log R: bucket b is annulus b (no table load)
    // plan: kind index (0..n_kinds-1) of each kernel in the group, or -1
    int k_mass, k_v2, k_v1;
    int k_gh[7];
    // shells: l and m of each kind, and the factor of the real Y_lm (N_lm, times sqrt2 for m != 0)
    signed char alm_l[kMaxKinds], alm_m[kMaxKinds];
    double alm_norm[kMaxKinds];
    float alm_norm_f[kMaxKinds];
};

struct Model {
    // potential
    int pot;                      // 0 Hernquist, 1 Hernquist + NFW, 2 log
    double G, M, a, Ms, rs, v0, r0, q;
    double phi_min;
    // projection
    double sin_i, cos_i;
    // observables
    int n_groups, J, n_ap_total, n_edges_total, n_lut;
    GroupDesc g[kMaxGroups];
    // priors
    int mode, nE, nx, e_spacing, signed_lz, update_every, ncell;
    double s_lo, s_den;           // E-axis map: f = (s(E) - s_lo) / s_den
    // circular orbits: closed form (Hernquist) or table of E_c(ln R)
    int lc_closed, lc_n;
    double lc_lnr0, lc_dlnr;
    // step
    double dt, eps, mu, alpha;
    int update_rule, renormalize;
    long long n_relax;
    // fixed point: value = words / scale
    double fx_w, fx_v2, fx_gh, v2max;
    int wps;                      // int64 words per sum in the global sums
    int hist_words, off_total, off_grid, off_count;
    int rec_len;                  // doubles per aperture record of the force of change
    // aperture cache: the deposit of a step stores each particle's apertures for the
    // force of change at the start of the next (same positions): 0 none, 1 two groups
    // of at most 255 apertures (8 bits each), 2 one group (16 bits)
    int ap_cache;
    // the acceleration at the current positions is kept between steps (always in FP64)
    int cache_accel;
    // FP64 mode with the aperture cache: exp(-nu^2/2) of this group's aperture (the
    // first group with Gauss-Hermite kernels, -1 none) is also kept from the deposit
    // for the next force of change (same nu, same value)
    int gx_group;
    // prior smoothing (Sec. 2.3.2): 0 off; lambda > 0 fixed, else chosen by GCV
    int smooth;
    double smooth_lambda;
    // grid-less moving priors (Sec. 7): half widths, in cells, of the window of cells
    // centred on each cell whose particles' mean weight is its prior; 0, 0: the cell mean
    int pwin_E, pwin_x;
    // global-deposit kernel: apertures [win_lo, win_lo + win_n) of group win_group keep
    // block-shared sums (the densest range, placed at load); the rest deposit globally
    int win_group, win_lo, win_n;
    // one shard of a fit split over processes: the step kernel leaves its integer sums for
    // the caller to add over the shards, and k_finalize runs the finalize afterwards;
    // n_all is the particle count of the whole fit (the local count when not sharded)
    int shard;
    long long n_all;
    // self-consistent stellar potential (pot 3, Sec. 6): phi = Upsilon phi_star + log halo,
    // phi_star the multipole expansion of the particles' luminosity on scf_n grid radii with
    // harmonics l <= scf_lmax (scf_nlm = (scf_lmax + 1)^2, index l (l + 1) + m). Its sums
    // are the slots [off_scf, off_scf + scf_n scf_nlm), deposited on update steps; with the
    // mass-to-light fit (eps_ups > 0) the derivatives D_j of the observables are the slots
    // [off_dups, off_dups + n_dups). nslots counts every slot of the sums.
    int scf_n, scf_lmax, scf_nlm, off_scf, off_dups, n_dups, nslots;
    double eps_ups, fx_dv;
    const double *scf_r;   // device: grid radii
    double *scf_tab;       // device: per interval j = 0..scf_n, (TA_lm, TB_lm), Upsilon and
                           // -4 pi G/(2l+1) folded in (see scf_field)
    float *scf_tabf;       // FP32 copy
    double *scf_coef;      // device: a_lm,k of the last expansion (scf_n x scf_nlm)
    double scf_norm[49];   // factor of Y_lm (N_lm, sqrt2 N_lm for m != 0) by index
    float scf_norm_f[49];
    // the finalize of a step runs as k_finalize over several blocks instead of in the last
    // block of the step kernel (see configure_kernels)
    int fin_wide;
    // FP64 mode: the potential's constants are in the range of the integer force factors
    // (big_range), and whether the tables of the integer functions are in shared memory
    int int_force, tab_smem;
    // global-deposit kernel: the prior grid's sums are block-shared
    int cells_smem;
    // shell groups: highest l, and the kind of each (l, m) (index l (l + 1) + m) or -1
    int alm_lmax[kMaxGroups];
    signed char alm_k[kMaxGroups][56];
};

constexpr unsigned kApNone8 = 0xFFu, kApNone16 = 0xFFFFu;
constexpr unsigned kApUncached = 0xFFFFFFFFu;  // no cached code: locate the apertures

// Compile-time shape of an observable group, for step kernels specialised to a
// configuration: bits for the kernels it deposits and its geometry. kDyn: read the
// shape from the runtime GroupDesc (the generic kernel); 0: no such group.
constexpr unsigned kBitMass = 1u, kBitV2 = 2u, kBitV1 = 4u, kBitPix = 1u << 15, kBitShell = 1u << 16;
constexpr unsigned kDyn = 0xFFFFFFFFu;
__host__ __device__ constexpr unsigned bit_gh(int n) { return 8u << n; }
__host__ __device__ constexpr int mask_max_gh(unsigned m, int n = 6)
{
    return n < 0 ? -1 : ((m & bit_gh(n)) ? n : mask_max_gh(m, n - 1));
}

template <unsigned M>
struct GP {
    static constexpr unsigned mask = M;
    static constexpr bool dyn = M == kDyn;
    __device__ static bool present(const Model &m, int g)
    {
        if constexpr (dyn) return g < m.n_groups;
        else return M != 0u;
    }
    __device__ static bool pixels(const GroupDesc &G)
    {
        if constexpr (dyn) return G.geometry == 1;
        else return (M & kBitPix) != 0u;
    }
    __device__ static bool shells(const GroupDesc &G)
    {
        if constexpr (dyn) return G.geometry == 2;
        else return (M & kBitShell) != 0u;
    }
    __device__ static bool mass(const GroupDesc &G)
    {
        if constexpr (dyn) return G.k_mass >= 0;
        else return (M & kBitMass) != 0u;
    }
    __device__ static bool v2(const GroupDesc &G)
    {
        if constexpr (dyn) return G.k_v2 >= 0;
        else return (M & kBitV2) != 0u;
    }
    __device__ static bool v1(const GroupDesc &G)
    {
        if constexpr (dyn) return G.k_v1 >= 0;
        else return (M & kBitV1) != 0u;
    }
    __device__ static bool gh(const GroupDesc &G, int n)
    {
        if constexpr (dyn) return G.k_gh[n] >= 0;
        else return (M & bit_gh(n)) != 0u;
    }
    __device__ static int max_gh(const GroupDesc &G)
    {
        if constexpr (dyn) return G.max_gh;
        else return mask_max_gh(M);
    }
};

// Calls f(GP<M>{}, g) for each present group g, with g a compile-time constant.
template <int G0, unsigned M, unsigned... Rest, class F>
__device__ __forceinline__ void each_group(const Model &m, F &&f)
{
    if (GP<M>::present(m, G0)) f(GP<M>{}, G0);
    if constexpr (sizeof...(Rest) > 0) each_group<G0 + 1, Rest...>(m, f);
}

// Model constants in the state type, so that the FP32 path runs no FP64 operation. The
// batched kernel copies a fit's constants into shared memory in 8-byte words: the struct is
// kept a multiple of 16 bytes so that every element of an array of them is 8-byte aligned.
template <class T>
struct alignas(16) Cst {
    T GM, a, GMs, rs, v0sq, r0sq, q2, phi_min, hn_phi0, sin_i, cos_i;
    T dt, hdt, dteps, mu, v2max, fx_w, fx_v2, fx_gh, fx_dv;
    T s_lo, s_den, e_scale, nE, nx;
    T lc_lnr0, lc_dlnr, lc_r0, lc_rmax;
    T iq2;  // 1/q2
};

template <class T>
inline Cst<T> make_cst(const Model &m)
{
    Cst<T> k;
    k.GM = T(m.G * m.M); k.a = T(m.a); k.GMs = T(m.G * m.Ms); k.rs = T(m.rs);
    k.iq2 = T(1.0 / (m.q * m.q));
    k.v0sq = T(m.v0 * m.v0); k.r0sq = T(m.r0 * m.r0); k.q2 = T(m.q * m.q);
    k.phi_min = T(m.phi_min); k.hn_phi0 = T(m.rs > 0 ? -m.G * m.Ms / m.rs : 0.0);
    k.sin_i = T(m.sin_i); k.cos_i = T(m.cos_i);
    k.dt = T(m.dt); k.hdt = T(0.5 * m.dt); k.dteps = T(m.dt * m.eps); k.mu = T(m.mu);
    k.v2max = T(m.v2max); k.fx_w = T(m.fx_w); k.fx_v2 = T(m.fx_v2); k.fx_gh = T(m.fx_gh); k.fx_dv = T(m.fx_dv);
    k.s_lo = T(m.s_lo); k.s_den = T(m.s_den);
    k.e_scale = T(m.G * m.M > 0 ? m.a / (m.G * m.M) : 0.0);
    k.nE = T(m.nE); k.nx = T(m.nx);
    k.lc_lnr0 = T(m.lc_lnr0); k.lc_dlnr = T(m.lc_dlnr);
    k.lc_r0 = T(exp(m.lc_lnr0)); k.lc_rmax = T(exp(m.lc_lnr0 + (m.lc_n - 1) * m.lc_dlnr));
    return k;
}

// Per-fit scalars living in device memory, written by the finalize.
struct Scalars {
    long long t;        // steps completed
    double wscale;      // current weight = wscale * stored weight (mixed mode)
    double lwscale;     // ln wscale: current ln w = stored ln w + lwscale (FP64 mode)
    double lwhat_flat;  // ln of the flat prior (-inf when it reads 0)
    double W0;          // initial total weight
    double what_flat;   // flat prior W0/N (global entropy)
    double chi2;
    double Wsum;        // total stored weight of the last deposit
    double Wcheck;      // floating-point sum of the deposited weights (range check only)
    double Wrange;      // largest total weight the fixed-point sums can hold
    int pending;        // the previous step's force of change is still to be applied
    unsigned err;       // latched kErr* bits
    unsigned blocks_done;  // blocks of the running step kernel that have flushed their sums
    int smooth_pending;    // new raw cell means wait for the prior smoothing kernels
    unsigned smooth_blocks;   // blocks of the running smoothing kernel that have finished
    double smooth_lambda;  // smoothing weight of the last prior update
    double ups;            // mass-to-light ratio of the self-consistent potential
};

// What every block of a step reads before its first particle, written once per step by the
// finalize (the flags of step t + 1 in the types the step uses: a 64-bit modulo and an FP64
// division in every thread of every block cost 9,500 cycles of the mixed step at 2M particles,
// the FP64 pipe being that narrow; 1,000 now). Kept apart from Scalars, whose layout is that
// of the checkpoint files.
struct alignas(16) StepHead {
    int pending, prior_step, scf_step;
    float wscale, iwhat;      // mixed mode: weight scale, 1/flat prior (0 when it reads 0)
    int fresh;                // the self-consistent potential was rebuilt since the last push
    double lwscale, lwhat;    // FP64 mode: ln of both
};

template <class T>
struct State {
    T *x, *y, *z, *vx, *vy, *vz, *w;
    T *fa;            // force factor of the acceleration at the current positions (Model::cache_accel)
    T *ax, *ay, *az;  // self-consistent potential: the acceleration itself
    uint16_t *cell;
    uint16_t *ap;     // cached apertures (Model::ap_cache), null without the cache
    T *gx;            // cached exp(-nu^2/2) of Model::gx_group (FP64 mode), else null
    long long n;
};

// FP64 mode stores ln w instead of w: the exponential force-of-change update is
// then an addition and the entropy term -ln(w/what) a subtraction, so the only
// transcendental left per particle for the weight is the exp that recovers w for
// the deposit (mixed mode keeps w: its FP32 ln w would lose ~1e-6 relative per step).
template <class T>
constexpr bool kLogWeights = sizeof(T) == 8;

// The step can keep a(x_t) from the closing half-kick of one step for the opening
// half-kick of the next (the same function of the same positions, so bit-identical
// to recomputing it). Every potential here has a = -f (x, y, z) (spherical) or
// f (x, y, z / q^2) (flattened log halo) with one scalar force factor f, so the factor
// is kept (one state array read and written) and the components are rebuilt from it
// with the same multiplications: bit-identical to keeping the three components, in a
// third of the traffic. FP64 mode always does (it is bound by the FP64 pipe, not by
// HBM); mixed mode does where the force is dear (Model::cache_accel: the Hernquist +
// NFW potential, whose halo term takes a logarithm and a division).
template <class T>
constexpr bool kCacheAccel = sizeof(T) == 8;

// The self-consistent potential is not of the force-factor form: its three components are
// kept, and formed anew after a step that rebuilt the expansion (StepHead::fresh).
template <class T>
__host__ __device__ __forceinline__ bool keeps_accel(const Model &m)
{
    return m.pot != 3 && (kCacheAccel<T> || m.cache_accel);
}

// The finalize works through the observables in chunks of one warp: up to 32 consecutive
// apertures of one kind of one group, ordered by group, then aperture range, then kind, so
// that one warp sums a chunk's Delta_j^2 and one block holds every coefficient of a range of
// apertures. chi^2 adds the chunks in this order whatever the number of blocks and threads.
// The force-of-change records are linear in the coefficients c_j: an element of a record is
// sum_k coef_k c_(j0 + k stride) over the kinds of its group, with the factors laid out here
// (see upload_plan), and only the elements that are ever non-zero are listed.
struct ObsRow {
    double iscale, post, cw, Y, sig, isig;  // 1/fixed-point scale; factor of the raw sum; post / sig; data
    int j, pad;                             // observable, -1 for the padding of a chunk
};
struct RecElem {
    int dst, j0, stride, nk;  // element of the records; its terms
};
struct FinPlan {
    int n_chunks, n_elems, n_ranges, pad;
    const ObsRow *rows;      // 32 per chunk
    const RecElem *elems;    // ordered by aperture range
    const double *coef;      // [kind][element]
    const int2 *range;       // per aperture range: first chunk and first element (n_ranges + 1)
    double *csum;            // per chunk: sum of Delta_j^2 (finalize over several blocks)
};

struct Buffers {
    const unsigned char *tab;        // the tables of the step in the state type (see TabLayout)
    StepHead *head;
    const double *Vp, *isp;          // per aperture V_p and 1/sigma_p
    const float *Vpf, *ispf;         // FP32 copies of V_p and 1/sigma_p (mixed mode)
    const double *lcE;               // E_c table
    const float *lcEf;               // FP32 copy of it (mixed mode)
    const double *sig;
    const int *obs_kind;             // per observable: kind
    FinPlan plan;                    // the order of the finalize
    double *c;                       // per observable: coefficient of the force of change
    double *rec;                     // per aperture: the data term of eq. modFOC as polynomials in nu
    float *recf;                     // FP32 copy of rec (mixed mode reads it from global memory)
    double *prior;                   // per cell: prior (cell mean weight)
    double *iprior;                  // per cell: 1/prior (0 when the prior reads as 0)
    float *ipriorf;                  // FP32 copy of iprior (mixed mode)
    double *lprior;                  // per cell: ln prior (-inf when the prior reads as 0)
    long long *prior_count;          // per cell: particle count at the last update
    double *prior_raw;               // per cell: raw cell mean before smoothing (smoothing on)
    unsigned long long *pwin;        // window priors: (WPS + 1) x ncell words of cumulative sums
    const double *sV, *sVT, *sD;     // smoothing: eigenvectors of the grid penalty (V, V^T) and eigenvalues
    double *spart, *sz, *ss;         // smoothing scratch: chunk partial sums, V^T y, smoothed coefficients
    long long *hist;                 // global fixed-point sums
    double *ytil, *yraw, *delta;
    Scalars *sc;
};

// ---------------------------------------------------------------- math helpers
// FP32 (mixed mode) uses the hardware approximations on the device: exp and log
// through ex2/lg2 (relative error ~2^-21 |x| for exp), division through rcp. FP64
// keeps the correctly rounded functions.
__host__ __device__ __forceinline__ float d_sqrt(float x) { return sqrtf(x); }
__host__ __device__ __forceinline__ double d_sqrt(double x) { return sqrt(x); }
__host__ __device__ __forceinline__ float d_exp(float x)
{
#ifdef __CUDA_ARCH__
    return __expf(x);
#else
    return expf(x);
#endif
}
__host__ __device__ __forceinline__ double d_exp(double x) { return exp(x); }
__host__ __device__ __forceinline__ float d_log(float x)
{
#ifdef __CUDA_ARCH__
    return __logf(x);
#else
    return logf(x);
#endif
}
__host__ __device__ __forceinline__ double d_log(double x) { return log(x); }
__host__ __device__ __forceinline__ float d_div(float a, float b)
{
#ifdef __CUDA_ARCH__
    return __fdividef(a, b);
#else
    return a / b;
#endif
}
__host__ __device__ __forceinline__ double d_div(double a, double b) { return a / b; }
__host__ __device__ __forceinline__ float d_log1p(float x) { return log1pf(x); }
__host__ __device__ __forceinline__ double d_log1p(double x) { return log1p(x); }
__host__ __device__ __forceinline__ float d_floor(float x) { return floorf(x); }
__host__ __device__ __forceinline__ double d_floor(double x) { return floor(x); }
// Tests the FP64 step makes on bit patterns, so that they run on the integer pipe
// instead of the FP64 pipe (which bounds that step); FP32 keeps plain compares.
__host__ __device__ __forceinline__ bool is_zero(float v) { return v == 0.f; }
__host__ __device__ __forceinline__ bool is_zero(double v)
{
    return (bits_of(v) << 1) == 0;  // +0 or -0
}
__host__ __device__ __forceinline__ bool is_one(float v) { return v == 1.f; }
__host__ __device__ __forceinline__ bool is_one(double v) { return bits_of(v) == 0x3ff0000000000000ll; }
// a > b for a, b >= 0 (FP64: a positive NaN counts as greater)
__device__ __forceinline__ bool gt_nonneg(float a, float b) { return a > b; }
__device__ __forceinline__ bool gt_nonneg(double a, double b)
{
    return bits_of(a) > bits_of(b);
}
__device__ __forceinline__ bool is_neg_inf(double v)
{
    return bits_of(v) == static_cast<long long>(0xFFF0000000000000ull);
}

__host__ __device__ __forceinline__ bool d_finite(float x) { return isfinite(x); }
__host__ __device__ __forceinline__ bool d_finite(double x) { return isfinite(x); }

// ---------------------------------------------------------------- potentials

// a / q^2 of the flattened halo. FP64: the product with 1/q^2 and its exact residual (3 FP64
// instructions where a division takes 10), the correctly rounded quotient up to rare ties.
__host__ __device__ __forceinline__ float div_q2(const Cst<float> &k, float a) { return d_div(a, k.q2); }
__host__ __device__ __forceinline__ double div_q2(const Cst<double> &k, double a)
{
    const double t = a * k.iq2;
    return fma(fma(-t, k.q2, a), k.iq2, t);
}

// NFW enclosed-mass factor mu(q) = ln(1+q) - q/(1+q), FP64. For small q the two terms
// cancel: below q = 1e-3 the alternating series sum_k (-1)^k (k-1)/k q^k (Horner).
template <class T>
__host__ __device__ __forceinline__ T nfw_mu(T qq)
{
    if (qq < T(1e-3)) {
        T s = T(-10.0 / 11.0);
        s = fma(qq, s, T(9.0 / 10.0));
        s = fma(qq, s, T(-8.0 / 9.0));
        s = fma(qq, s, T(7.0 / 8.0));
        s = fma(qq, s, T(-6.0 / 7.0));
        s = fma(qq, s, T(5.0 / 6.0));
        s = fma(qq, s, T(-4.0 / 5.0));
        s = fma(qq, s, T(3.0 / 4.0));
        s = fma(qq, s, T(-2.0 / 3.0));
        s = fma(qq, s, T(0.5));
        return qq * qq * s;
    }
    return d_log1p(qq) - d_div(qq, T(1) + qq);
}

// FP32: ln(1+q) and mu(q) together without the library log1p. Below q = 1 both come
// from the series in s = q/(2+q) <= 1/3: ln(1+q) = 2 atanh(s) = 2 s sum_{k>=0} s^(2k)/(2k+1),
// and, since 2s - q/(1+q) = s t exactly (t = q/(1+q)),
//   mu = ln(1+q) - t = s t + 2 s^3 P(s^2),  P(u) = sum_{k>=0} u^k/(2k+3),
// a sum of positive terms with no cancellation (8 terms of P, truncation below 1e-9
// relative). Above, ln(1+q) from the hardware log2 (__logf: a few ulp) and
// mu = ln(1+q) - t >= 0.19 without cancellation.
__host__ __device__ __forceinline__ void nfw_logs(float q, float &l1, float &mu)
{
    const float t = d_div(q, 1.f + q);
    if (q < 1.f) {
        const float s = d_div(q, 2.f + q), u = s * s;
        float P = 1.f / 17.f;
#pragma unroll
        for (int k = 6; k >= 0; --k) P = fmaf(u, P, 1.f / float(2 * k + 3));
        const float s3P2 = 2.f * (s * u) * P;
        l1 = fmaf(2.f, s, s3P2);
        mu = fmaf(s, t, s3P2);
    } else {
        l1 = d_log(1.f + q);
        mu = l1 - t;
    }
}

// 1/n of a small integer, 1 <= n <= 6 (a division in the inner recurrences otherwise).
template <class T>
__device__ __forceinline__ T inv_small(int n)
{
    return n == 1 ? T(1) : n == 2 ? T(0.5) : n == 3 ? T(1.0 / 3.0) : n == 4 ? T(0.25) : n == 5 ? T(0.2) : T(1.0 / 6.0);
}

// Square root and quotient (b > 0) of the shell geometry: on the integer pipe in FP64.
__device__ __forceinline__ float g_sqrt(float x) { return d_sqrt(x); }
__device__ __forceinline__ double g_sqrt(double x) { return sqrt_int(x); }
__device__ __forceinline__ float g_div(float a, float b) { return d_div(a, b); }
__device__ __forceinline__ double g_div(double a, double b) { return div_int(a, b); }

// ---------------------------------------------------------------- self-consistent potential
//
// The stellar potential of pot 3 (Sec. 6) is the multipole expansion of the particles'
// luminosity on grid radii r_0 < ... < r_{n-1} (thin shells, see the host's description
// at m2m_potential). At r in the interval j (r_{j-1} <= r < r_j, r_{-1} = 0, r_n = infinity):
//   phi_star(x) = sum_lm [TA_lm(j) r^-(2l+1) + TB_lm(j)] R_lm(x),
// with R_lm = r^l Y_lm the regular solid harmonic, TA_lm(j) = C_l sum_{k<j} a_lm,k r_k^l (the
// shells inside) and TB_lm(j) = C_l sum_{k>=j} a_lm,k r_k^-(l+1) (the shells outside),
// C_l = -4 pi G Upsilon/(2l+1); the finalize builds these tables on update steps. R_lm =
// N_lm T_lm(z, r^2) Re or Im (x + iy)^m, where T_mm = (2m-1)!!, T_{m+1,m} = (2m+1) z T_mm and
// (l-m) T_lm = (2l-1) z T_{l-1,m} - (l+m-1) r^2 T_{l-2,m} (the recurrences of the associated
// Legendre functions times r^(l-m)); the gradient follows the same recurrences, carried as
// derivatives in z and r^2, with d(x + iy)^m = m (x + iy)^(m-1) (dx + i dy).
constexpr int kScfLmax = 6;
constexpr int kScfMaxRadii = 64;

template <class T>
__device__ __forceinline__ const T *scf_table(const Model &m);
template <>
__device__ __forceinline__ const double *scf_table<double>(const Model &m) { return m.scf_tab; }
template <>
__device__ __forceinline__ const float *scf_table<float>(const Model &m) { return m.scf_tabf; }

// Number of grid radii with r_k^2 <= r2: the interval j of the point.
template <class T>
__device__ __forceinline__ int scf_interval(const Model &m, T r2)
{
    int lo = 0, hi = m.scf_n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        const T rk = T(__ldg(m.scf_r + mid));
        if (rk * rk <= r2) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// phi_star (Upsilon included) at (x, y, z) and, if g is not null, its gradient.
template <class T>
__device__ T scf_field(const Model &m, T x, T y, T z, T *g)
{
    const T r2 = fma(x, x, fma(y, y, z * z));
    const int j = scf_interval(m, r2);
    const T *tab = scf_table<T>(m) + size_t(j) * m.scf_nlm * 2;
    const bool inner = j > 0;  // then r >= r_0 > 0
    const T ir2 = inner ? g_div(T(1), r2) : T(0);
    const T ir = inner ? g_sqrt(ir2) : T(0);
    const int L = m.scf_lmax;
    T phi = T(0), gx = T(0), gy = T(0), gz = T(0);
    T cm = T(1), sm = T(0), cm1 = T(0), sm1 = T(0);  // (x + iy)^m and (x + iy)^(m-1)
    T dfac = T(1);                                  // (2m-1)!!
    T irm = ir;                                     // r^-(2m+1)
    for (int mm = 0; mm <= L; ++mm) {
        T t1 = dfac, t1z = T(0), t1r = T(0);  // T_l and its z, r^2 derivatives, l = mm
        T t0 = T(0), t0z = T(0), t0r = T(0);  // T_(l-1)
        T irl = irm;
        for (int l = mm; l <= L; ++l) {
            if (l > mm) {  // the recurrence in l
                const T a = T(2 * l - 1), bq = T(l + mm - 1), il = inv_small<T>(l - mm);
                const T tn = (a * z * t1 - bq * r2 * t0) * il;
                const T tnz = (a * (t1 + z * t1z) - bq * r2 * t0z) * il;
                const T tnr = (a * z * t1r - bq * (t0 + r2 * t0r)) * il;
                t0 = t1; t0z = t1z; t0r = t1r;
                t1 = tn; t1z = tnz; t1r = tnr;
                irl *= ir2;
            }
            for (int v = 0; v < (mm > 0 ? 2 : 1); ++v) {
                const int idx = l * (l + 1) + (v == 0 ? mm : -mm);
                const T ta = tab[2 * idx], tb = tab[2 * idx + 1];
                const T N = sizeof(T) == 8 ? T(m.scf_norm[idx]) : T(m.scf_norm_f[idx]);
                const T P = v == 0 ? cm : sm;
                const T R = N * t1 * P;
                const T coef = fma(ta, irl, tb);
                phi = fma(coef, R, phi);
                if (g) {
                    // grad P: cos (m C_(m-1), -m S_(m-1), 0); sin (m S_(m-1), m C_(m-1), 0)
                    const T fm = T(mm);
                    const T px = v == 0 ? fm * cm1 : fm * sm1, py = v == 0 ? -fm * sm1 : fm * cm1;
                    const T gRx = N * fma(T(2) * x * t1r, P, t1 * px);
                    const T gRy = N * fma(T(2) * y * t1r, P, t1 * py);
                    const T gRz = N * (t1z + T(2) * z * t1r) * P;
                    const T rad = ta * T(2 * l + 1) * irl * ir2 * R;  // d r^-(2l+1) / dx_c = -(2l+1) r^-(2l+3) x_c
                    gx = fma(coef, gRx, gx) - rad * x;
                    gy = fma(coef, gRy, gy) - rad * y;
                    gz = fma(coef, gRz, gz) - rad * z;
                }
            }
        }
        cm1 = cm;
        sm1 = sm;
        const T cn = fma(cm, x, -(sm * y));
        sm = fma(cm, y, sm * x);
        cm = cn;
        dfac *= T(2 * mm + 1);
        irm *= ir2;
    }
    if (g) {
        g[0] = gx;
        g[1] = gy;
        g[2] = gz;
    }
    return phi;
}

// Potential and acceleration of the flattened logarithmic halo (eq. log_halo).
template <class T>
__host__ __device__ __forceinline__ T log_halo_phi(const Cst<T> &k, T x, T y, T z)
{
    const T D = fma(x, x, fma(y, y, k.r0sq)) + d_div(z * z, k.q2);
    return T(0.5) * k.v0sq * d_log(D);
}

template <class T>
__device__ __forceinline__ T scf_potential(const Model &m, const Cst<T> &k, T x, T y, T z)
{
#ifdef __CUDA_ARCH__
    return scf_field<T>(m, x, y, z, nullptr) + log_halo_phi(k, x, y, z);
#else
    return T(0);
#endif
}

template <class T>
__device__ __forceinline__ void scf_accel(const Model &m, const Cst<T> &k, T x, T y, T z, T &ax, T &ay, T &az)
{
    T g[3];
    scf_field<T>(m, x, y, z, g);
    const T D = fma(x, x, fma(y, y, k.r0sq)) + g_div(z * z, k.q2);
    const T f = -g_div(k.v0sq, D);
    ax = fma(f, x, -g[0]);
    ay = fma(f, y, -g[1]);
    az = g_div(f * z, k.q2) - g[2];
}

// Energy and v_c^2 of the circular orbit of radius R on the x axis of the self-consistent
// potential. There theta = pi/2 and phi = 0, so within an interval of the grid phi_star is
// sum_l A_l R^-(l+1) + B_l R^l, with A_l, B_l summed over m by the finalize (scf_axis), and its
// derivative R d/dR follows term by term: some ten operations per l where the field takes a
// hundred per (l, m), in the bisection for Lc(E) that runs 60 times per particle and update.
template <class T>
__device__ __forceinline__ T scf_circ(const Model &m, const Cst<T> &k, T R, T &vc2)
{
    const T R2 = R * R;
    const int j = scf_interval(m, R2);
    const double *ax = m.scf_tab + size_t(m.scf_n + 1) * m.scf_nlm * 2 + size_t(j) * (m.scf_lmax + 1) * 2;
    const T iR = j > 0 ? g_div(T(1), R) : T(0);
    T phi = T(0), v = T(0), a = iR, p = T(1);
    for (int l = 0; l <= m.scf_lmax; ++l) {
        const T ta = T(__ldcg(ax + 2 * l)) * a, tb = T(__ldcg(ax + 2 * l + 1)) * p;
        phi += ta + tb;
        v += T(l) * tb - T(l + 1) * ta;
        a *= iR;
        p *= R;
    }
    const T D = R2 + k.r0sq;
    phi += T(0.5) * k.v0sq * d_log(D);
    vc2 = v + g_div(k.v0sq * R2, D);
    return phi + T(0.5) * vc2;
}

// -phi of the spherical potentials at r (ir = 1/r), G M/(r + a) + G M_s ln(1 + r/r_s)/r, and, if
// vc2 is not null, v_c^2 = G M r/(r + a)^2 + G M_s mu/r.
__host__ __device__ __forceinline__ Big well_big(const Model &m, const Cst<double> &k, const Big &r, const Big &ir,
                                                 const u64 *ln, Big *vc2)
{
    const Big gz = big_norm(big_mul_raw(big_rcp(big_add(r, big_of(k.a))), big_of(k.GM)));
    Big w = gz;
    if (vc2) {
        const Big z = big_rcp(big_add(r, big_of(k.a)));
        *vc2 = big_norm(big_mul_raw(big_mul_raw(gz, z), r));
    }
    if (m.pot == 1) {
        Big l1;
        const Big mu = nfw_mu_big(k.rs, r, ln, &l1);
        const Big h = big_norm(big_mul_raw(ir, big_of(k.GMs)));
        w = big_add(w, big_norm(big_mul_raw(h, l1)));
        if (vc2) *vc2 = big_add(*vc2, big_norm(big_mul_raw(h, mu)));
    }
    return w;
}

// fn: FP64 mode, the tables of the integer functions (null: the library's).
struct FnTables {
    const u64 *et, *ln;
};

// The potential. SCF: whether the code of the self-consistent one is compiled in (only the generic
// step kernel and the helpers around it need it; the kernels specialised to an observable
// shape run the other potentials without its registers).
template <class T, bool SCF = true>
__host__ __device__ __forceinline__ T potential(const Model &m, const Cst<T> &k, T x, T y, T z,
                                                FnTables fn = FnTables{nullptr, nullptr})
{
#ifdef __CUDA_ARCH__
    if constexpr (SCF) {
        if (m.pot == 3) return scf_potential(m, k, x, y, z);
    }
#endif
    if (m.pot == 2) {
        const T D = fma(x, x, fma(y, y, k.r0sq)) + d_div(z * z, k.q2);
        return T(0.5) * k.v0sq * d_log(D);
    }
    if constexpr (sizeof(T) == 8) {
        const T r2 = fma(x, x, fma(y, y, z * z));
        if (fn.ln && m.int_force && big_range(r2)) {
            Big r, ir;
            big_rsqrt(big_of(r2), ir, r);
            return -big_double(well_big(m, k, r, ir, fn.ln, nullptr));
        }
    }
    const T r = d_sqrt(fma(x, x, fma(y, y, z * z)));
    T phi = -d_div(k.GM, r + k.a);
    if (m.pot == 1) {
        if (!(r > T(0))) return phi + k.hn_phi0;
        T l1;
        if constexpr (sizeof(T) == 4) {
            T mu;
            nfw_logs(d_div(r, k.rs), l1, mu);
        } else {
            l1 = d_log1p(d_div(r, k.rs));
        }
        phi -= d_div(k.GMs * l1, r);
    }
    return phi;
}

// Force factor f of the acceleration at (x, y, z): a = -f (x, y, z) in the spherical
// potentials (f = g(r)/r with g = G M(<r)/r^2), a = f (x, y, z/q^2) in the flattened log
// halo (f = -v0^2/D). lnt: FP64 mode, the logarithm table of the integer force factors
// (fp64_int.cuh); null takes the library functions. Per particle the Hernquist factor costs 3
// FP64 instructions so instead of 27 (with the halo 3 instead of about 90).
template <class T>
__host__ __device__ __forceinline__ T accel_factor(const Model &m, const Cst<T> &k, T x, T y, T z,
                                                   const u64 *lnt = nullptr)
{
    if (m.pot == 2) {
        if constexpr (sizeof(T) == 8) {
            const T D = fma(x, x, fma(y, y, k.r0sq)) + (lnt && m.int_force ? div_q2(k, z * z) : d_div(z * z, k.q2));
            if (lnt && m.int_force && big_range(D))
                return -big_double(big_norm(big_mul_raw(big_rcp(big_of(D)), big_of(k.v0sq))));
            return -d_div(k.v0sq, D);
        }
        const T D = fma(x, x, fma(y, y, k.r0sq)) + d_div(z * z, k.q2);
        return -d_div(k.v0sq, D);
    }
    const T r2 = fma(x, x, fma(y, y, z * z));
    if constexpr (sizeof(T) == 8) {
        if (lnt && m.int_force && big_range(r2)) {
            Big r, ir;
            big_rsqrt(big_of(r2), ir, r);
            Big f = hernquist_big(k.GM, k.a, r, ir);
            if (m.pot == 1) f = big_add(f, nfw_big(k.GMs, k.rs, r, ir, lnt));
            return big_double(f);
        }
    }
    if (is_zero(r2)) return T(0);
    const T r = d_sqrt(r2);
    const T ra = r + k.a;
    T f = d_div(k.GM, ra * ra * r);
    if (m.pot == 1) {
        T mu;
        if constexpr (sizeof(T) == 4) {
            T l1;
            nfw_logs(d_div(r, k.rs), l1, mu);
        } else {
            mu = nfw_mu(d_div(r, k.rs));
        }
        f += d_div(k.GMs * mu, r2 * r);
    }
    return f;
}

// The acceleration from its force factor (see accel_factor).
template <class T>
__host__ __device__ __forceinline__ void accel_from(const Model &m, const Cst<T> &k, T f, T x, T y, T z, T &ax,
                                                    T &ay, T &az)
{
    if (m.pot == 2) {
        ax = f * x;
        ay = f * y;
        az = m.int_force ? div_q2(k, f * z) : d_div(f * z, k.q2);
        return;
    }
    ax = -f * x;
    ay = -f * y;
    az = -f * z;
}

template <class T, bool SCF = true>
__host__ __device__ __forceinline__ void accel(const Model &m, const Cst<T> &k, T x, T y, T z, T &ax, T &ay,
                                               T &az)
{
#ifdef __CUDA_ARCH__
    if constexpr (SCF) {
        if (m.pot == 3) {
            scf_accel(m, k, x, y, z, ax, ay, az);
            return;
        }
    }
#endif
    accel_from(m, k, accel_factor(m, k, x, y, z), x, y, z, ax, ay, az);
}

// v += dt/2 a from the force factor. FP64 forms dt f/2 once (four FP64 instructions instead
// of six; the spherical potentials, and x, y of the halo).
__device__ __forceinline__ void kick(const Model &m, const Cst<float> &k, float f, float x, float y, float z, float &vx,
                                     float &vy, float &vz)
{
    float ax, ay, az;
    accel_from(m, k, f, x, y, z, ax, ay, az);
    vx = fma(k.hdt, ax, vx);
    vy = fma(k.hdt, ay, vy);
    vz = fma(k.hdt, az, vz);
}
__device__ __forceinline__ void kick(const Model &m, const Cst<double> &k, double f, double x, double y, double z,
                                     double &vx, double &vy, double &vz)
{
    const double h = m.pot == 2 ? k.hdt * f : -(k.hdt * f);
    vx = fma(h, x, vx);
    vy = fma(h, y, vy);
    vz = fma(m.pot == 2 ? (m.int_force ? div_q2(k, h) : d_div(h, k.q2)) : h, z, vz);
}

// One kick-drift-kick leap-frog step from the force factor f at the start position;
// returns the factor at the end position in f.
template <class T>
__device__ __forceinline__ void leapfrog_from(const Model &m, const Cst<T> &k, T &x, T &y, T &z, T &vx, T &vy, T &vz,
                                              T &f, const u64 *lnt)
{
    kick(m, k, f, x, y, z, vx, vy, vz);
    x = fma(k.dt, vx, x);
    y = fma(k.dt, vy, y);
    z = fma(k.dt, vz, z);
    f = accel_factor(m, k, x, y, z, lnt);
    kick(m, k, f, x, y, z, vx, vy, vz);
}

// One kick-drift-kick leap-frog step.
template <class T>
__device__ __forceinline__ void leapfrog(const Model &m, const Cst<T> &k, T &x, T &y, T &z, T &vx, T &vy, T &vz)
{
    T f = accel_factor(m, k, x, y, z);
    leapfrog_from(m, k, x, y, z, vx, vy, vz, f, nullptr);
}

// The same from the acceleration (ax, ay, az) at the start, which becomes that at the end
// (the self-consistent potential).
template <class T>
__device__ __forceinline__ void leapfrog_scf(const Model &m, const Cst<T> &k, T &x, T &y, T &z, T &vx, T &vy, T &vz,
                                             T &ax, T &ay, T &az)
{
    vx = fma(k.hdt, ax, vx);
    vy = fma(k.hdt, ay, vy);
    vz = fma(k.hdt, az, vz);
    x = fma(k.dt, vx, x);
    y = fma(k.dt, vy, y);
    z = fma(k.dt, vz, z);
    accel<T, true>(m, k, x, y, z, ax, ay, az);
    vx = fma(k.hdt, ax, vx);
    vy = fma(k.hdt, ay, vy);
    vz = fma(k.hdt, az, vz);
}

// ---------------------------------------------------------------- observables

// Sky coordinates for the line of sight n = (0, sin i, cos i): X = x (not
// returned), Y = y cos i - z sin i, v_los = vy sin i + vz cos i.
template <class T>
__device__ __forceinline__ void project(const Cst<T> &k, T y, T z, T vy, T vz, T &Y, T &vlos)
{
    if (sizeof(T) == 8 && is_zero(k.sin_i) && is_one(k.cos_i)) {  // face on: the same values, no FP64 instruction
        Y = y;
        vlos = vz;
        return;
    }
    Y = fma(y, k.cos_i, -(z * k.sin_i));
    vlos = fma(vy, k.sin_i, vz * k.cos_i);
}

// x >= 0 truncated to FP32 (0 below its normal range, its largest value above) with integer
// operations: the conversion would wait for the FP64 pipe.
__device__ __forceinline__ float float_near(double x)
{
    const int hi = __double2hiint(x) - ((1023 - 127) << 20);
    const unsigned lo = unsigned(__double2loint(x));
    return hi < (1 << 20) ? 0.f : (hi >= (255 << 20) ? 3.4e38f : __uint_as_float((unsigned(hi) << 3) | (lo >> 29)));
}

// Aperture of sky point (X, Y) in group G, or -1: half-open annuli
// [edge_p, edge_p+1) in R = sqrt(X^2 + Y^2), decided on R^2 against squared edges
// (so the decision can differ from one made on R only within a few ulp of an
// edge), or pixel p = py nx + px with px = floor((X - xlo) nx / (xhi - xlo)).
// Annuli start from a candidate found from log2 R^2 in FP32 (the annulus itself
// for log-uniform edges, else a lookup table) and are corrected by exact
// comparisons; without a table (lut_n = 0) a binary search is used.
//
// FP64: for R^2 >= 0 the IEEE bit pattern orders like the value, so the
// comparisons run on the integer pipe.
template <unsigned M>
__device__ __forceinline__ int aperture(const GroupDesc &G, const double *esq, const unsigned short *lut,
                                        double X, double Y)
{
    if (!GP<M>::pixels(G)) {
        const double R2 = fma(X, X, Y * Y);
        const long long r = bits_of(R2);
        const double *e = esq + G.edge_off;
        if (r < bits_of(e[0]) || r >= bits_of(e[G.n_ap])) return -1;
        int p;
        if (G.lut_n > 0) {
            int b = __float2int_rd((__log2f(float_near(R2)) - G.l0) * G.lscale);
            b = b < 0 ? 0 : (b >= G.lut_n ? G.lut_n - 1 : b);
            p = G.lut_identity ? b : int(lut[G.lut_off + b]);
            // the candidate is right but within rounding of an edge or for crowded edges
            if (r < bits_of(e[p]) || r >= bits_of(e[p + 1])) {
                while (p > 0 && r < bits_of(e[p])) --p;
                while (r >= bits_of(e[p + 1])) ++p;
            }
        } else {
            int lo = 0, hi = G.n_ap;  // e[lo] <= R^2 < e[hi]
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (bits_of(e[mid]) <= r) lo = mid;
                else hi = mid;
            }
            p = lo;
        }
        return p;
    }
    const double fx = floor((X - G.xlo) * G.nx / G.xw);
    const double fy = floor((Y - G.ylo) * G.ny / G.yw);
    if (!(fx >= 0.0) || !(fx < G.nx) || !(fy >= 0.0) || !(fy < G.ny)) return -1;
    return int(fy) * G.nx + int(fx);
}

template <unsigned M>
__device__ __forceinline__ int aperture(const GroupDesc &G, const float *e2s, const unsigned short *lut, float X,
                                        float Y)
{
    if (!GP<M>::pixels(G)) {
        const float R2 = fmaf(X, X, Y * Y);
        if (!(R2 >= G.e0sq_f) || !(R2 < G.ensq_f)) return -1;
        int b = __float2int_rd((__log2f(R2) - G.l0) * G.lscale);
        b = b < 0 ? 0 : (b >= G.lut_n ? G.lut_n - 1 : b);
        int p = G.lut_identity ? b : int(lut[G.lut_off + b]);
        const float *e = e2s + G.edge_off;
        // the candidate is right but within rounding of an edge or for crowded edges
        if (R2 < e[p] || R2 >= e[p + 1]) {
            while (p > 0 && R2 < e[p]) --p;
            while (R2 >= e[p + 1]) ++p;
        }
        return p;
    }
    const float fx = floorf((X - G.xlo_f) * G.ixw);
    const float fy = floorf((Y - G.ylo_f) * G.iyw);
    if (!(fx >= 0.f) || !(fx < float(G.nx)) || !(fy >= 0.f) || !(fy < float(G.ny))) return -1;
    return int(fy) * G.nx + int(fx);
}

// ---------------------------------------------------------------- kernel values

// c_n = sqrt(2^(1-n)/n!): K_n = 2 sqrt(pi) u_n(nu) = c_n H_n(nu) exp(-nu^2/2) (eq. lumghn).
__host__ __device__ constexpr double gh_c(int n)
{
    return n == 0 ? 1.4142135623730950488
         : n == 1 ? 1.0
         : n == 2 ? 0.5
         : n == 3 ? 0.20412414523193150818
         : n == 4 ? 0.072168783648703220563
         : n == 5 ? 0.022821773229381921355
                  : 0.0065881721129167866018;
}

enum { kClassMass = 0, kClassVel = 1, kClassGH = 2 };  // fixed-point scale class

template <class T>
struct Tables {
    const T *esq;         // per group squared edges
    const unsigned short *lut;
    const T *vp, *isp;
    const u64 *et, *ln;   // FP64 mode: the tables of exp_int and ln_frac (null without one)
};

// Tables of the observables without a context: constant memory instead of a fit's tables.
struct StaticTables {
    const double *esq;
    const unsigned short *lut;
    const double *vp, *isp;
    const double *e2;     // 2^(j/32), j < 32 (exp_tab)
};

// exp of the weights, and exp(-t/2) of the kernel values: the ex2-based approximation in mixed
// mode, the integer exponential in FP64 mode.
__device__ __forceinline__ float kexp(const Tables<float> &, float x) { return __expf(x); }
__device__ __forceinline__ double kexp(const Tables<double> &tb, double x) { return exp_int(x, tb.et); }
__device__ __forceinline__ float kexp_mhalf(const Tables<float> &, float t) { return __expf(-0.5f * t); }
__device__ __forceinline__ double kexp_mhalf(const Tables<double> &tb, double t) { return exp_mhalf(t, tb.et); }
__device__ __forceinline__ double kexp_mhalf(const StaticTables &tb, double t) { return exp_tab(-0.5 * t, tb.e2); }

// Coefficient of t^k, t = nu^2, in c_n H_n(nu) (n even) or c_n H_n(nu)/nu (n odd), from the
// explicit sum H_n = n! sum_j (-1)^j (2 nu)^(n-2j) / (j! (n-2j)!).
__host__ __device__ constexpr double gh_coef(int n, int k)
{
    const int j = n / 2 - k, p = n - 2 * j;
    double v = gh_c(n) * (j % 2 ? -1.0 : 1.0);
    for (int i = 2; i <= n; ++i) v *= i;
    for (int i = 2; i <= j; ++i) v /= i;
    for (int i = 2; i <= p; ++i) v /= i;
    for (int i = 0; i < p; ++i) v *= 2.0;
    return v;
}
template <int n, class T>
__device__ __forceinline__ T gh_poly(T t)
{
    T s = T(gh_coef(n, n / 2));
#pragma unroll
    for (int k = n / 2 - 1; k >= 0; --k) s = fma(s, t, T(gh_coef(n, k)));
    return s;
}

// a b of the kernel values: in FP64 on the integer pipe (mul_int), correctly rounded up to ties.
__device__ __forceinline__ float product(float a, float b) { return a * b; }
__device__ __forceinline__ double product(double a, double b) { return mul_int(a, b); }

// Emits emit(slot, w K_slot, class, kind index in the group) for every kernel of group G
// at aperture p:
// surface mass (K = 1), v_los^2 (vv), v_los, and the Gauss-Hermite b_n: c_n H_n(nu) as a
// polynomial in nu^2 times w exp(-nu^2/2), times nu for odd n (8 multiplications and fused
// multiply-adds for h3 and h4, 15 by the recurrence in n).
template <unsigned M, class T, class TB, class F>
__device__ __forceinline__ void group_kernels(const GroupDesc &G, const TB &tb, int p, T vlos, T vv, T w, F &&emit,
                                              T *gexp_out = nullptr)
{
    using P = GP<M>;
    const int base = G.obs_off + p;
    if (P::mass(G)) emit(base + G.k_mass * G.n_ap, w, kClassMass, G.k_mass);
    if (P::v2(G)) emit(base + G.k_v2 * G.n_ap, product(w, vv), kClassVel, G.k_v2);
    if (P::v1(G)) emit(base + G.k_v1 * G.n_ap, w * vlos, kClassVel, G.k_v1);
    if (P::max_gh(G) >= 0) {
        const T nu = (vlos - tb.vp[G.ap_off + p]) * tb.isp[G.ap_off + p];
        const T t = product(nu, nu);
        const T ge = kexp_mhalf(tb, t);
        if (gexp_out) *gexp_out = ge;
        const T we = product(w, ge), wo = product(we, nu);
        auto put = [&](auto N) {
            constexpr int n = decltype(N)::value;
            if (P::gh(G, n)) emit(base + G.k_gh[n] * G.n_ap, product(gh_poly<n>(t), n % 2 ? wo : we), kClassGH, G.k_gh[n]);
        };
        put(std::integral_constant<int, 0>{});
        put(std::integral_constant<int, 1>{});
        put(std::integral_constant<int, 2>{});
        put(std::integral_constant<int, 3>{});
        put(std::integral_constant<int, 4>{});
        put(std::integral_constant<int, 5>{});
        put(std::integral_constant<int, 6>{});
    }
}

// The data term of eq. modFOC, sum_j K_j c_j, for one particle. In aperture p of a
// group every kernel is a polynomial in nu = (v_los - V_p)/sigma_p, the Gauss-
// Hermite ones times exp(-nu^2/2), so the finalize folds the coefficients c_j into
// one record per aperture, r = [V_p, 1/sigma_p, q0, q1, q2, p0 .. p_nmax], and
// sum_j K_j c_j = q0 + q1 nu + q2 nu^2 + exp(-nu^2/2) sum_n p_n nu^n
// (groups without Gauss-Hermite kernels use V = 0, 1/sigma = 1, i.e. nu = v_los).
// The first n values of a record (n <= 12), with 16-byte loads: records start on 16-byte
// boundaries (Model::rec_len is a multiple of 4).
__device__ __forceinline__ void load_record(const float *r, float *v, int n)
{
#pragma unroll
    for (int q = 0; q < 3; ++q)
        if (4 * q < n) {
            const float4 a = reinterpret_cast<const float4 *>(r)[q];
            v[4 * q] = a.x;
            v[4 * q + 1] = a.y;
            v[4 * q + 2] = a.z;
            v[4 * q + 3] = a.w;
        }
}
__device__ __forceinline__ void load_record(const double *r, double *v, int n)
{
#pragma unroll
    for (int q = 0; q < 6; ++q)
        if (2 * q < n) {
            const double2 a = reinterpret_cast<const double2 *>(r)[q];
            v[2 * q] = a.x;
            v[2 * q + 1] = a.y;
        }
}

template <unsigned M, class T>
__device__ __forceinline__ T group_data(const Model &m, const GroupDesc &G, const Tables<T> &tb, const T *rec, int p,
                                        T vlos, const T *gexp = nullptr)
{
    const T *rp = rec + (G.ap_off + p) * m.rec_len;
    const int nmax = GP<M>::max_gh(G);
    if (!GP<M>::v2(G) && !GP<M>::v1(G) && nmax < 0) return rp[2];  // surface mass only: a constant
    T r[12];
    load_record(rp, r, 6 + nmax);
    const T nu = (vlos - r[0]) * r[1];
    T d = fma(nu, fma(nu, r[4], r[3]), r[2]);
    if (nmax >= 0) {
        T poly = T(0);
#pragma unroll
        for (int n = 6; n >= 0; --n)
            if (n <= nmax) poly = fma(poly, nu, r[5 + n]);
        d = fma(gexp ? *gexp : kexp_mhalf(tb, nu * nu), poly, d);
    }
    return d;
}

// ---- shells: the spherical-harmonic density coefficients of eq. alm
//
// a_lm,p = sum_i w_i gamma_p(r_i) Y_lm(theta_i, phi_i) on grid radii r_0 < ... < r_{n-1}
// (the total luminosity is carried by the weights). gamma is the cloud-in-cell weight:
// between r_{p-1} and r_p linear in r, inside r_0 all on point 0, none beyond r_{n-1}.
// Y_lm is the real spherical harmonic of unit norm without the Condon-Shortley phase,
// from the recurrences P_m^m = (2m-1)!! sin^m, P_{m+1}^m = (2m+1) cos P_m^m,
// (l-m) P_l^m = (2l-1) cos P_{l-1}^m - (l+m-1) P_{l-2}^m, and cos(m phi), sin(m phi) as the
// powers of cos phi + i sin phi.

// Grid points and cloud-in-cell weights of squared radius r2 (the group's squared grid
// radii at esq + edge_off): returns 0, 1 (point p0, weight 1) or 2 (p0 and p0 + 1).
template <class T>
__device__ __forceinline__ int shell_cic(const GroupDesc &G, const T *esq, T r2, int &p0, T &g0, T &g1)
{
    const T *e = esq + G.edge_off;
    const int n = G.n_ap;
    if (!(r2 < e[n - 1])) return 0;
    if (r2 < e[0]) {
        p0 = 0;
        g0 = T(1);
        g1 = T(0);
        return 1;
    }
    int lo = 0, hi = n - 1;  // e[lo] <= r2 < e[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (e[mid] <= r2) lo = mid;
        else hi = mid;
    }
    const T r = g_sqrt(r2), ra = g_sqrt(e[lo]), rb = g_sqrt(e[hi]);
    const T d = rb - ra;
    p0 = lo;
    g0 = g_div(rb - r, d);
    g1 = g_div(r - ra, d);
    return 2;
}

// Direction cosines of (x, y, z): cos and sin of theta (from the z axis) and of phi;
// theta = 0 at the centre and phi = 0 on the z axis.
template <class T>
__device__ __forceinline__ void shell_angles(T x, T y, T z, T &ct, T &st, T &cp, T &sp)
{
    // explicit fused forms: the same rounding in every kernel that inlines this
    const T R2 = fma(x, x, y * y);
    const T R = g_sqrt(R2), r = g_sqrt(fma(z, z, R2));
    const bool c = r > T(0), a = R > T(0);
    ct = c ? g_div(z, r) : T(1);
    st = c ? g_div(R, r) : T(0);
    cp = a ? g_div(x, R) : T(1);
    sp = a ? g_div(y, R) : T(0);
}

// f(kk, Y_lm) for every kind kk of shell group g: one sweep over l for each |m| (every P_l^m once,
// for the cosine and the sine; a sweep per kind takes three times as many FP64 instructions
// for l <= 4).
template <class T, class F>
__device__ __forceinline__ void shell_sweep(const Model &m, int g, const GroupDesc &G, T ct, T st, T cp, T sp, F &&f)
{
    const int L = m.alm_lmax[g];
    T cm = T(1), sm = T(0), pmm = T(1);
    for (int mm = 0; mm <= L; ++mm) {
        T p0 = T(0), p1 = pmm;
        for (int l = mm; l <= L; ++l) {
            if (l > mm) {
                const T p2 = fma(ct * T(2 * l - 1), p1, -(T(l + mm - 1) * p0)) * inv_small<T>(l - mm);
                p0 = p1;
                p1 = p2;
            }
            for (int v = 0; v < (mm > 0 ? 2 : 1); ++v) {
                const int kk = m.alm_k[g][l * (l + 1) + (v == 0 ? mm : -mm)];
                if (kk < 0) continue;
                const T nrm = sizeof(T) == 8 ? T(G.alm_norm[kk]) : T(G.alm_norm_f[kk]);
                f(kk, nrm * p1 * (v == 0 ? cm : sm));
            }
        }
        const T cn = fma(cm, cp, -(sm * sp));
        sm = fma(sm, cp, cm * sp);
        cm = cn;
        pmm *= T(2 * mm + 1) * st;
    }
}

// emit(slot, w K_slot, class, kind index) for every a_lm of the group at the particle's
// one or two grid points.
template <class T, class F>
__device__ __forceinline__ void shell_kernels(const Model &m, int g, const Tables<T> &tb, T x, T y, T z, T w, F &&emit)
{
    const GroupDesc &G = m.g[g];
    int p0 = 0;
    T g0 = T(0), g1 = T(0);
    const int np = shell_cic(G, tb.esq, fma(z, z, fma(x, x, y * y)), p0, g0, g1);
    if (np == 0) return;
    T ct, st, cp, sp;
    shell_angles(x, y, z, ct, st, cp, sp);
    shell_sweep(m, g, G, ct, st, cp, sp, [&](int kk, T Y) {
        const T v = w * Y;
        const int j = G.obs_off + kk * G.n_ap + p0;
        emit(j, g0 * v, kClassGH, kk);
        if (np == 2) emit(j + 1, g1 * v, kClassGH, kk);
    });
}

// sum_j K_j c_j over the group's a_lm: the records of a shell group hold c_j per kind.
template <class T>
__device__ __forceinline__ T shell_data(const Model &m, int g, const Tables<T> &tb, const T *rec, T x, T y, T z)
{
    const GroupDesc &G = m.g[g];
    int p0 = 0;
    T g0 = T(0), g1 = T(0);
    const int np = shell_cic(G, tb.esq, fma(z, z, fma(x, x, y * y)), p0, g0, g1);
    if (np == 0) return T(0);
    T ct, st, cp, sp;
    shell_angles(x, y, z, ct, st, cp, sp);
    const T *r0 = rec + (G.ap_off + p0) * m.rec_len;
    T d0 = T(0), d1 = T(0);
    shell_sweep(m, g, G, ct, st, cp, sp, [&](int kk, T Y) {
        d0 = fma(Y, r0[kk], d0);
        if (np == 2) d1 = fma(Y, r0[m.rec_len + kk], d1);
    });
    return fma(g0, d0, g1 * d1);
}

template <unsigned... Ms, class T>
__device__ __forceinline__ T data_term(const Model &m, const Tables<T> &tb, const T *rec, T x, T y, T z, T X,
                                       T Y, T vlos)
{
    T data = T(0);
    each_group<0, Ms...>(m, [&](auto P, int g) {
        constexpr unsigned M = decltype(P)::mask;
        const GroupDesc &G = m.g[g];
        if (GP<M>::shells(G)) {
            data += shell_data(m, g, tb, rec, x, y, z);
            return;
        }
        const int p = aperture<M>(G, tb.esq, tb.lut, X, Y);
        if (p >= 0) data += group_data<M>(m, G, tb, rec, p, vlos);
    });
    return data;
}

// Aperture of group g in a cached code (Model::ap_cache), -1 outside.
__device__ __forceinline__ int ap_decode(const Model &m, unsigned code, int g)
{
    if (m.ap_cache == 2) return code == kApNone16 ? -1 : int(code);
    const unsigned a = (code >> (8 * g)) & 0xFFu;
    return a == kApNone8 ? -1 : int(a);
}

__device__ __forceinline__ unsigned ap_encode(const Model &m, unsigned code, int g, int p)
{
    if (m.ap_cache == 2) return p < 0 ? kApNone16 : unsigned(p);
    return (code & ~(0xFFu << (8 * g))) | ((p < 0 ? kApNone8 : unsigned(p)) << (8 * g));
}

// data_term with the apertures taken from a cached code.
template <unsigned... Ms, class T>
__device__ __forceinline__ T data_term_cached(const Model &m, const Tables<T> &tb, const T *rec, unsigned code,
                                              T vlos, const T *gexp)
{
    T data = T(0);
    each_group<0, Ms...>(m, [&](auto P, int g) {
        constexpr unsigned M = decltype(P)::mask;
        const int p = ap_decode(m, code, g);
        if (p >= 0) data += group_data<M>(m, m.g[g], tb, rec, p, vlos, g == m.gx_group ? gexp : nullptr);
    });
    return data;
}

// ---- deposits of the self-consistent potential

// emit(slot, w gamma_k Y_lm) of the expansion (Sec. 6): the particle's luminosity on its
// one or two grid points, cloud-in-cell weights as eq. alm except that r < r_0 goes wholly to
// point 0 and r >= r_{n-1} wholly to point n-1; Y_lm from the associated-Legendre recurrences
// in cos(theta) and the powers of cos(phi) + i sin(phi).
template <class T, class F>
__device__ __forceinline__ void scf_deposit(const Model &m, T x, T y, T z, T w, F &&emit)
{
    const T r2 = fma(x, x, fma(y, y, z * z));
    const int j = scf_interval(m, r2);
    int k0;
    T g0 = T(1), g1 = T(0);
    if (j == 0) {
        k0 = 0;
    } else if (j == m.scf_n) {
        k0 = m.scf_n - 1;
    } else {
        const T r = d_sqrt(r2), ra = T(__ldg(m.scf_r + j - 1)), rb = T(__ldg(m.scf_r + j));
        k0 = j - 1;
        g0 = d_div(rb - r, rb - ra);
        g1 = d_div(r - ra, rb - ra);
    }
    T ct, st, cp, sp;
    shell_angles(x, y, z, ct, st, cp, sp);
    const int L = m.scf_lmax, nlm = m.scf_nlm;
    const int s0 = m.off_scf + k0 * nlm;
    T cm = T(1), sm = T(0), pmm = T(1);
    for (int mm = 0; mm <= L; ++mm) {
        T p0 = T(0), p1 = pmm;
        for (int l = mm; l <= L; ++l) {
            if (l > mm) {
                const T p2 = fma(ct * T(2 * l - 1), p1, -(T(l + mm - 1) * p0)) * inv_small<T>(l - mm);
                p0 = p1;
                p1 = p2;
            }
            for (int v = 0; v < (mm > 0 ? 2 : 1); ++v) {
                const int idx = l * (l + 1) + (v == 0 ? mm : -mm);
                const T N = sizeof(T) == 8 ? T(m.scf_norm[idx]) : T(m.scf_norm_f[idx]);
                const T Y = N * p1 * (v == 0 ? cm : sm);
                const T wy = w * Y;
                emit(s0 + idx, g0 * wy);
                if (g1 != T(0)) emit(s0 + nlm + idx, g1 * wy);
            }
        }
        const T cn = fma(cm, cp, -(sm * sp));
        sm = fma(sm, cp, cm * sp);
        cm = cn;
        pmm *= T(2 * mm + 1) * st;
    }
}

// emit(observable, D, class) of the derivatives of the kinematic kernels of group G at
// aperture p with respect to ln Upsilon when the velocities scale as Upsilon^(1/2):
// D = 1/2 w v_los dK/dv_los; w v_los^2 for v_los^2 (class kClassVel), and for b_n, with
// K_n = c_n H_n(nu) e^(-nu^2/2), 1/2 w v_los c_n (2n H_(n-1) - nu H_n) e^(-nu^2/2)/sigma_p
// (class kClassDv).
constexpr int kClassDv = 3;
template <unsigned M, class T, class F>
__device__ __forceinline__ void group_dkernels(const GroupDesc &G, const Tables<T> &tb, int p, T vlos, T w, F &&emit)
{
    using P = GP<M>;
    const int base = G.obs_off + p;
    if (P::v2(G)) emit(base + G.k_v2 * G.n_ap, w * vlos * vlos, kClassVel);
    const int nmax = P::max_gh(G);
    if (nmax >= 0) {
        const T is = tb.isp[G.ap_off + p];
        const T nu = (vlos - tb.vp[G.ap_off + p]) * is;
        const T half = T(0.5) * w * vlos * is * kexp_mhalf(tb, nu * nu);
        T hm1 = T(0), h = T(1);  // H_(n-1), H_n at n = 0
#pragma unroll
        for (int n = 0; n <= 6; ++n) {
            if (n <= nmax) {
                if (P::gh(G, n)) emit(base + G.k_gh[n] * G.n_ap, T(gh_c(n)) * half * fma(T(2 * n), hm1, -(nu * h)),
                                      kClassDv);
                const T hn1 = fma(T(2) * nu, h, -(T(2 * n) * hm1));
                hm1 = h;
                h = hn1;
            }
        }
    }
}

// ---------------------------------------------------------------- priors

// v_c^2 = R |a(R)| and the potential at radius R on the x axis (R >= 0), for the
// spherical potentials without the square root of R^2 and with one logarithm for the
// NFW halo (shared by its potential and its enclosed mass); the flattened log halo
// through accel and potential.
template <class T, bool SCF = true>
__host__ __device__ __forceinline__ void circ_terms(const Model &m, const Cst<T> &k, T R, T &vc2, T &phi,
                                                    FnTables fn = FnTables{nullptr, nullptr})
{
    if constexpr (sizeof(T) == 8) {
        if (m.pot < 2 && fn.ln && m.int_force && big_range(R)) {
            const Big r = big_of(R);
            Big v;
            phi = -big_double(well_big(m, k, r, big_rcp(r), fn.ln, &v));
            vc2 = big_double(v);
            return;
        }
    }
    if (m.pot >= 2) {
        T ax, ay, az;
        accel<T, SCF>(m, k, R, T(0), T(0), ax, ay, az);
        vc2 = -R * ax;
        phi = potential<T, SCF>(m, k, R, T(0), T(0));
        return;
    }
    const T ra = R + k.a;
    vc2 = d_div(k.GM * R, ra * ra);
    phi = -d_div(k.GM, ra);
    if (m.pot == 1) {
        if (R > T(0)) {
            const T q = d_div(R, k.rs);
            T l1, mu;
            if constexpr (sizeof(T) == 4) {
                nfw_logs(q, l1, mu);
            } else {
                // mu(q) = ln(1+q) - q/(1+q); its series where the two terms cancel
                l1 = d_log1p(q);
                mu = q < T(1e-3) ? nfw_mu(q) : l1 - d_div(q, T(1) + q);
            }
            vc2 += d_div(k.GMs * mu, R);
            phi -= d_div(k.GMs * l1, R);
        } else {
            phi += k.hn_phi0;
        }
    }
}

// Energy of the circular orbit of radius R in the equatorial plane: phi(R) + v_c^2/2.
template <class T, bool SCF = true>
__host__ __device__ __forceinline__ T circ_energy(const Model &m, const Cst<T> &k, T R,
                                                  FnTables fn = FnTables{nullptr, nullptr})
{
    T vc2, phi;
    circ_terms<T, SCF>(m, k, R, vc2, phi, fn);
    return phi + T(0.5) * vc2;
}

// Square root, quotient (b > 0), exponential and logarithm of the prior binning: FP64 on the
// integer pipe where fn has the tables.
__device__ __forceinline__ float p_sqrt(float x, FnTables) { return d_sqrt(x); }
__device__ __forceinline__ double p_sqrt(double x, FnTables fn) { return fn.et ? sqrt_int(x) : sqrt(x); }
__device__ __forceinline__ float p_div(float a, float b, FnTables) { return d_div(a, b); }
__device__ __forceinline__ double p_div(double a, double b, FnTables fn) { return fn.et ? div_int(a, b) : a / b; }
__device__ __forceinline__ float p_exp(float x, FnTables) { return d_exp(x); }
__device__ __forceinline__ double p_exp(double x, FnTables fn) { return fn.et ? exp_int(x, fn.et) : exp(x); }
__device__ __forceinline__ float p_log(float x, FnTables) { return d_log(x); }
__device__ __forceinline__ double p_log(double x, FnTables fn) { return fn.ln ? log_int(x, fn.ln) : log(x); }

// The E_c table in the state type: FP64, or its FP32 copy (a conversion of each of the twenty
// values a search reads would go through the FP64 pipe).
template <class T>
using LcTable = T;
template <class T>
__device__ __forceinline__ const T *lc_table(const Buffers &b);
template <>
__device__ __forceinline__ const double *lc_table<double>(const Buffers &b) { return b.lcE; }
template <>
__device__ __forceinline__ const float *lc_table<float>(const Buffers &b) { return b.lcEf; }

// Lc(E): closed form for the Hernquist potential (E_c = -(u+1)/(2u^2) GM/a with
// u = R/a + 1), otherwise the host table of E_c(ln R) bracketed by binary search,
// interpolated, and refined by secant steps on E_c(R) = E.
template <class T, bool SCF = true>
__device__ T circular_L(const Model &m, const Cst<T> &k, const LcTable<T> *lcE, T E, FnTables fn)
{
    if (m.pot < 2 && !(E < T(0))) return T(0);
    if (m.lc_closed) {
        const T e = E * k.e_scale;
        if (!(e > T(-1))) return T(0);
        const T u = p_div(T(1) + p_sqrt(T(1) - T(8) * e, fn), T(-4) * e, fn);
        const T R = k.a * (u - T(1));
        const T ra = R + k.a;
        return p_div(R * p_sqrt(k.GM * R, fn), ra, fn);
    }
    if (!(E > k.phi_min)) return T(0);
    const int n = m.lc_n;
    int lo = 0, hi = n - 1;
    T R;
    if (SCF && m.pot == 3) {
        // The self-consistent potential need not be lowest at the centre (its l > 0 terms can
        // lower it off the axis), and its thin shells put kinks in E_c(R) at the grid radii,
        // so E_c(R) = E may have no root below phi(0) and is not smooth: Lc(E) by plain
        // bisection, from [0, 1] doubled until it brackets the root (no circular orbit
        // below E_c(0) = phi(0)).
        T v = T(0);
        if (!(E > scf_circ(m, k, T(0), v))) return T(0);
        T hi = T(1), lo = T(0);
        while (hi < T(1e15) && scf_circ(m, k, hi, v) <= E) hi *= T(2);
        for (int it = 0; it < 400; ++it) {
            const T mid = T(0.5) * (lo + hi);
            if (!(mid > lo) || !(mid < hi)) break;
            if (scf_circ(m, k, mid, v) <= E) lo = mid;
            else hi = mid;
        }
        R = T(0.5) * (lo + hi);
        scf_circ(m, k, R, v);
        return R * d_sqrt(v);
    }
    if (!(E > T(__ldg(lcE)))) {
        R = k.lc_r0;
    } else if (!(E < T(__ldg(lcE + n - 1)))) {
        R = k.lc_rmax;
    } else {
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (T(__ldg(lcE + mid)) <= E) lo = mid;
            else hi = mid;
        }
        if constexpr (sizeof(T) == 4) {
            // FP32: inverse cubic interpolation of ln R in E through the four table
            // points around the bracket (Lagrange), clamped to the bracket. Its error,
            // of order (table step)^4 ~ 4e-9 in ln R, is below FP32 resolution, so no
            // refinement by the force is needed.
            int j0 = lo - 1;
            j0 = j0 < 0 ? 0 : (j0 > n - 4 ? n - 4 : j0);
            T xe[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) xe[q] = T(__ldg(lcE + j0 + q));
            T lnr = T(0);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                T li = T(1);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (q != i) li *= d_div(E - xe[q], xe[i] - xe[q]);
                lnr += li * (k.lc_lnr0 + T(j0 + i) * k.lc_dlnr);
            }
            const T ylo = k.lc_lnr0 + T(lo) * k.lc_dlnr;
            R = d_exp(fminf(fmaxf(lnr, ylo), ylo + k.lc_dlnr));
        } else {
            const T e0 = T(__ldg(lcE + lo)), e1 = T(__ldg(lcE + hi));
            const T fr = p_div(E - e0, e1 - e0, fn);
            R = p_exp(k.lc_lnr0 + (T(lo) + fr) * k.lc_dlnr, fn);
            // secant refinement, starting from the table segment's slope
            const T Ra = p_exp(k.lc_lnr0 + T(lo) * k.lc_dlnr, fn);
            const T Rb = p_exp(k.lc_lnr0 + T(hi) * k.lc_dlnr, fn);
            T r0 = R, f0 = circ_energy<T, SCF>(m, k, r0, fn) - E;
            T r1 = r0 - f0 * p_div(Rb - Ra, e1 - e0, fn);
            for (int it = 0; it < 3; ++it) {
                const T f1 = circ_energy<T, SCF>(m, k, r1, fn) - E;
                if (f1 == f0) break;
                const T r2 = r1 - f1 * d_div(r1 - r0, f1 - f0);
                r0 = r1;
                f0 = f1;
                r1 = r2;
            }
            R = r1;
        }
    }
    T vc2, phi;
    circ_terms<T, SCF>(m, k, R, vc2, phi, fn);
    return R * p_sqrt(vc2, fn);
}

// Cell k*nx + l of a particle: E bin from the chosen spacing (clamped), circularity
// bin from x = L/Lc(E) (x = Lz/Lc(E) on [-1, 1] for the signed variant, clamped).
template <class T, bool SCF = true>
__device__ __forceinline__ int prior_cell(const Model &m, const Cst<T> &k, const LcTable<T> *lcE, T x, T y, T z,
                                          T vx, T vy, T vz, FnTables fn)
{
    const T E = fma(T(0.5), fma(vx, vx, fma(vy, vy, vz * vz)), potential<T, SCF>(m, k, x, y, z, fn));
    const T Lz = fma(x, vy, -(y * vx));
    T L;
    if (m.signed_lz) {
        L = Lz;
    } else {
        const T Lx = fma(y, vz, -(z * vy)), Ly = fma(z, vx, -(x * vz));
        L = p_sqrt(fma(Lx, Lx, fma(Ly, Ly, Lz * Lz)), fn);
    }
    const T Lc = circular_L<T, SCF>(m, k, lcE, E, fn);
    T xc = (Lc > T(0)) ? p_div(L, Lc, fn) : T(0);
    const T xmin = m.signed_lz ? T(-1) : T(0);
    xc = xc < xmin ? xmin : (xc > T(1) ? T(1) : xc);
    T f;
    if (m.e_spacing == 0) f = (E >= T(0)) ? T(1) : p_div(p_log(-E, fn) - k.s_lo, k.s_den, fn);
    else if (m.e_spacing == 1) f = p_div(p_exp(E, fn) - k.s_lo, k.s_den, fn);
    else f = p_div(E - k.s_lo, k.s_den, fn);
    const T fk = d_floor(f * k.nE);
    const int kb = !(fk >= T(0)) ? 0 : (fk >= k.nE ? m.nE - 1 : int(fk));
    const T fl = d_floor(p_div(xc - xmin, T(1) - xmin, fn) * k.nx);
    const int lb = !(fl >= T(0)) ? 0 : (fl >= k.nx ? m.nx - 1 : int(fl));
    return kb * m.nx + lb;
}

// ---------------------------------------------------------------- fixed point
//
// Global sums are int64 words: FP64 mode uses two per slot (integer part and the
// next 32 fraction bits of v*scale), mixed mode one (round(v*scale)). Integer
// sums are exact, so the result does not depend on the order of the additions.

// FP64: v*scale = hi + lo 2^-32 with hi = floor and lo in [0, 2^32), computed with
// integer operations on the IEEE fields (scale is a power of two): the 53-bit
// significand m and exponent give T = round(v*scale*2^32) = m 2^k, split into its
// high and low 32-bit parts. |v*scale| < 2^62 keeps k <= 42, so m 2^(k-32) < 2^63.
__device__ __forceinline__ void fx2(double v, double scale, long long &hi, long long &lo)
{
    const long long bits = bits_of(v);
    const int e = int((bits >> 52) & 0x7FF);
    if (e == 0) {  // zero (and subnormals, below any resolution used here)
        hi = 0;
        lo = 0;
        return;
    }
    const int se = int((bits_of(scale) >> 52) & 0x7FF) - 1023;
    const unsigned long long m = (static_cast<unsigned long long>(bits) & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int k = e - 1075 + se + 32;
    unsigned long long th, tl;
    if (k >= 32) {
        th = m << (k - 32);
        tl = 0;
    } else if (k >= 0) {
        th = m >> (32 - k);
        tl = (m << k) & 0xFFFFFFFFull;
    } else if (k > -63) {
        const unsigned long long r = (m + (1ull << (-k - 1))) >> (-k);
        th = r >> 32;
        tl = r & 0xFFFFFFFFull;
    } else {
        th = 0;
        tl = 0;
    }
    if (bits < 0) {
        hi = tl ? -static_cast<long long>(th) - 1 : -static_cast<long long>(th);
        lo = tl ? 4294967296ll - static_cast<long long>(tl) : 0;
    } else {
        hi = static_cast<long long>(th);
        lo = static_cast<long long>(tl);
    }
}

// Block-shared sums. Shared memory adds 32-bit integers natively, 64-bit ones only by a loop
// around a compare-and-swap that runs once per lane of a warp that meets on a slot, so a sum is
// kept in three 32-bit words.
// FP64 mode: the words of a 96-bit integer, modulo 2^96. The low word is added first, the old
// value it returns gives the carry, and so on up; the top word is added only where it and the
// carry are not zero together (for small values of either sign: -x has it all ones and the carry
// makes it 0), so a deposit is two shared atomics. (The 64-bit loops took a third of a small
// fit's step: 20,000 particles 22.9 -> 20.5 us a step.)
// Mixed mode: the fields of one 64-bit integer L = hi 2^32 + mid 2^16 + lo, mid, lo in [0, 2^16)
// and hi signed, added without carries (three atomics that return nothing; two words with a
// carry are 4 % slower at 2M particles, the returned value being waited for). At most
// kMaxParticlesPerBlock particles per block keep the sums of mid and lo below 2^31, and |sum of
// hi| < 2^31 follows from the fixed-point range.
constexpr long long kMaxParticlesPerBlock = 32768;

// Adds v and the carry c to *w; returns the carry out.
__device__ __forceinline__ unsigned add_word(unsigned *w, unsigned v, unsigned c)
{
    const unsigned a = v + c;
    const unsigned old = atomicAdd(w, a);
    return (old + a < a || a < c) ? 1u : 0u;
}

template <class T>
struct Acc;

template <>
struct Acc<double> {
    static __host__ __device__ size_t bytes(const Model &m) { return sizeof(int) * (3 * size_t(m.nslots) + size_t(m.ncell)); }
    // the fixed-point value of v * scale: hi + lo 2^-32
    struct Fx {
        long long hi, lo;
    };
    __device__ static Fx fx(double v, double scale)
    {
        Fx r;
        fx2(v, scale, r.hi, r.lo);
        return r;
    }
    __device__ static void put(void *base, int slot, const Fx &q)
    {
        unsigned *h = static_cast<unsigned *>(base) + 3 * slot;
        unsigned c = add_word(h, unsigned(q.lo), 0u);
        c = add_word(h + 1, unsigned(q.hi), c);
        const unsigned top = unsigned(static_cast<unsigned long long>(q.hi) >> 32) + c;
        if (top) atomicAdd(h + 2, top);
    }
    __device__ static void add(void *base, int slot, double v, double scale)
    {
        if (is_zero(v)) return;
        put(base, slot, fx(v, scale));
    }
    // word wd (0: integer part, 1: fraction) of a slot of the block's sums
    __device__ static long long word(const void *base, int slot, int wd)
    {
        const unsigned *h = static_cast<const unsigned *>(base) + 3 * slot;
        if (wd == 1) return static_cast<long long>(h[0]);
        return static_cast<long long>((static_cast<unsigned long long>(h[2]) << 32) | h[1]);
    }
};

template <>
struct Acc<float> {
    static __host__ __device__ size_t bytes(const Model &m) { return sizeof(int) * (3 * size_t(m.nslots) + size_t(m.ncell)); }
    // the fixed-point value of v * scale: one 64-bit integer, rounded to nearest
    struct Fx {
        long long L;
    };
    __device__ static Fx fx(float v, float scale) { return Fx{__float2ll_rn(v * scale)}; }
    __device__ static void put(void *base, int slot, const Fx &q)
    {
        int *h = static_cast<int *>(base) + 3 * slot;
        // the hi limb is added even when 0: cheaper than the branch around it
        atomicAdd(h, static_cast<int>(q.L >> 32));
        atomicAdd(h + 1, static_cast<int>((q.L >> 16) & 0xFFFF));
        atomicAdd(h + 2, static_cast<int>(q.L & 0xFFFF));
    }
    // a zero adds zeros: cheaper than the branch around it
    __device__ static void add(void *base, int slot, float v, float scale) { put(base, slot, fx(v, scale)); }
    __device__ static long long word(const void *base, int slot, int)
    {
        const int *q = static_cast<const int *>(base) + 3 * slot;
        return q[0] * 4294967296ll + q[1] * 65536ll + q[2];
    }
};

// Sums of the global-deposit kernel's shared slots (n of them), where space decides how much
// of a map has block-shared sums: FP64 as above, mixed two 32-bit words modulo 2^64 with a carry,
// those of one significance together (two thirds of the space of the three limbs, and one or
// two atomics each deposit).
template <class T>
struct WinAcc : Acc<T> {
    static constexpr int kWords = 3;
    __device__ static void add(void *base, int, int slot, T v, T scale) { Acc<T>::add(base, slot, v, scale); }
    __device__ static long long word(const void *base, int, int slot, int wd) { return Acc<T>::word(base, slot, wd); }
};
template <>
struct WinAcc<float> : Acc<float> {
    static constexpr int kWords = 2;
    __device__ static void add(void *base, int n, int slot, float v, float scale)
    {
        const long long L = fx(v, scale).L;
        unsigned *h = static_cast<unsigned *>(base) + slot;
        const unsigned c = add_word(h, unsigned(L), 0u);
        const unsigned top = unsigned(static_cast<unsigned long long>(L) >> 32) + c;
        if (top) atomicAdd(h + n, top);
    }
    __device__ static long long word(const void *base, int n, int slot, int)
    {
        const unsigned *h = static_cast<const unsigned *>(base) + slot;
        return static_cast<long long>((static_cast<unsigned long long>(h[n]) << 32) | h[0]);
    }
};

// Particle counts of the cells, behind the sums.
__host__ __device__ inline int cell_slots(const Model &m) { return m.cells_smem ? m.ncell : 0; }
__host__ __device__ inline int ga_slots(const Model &m)
{
    return cell_slots(m) + (m.win_n > 0 ? m.g[m.win_group].n_kinds * m.win_n : 0);
}
template <class T, bool GA = false>
__device__ __forceinline__ unsigned *acc_counts(void *base, const Model &m)
{
    return static_cast<unsigned *>(base) + (GA ? WinAcc<T>::kWords * ga_slots(m) : 3 * m.nslots);
}

// Per-thread running total of the deposited weight, in the same fixed point.
template <class T>
struct Total;

template <>
struct Total<double> {
    long long hi = 0, lo = 0;
    // The range check: the sum of hi 2^-20, with 2^43 (the whole range) for each weight whose own
    // words are out of it. At most kMaxParticlesPerBlock weights meet in a block's sum of it:
    // it cannot wrap.
    long long top = 0;
    __device__ void add(double v, double scale)
    {
        long long a, b;
        fx2(v, scale, a, b);
        hi += a;
        lo += b;
    }
    __device__ void add_fx(const Acc<double>::Fx &q, double w, double scale)
    {
        hi += q.hi;
        lo += q.lo;
        // w scale >= 2^62 on the exponents (infinity and NaN too): fx2 has dropped its high bits
        const int e = int(bits_of(w) >> 52 & 0x7ff) + int(bits_of(scale) >> 52 & 0x7ff) - 2 * 1023;
        top += e < 62 ? q.hi >> 20 : 1ll << 43;
    }
    // the deposited weight for the range check, in units of 2^20 (an FP64 sum would take the FP64 pipe)
    __device__ long long range_sum(double) const { return top; }
    __device__ static double range_value(long long v, double scale) { return double(v) * (1048576.0 * (1.0 / scale)); }
    __device__ long long word(int q, double) const { return q == 0 ? hi : lo; }
};

// Mixed mode: round(w * scale) of every weight summed in a 64-bit register, so the total
// is the exact integer sum and does not depend on how the particles are spread over
// threads and blocks.
template <>
struct Total<float> {
    long long s = 0;
    __device__ void add(float v, float scale) { s += __float2ll_rn(v * scale); }
    __device__ void add_fx(const Acc<float>::Fx &q, float, float) { s += q.L; }  // the range check: wdep
    __device__ float range_sum(float wdep) const { return wdep; }
    __device__ static double range_value(float v, float) { return double(v); }
    __device__ long long word(int, float) const { return s; }
};

// hi + lo 2^-32 in FP64, with the whole part of the fraction word carried first: how a sum is split
// over its two words depends on the blocks that added it, and beyond 2^53 the rounding of hi would too.
__device__ __forceinline__ double fx_join(long long hi, long long lo)
{
    return double(hi + (lo >> 32)) + double(lo & 0xffffffffll) * (1.0 / 4294967296.0);
}
template <int WPS>
__device__ __forceinline__ double fx_read(const long long *h, int slot)
{
    if (WPS == 1) return double(__ldcg(h + slot));
    return fx_join(__ldcg(h + 2 * slot), __ldcg(h + 2 * slot + 1));
}

// ---------------------------------------------------------------- force of change

// The data term sum_j K_j c_j at the particle's position, with the apertures from
// the cached code of the last deposit when there is one.
template <unsigned... Ms, class T>
__device__ __forceinline__ T foc_data(const Model &m, const Cst<T> &k, const Tables<T> &tb, const T *rec,
                                      unsigned code, const T *gexp, T x, T y, T z, T vy, T vz)
{
    T Y, vlos;
    project(k, y, z, vy, vz, Y, vlos);
    if (code != kApUncached) return data_term_cached<Ms...>(m, tb, rec, code, vlos, gexp);
    return data_term<Ms...>(m, tb, rec, x, y, z, x, Y, vlos);
}

// Weight after the force of change of eq. modFOC over one step, the kernel
// values taken at the particle's current position and the priors held fixed:
// F = mu dS/dw - sum_j K_j c_j, c_j = Delta_j/sigma_j (times 1/area for mass),
// dS/dw = -ln(w/what) (eq. S+) or -ln(w/what) - 1 (eq. entropy).
template <unsigned... Ms, class T>
__device__ __forceinline__ T foc_update(const Model &m, const Cst<T> &k, const Tables<T> &tb, const T *rec,
                                        unsigned code, const T *gexp, T iprior, T w, T x, T y, T z, T vy, T vz,
                                        unsigned &err)
{
    if (w == T(0)) return w;  // w = 0 is a fixed point
    const T data = foc_data<Ms...>(m, k, tb, rec, code, gexp, x, y, z, vy, vz);
    // A cell mean below the resolution of the fixed-point cell sums reads as 0
    // (iprior = 0); the particle's weight is then unresolved too and the entropy
    // term is dropped.
    T dS = iprior > T(0) ? -d_log(w * iprior) : T(0);
    if (m.mode == 0) dS -= T(1);
    const T h = k.dteps * fma(k.mu, dS, -data);
    T wn;
    if (m.update_rule == 0) wn = w * d_exp(h);
    else wn = w * (T(1) + h);
    if (!d_finite(wn)) err |= kErrNonFinite;
    else if (wn < T(0) || (m.update_rule == 1 && !(wn > T(0)))) err |= kErrNegWeight;
    return wn;
}

// The same update on u = ln w (FP64 mode): u + eps dt F for the exponential rule,
// u + ln(1 + eps dt F) for explicit Euler, with dS/dw = ln(what) - u.
template <unsigned... Ms, class T>
__device__ __forceinline__ T foc_update_log(const Model &m, const Cst<T> &k, const Tables<T> &tb, const T *rec,
                                            unsigned code, const T *gexp, T lprior, T u, T x, T y, T z, T vy, T vz,
                                            unsigned &err)
{
    if (is_neg_inf(u)) return u;  // w = 0 is a fixed point
    const T data = foc_data<Ms...>(m, k, tb, rec, code, gexp, x, y, z, vy, vz);
    // a prior that reads 0 (below the resolution of the cell sums) drops the entropy term
    T dS = !is_neg_inf(lprior) ? lprior - u : T(0);
    if (m.mode == 0) dS -= T(1);
    const T h = k.dteps * fma(k.mu, dS, -data);
    T un;
    if (m.update_rule == 0) {
        un = u + h;
    } else {
        if (!(h > T(-1))) {
            err |= (h != h) ? kErrNonFinite : kErrNegWeight;
            return u;
        }
        un = u + log1p(h);
    }
    // exp_int overflows above 709 (NaN of either sign is flagged too)
    const long long ub = bits_of(un);
    if ((ub & 0x7fffffffffffffffll) > 0x7ff0000000000000ll || ub > 0x4086280000000000ll) err |= kErrNonFinite;
    return un;
}

// ---------------------------------------------------------------- shared-memory layout

// The step's tables in the state type T, as one block of global memory per fit that a block
// of the step kernel copies into shared memory as it is, in 16-byte pieces: the force-of-
// change records, V_p and 1/sigma_p, 1/prior (ln prior in FP64 mode), the squared edges, the
// annulus lookup and in FP64 mode the tables of the exponential and the logarithm (read from
// global memory where they are what no longer fits, Model::tab_smem). The finalize writes the records and priors in
// place; the rest is laid out at creation. (Converting every table from FP64 in every block took
// 15,000 cycles of a step with 2,700 priors, and 5,800 with 300.) The global-deposit kernel and the
// weight read-out take the part from the priors on. Offsets in bytes.
struct TabLayout {
    int rec, vp, isp, prior, esq, lut, et, ln, bytes;
};

template <class T>
__host__ __device__ inline TabLayout tab_layout(const Model &m)
{
    auto up = [](size_t b) { return int((b + 15) / 16 * 16); };
    TabLayout t;
    t.rec = 0;
    t.vp = up(sizeof(T) * size_t(m.n_ap_total) * m.rec_len);
    t.isp = t.vp + up(sizeof(T) * size_t(m.n_ap_total));
    t.prior = t.isp + up(sizeof(T) * size_t(m.n_ap_total));
    t.esq = t.prior + up(sizeof(T) * size_t(m.ncell));
    t.lut = t.esq + up(sizeof(T) * size_t(m.n_edges_total));
    t.et = t.lut + up(sizeof(unsigned short) * size_t(m.n_lut));
    t.ln = t.et + (sizeof(T) == 8 ? kExpEntries * int(sizeof(u64)) : 0);
    t.bytes = t.ln + (sizeof(T) == 8 && m.pot < 2 ? 2 * kLnEntries * int(sizeof(u64)) : 0);
    return t;
}

template <class T>
struct Smem {
    void *h;               // fixed-point sums of the block (layout of Acc<T>)
    T *c, *iprior, *esq, *vp, *isp;  // c: the force-of-change records; iprior: 1/prior, or ln prior (FP64)
    unsigned short *lut;
    const u64 *et, *ln;    // tables of exp_int and ln_frac
    unsigned char *tab;    // start of the copied tables, and the range of them that is copied
    int tab_lo, tab_hi;
};

// Block sums of the global-deposit kernel, laid out as Acc<T> slots: the cells of the prior
// grid with their counts behind the slots (where they fit, Model::cells_smem), and the aperture
// window, one slot per kind and window aperture. (With the cells in global memory a prior update of
// 8M particles on 800 cells took 2.3 ms, ten times the other steps.)
template <class T>
__host__ __device__ inline size_t window_bytes(const Model &m)
{
    return (size_t(ga_slots(m)) * WinAcc<T>::kWords + cell_slots(m)) * sizeof(int);
}

// hist: 0 no block sums, 1 all (Acc<T>), 2 the aperture window of the global deposit
template <class T>
__host__ __device__ inline size_t acc_bytes_padded(const Model &m, int hist = 1)
{
    const size_t b = hist == 2 ? window_bytes<T>(m) : Acc<T>::bytes(m);
    return (b + 15) / 16 * 16;
}

// Dynamic shared memory of a kernel holding the block sums (with_hist) and all tables
// (with_rec) or those from the priors on; the global-deposit step kernel keeps its records,
// V_p and 1/sigma_p in global memory.
template <class T>
__host__ __device__ inline size_t smem_bytes(const Model &m, int with_hist, int with_rec = 1)
{
    const TabLayout t = tab_layout<T>(m);
    return (with_hist ? acc_bytes_padded<T>(m, with_hist) : 0) + size_t((m.tab_smem ? t.bytes : t.et) - (with_rec ? 0 : t.prior));
}

template <class T>
__device__ __forceinline__ Smem<T> carve(const Model &m, const Buffers &b, unsigned char *base, int with_hist,
                                         int with_rec = 1)
{
    const TabLayout t = tab_layout<T>(m);
    Smem<T> s;
    s.h = base;
    s.tab = base + (with_hist ? acc_bytes_padded<T>(m, with_hist) : 0);
    s.tab_lo = with_rec ? 0 : t.prior;
    s.tab_hi = m.tab_smem ? t.bytes : t.et;
    unsigned char *z = s.tab - s.tab_lo;
    s.c = reinterpret_cast<T *>(z + t.rec);
    s.vp = reinterpret_cast<T *>(z + t.vp);
    s.isp = reinterpret_cast<T *>(z + t.isp);
    s.iprior = reinterpret_cast<T *>(z + t.prior);
    s.esq = reinterpret_cast<T *>(z + t.esq);
    s.lut = reinterpret_cast<unsigned short *>(z + t.lut);
    s.et = reinterpret_cast<const u64 *>((m.tab_smem ? z : b.tab) + t.et);
    s.ln = reinterpret_cast<const u64 *>((m.tab_smem ? z : b.tab) + t.ln);
    return s;
}

// Starts the copy of bytes [lo, hi) (multiples of 16) of a fit's tables into shared memory
// (asynchronous 16-byte copies; the caller waits with tables_wait and then synchronises the block).
template <class T>
__device__ __forceinline__ void tables_range(const Buffers &b, const Smem<T> &s, int lo, int hi)
{
    const unsigned dst = static_cast<unsigned>(__cvta_generic_to_shared(s.tab)) + unsigned(lo - s.tab_lo);
    const unsigned char *src = b.tab + lo;
    for (int q = 16 * int(threadIdx.x); q < hi - lo; q += 16 * int(blockDim.x))
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + q), "l"(src + q) : "memory");
}
template <class T>
__device__ __forceinline__ void tables_start(const Buffers &b, const Smem<T> &s)
{
    tables_range<T>(b, s, s.tab_lo, s.tab_hi);
}
__device__ __forceinline__ void tables_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ---------------------------------------------------------------- force-of-change records

// A record folds the coefficients c_j of its aperture (see data_term): with v_los = V + s nu
// (s = sigma_p), mass contributes c to q0, v_los^2 contributes c (V^2, 2 V s, s^2) and v_los
// contributes c (V, s) to (q0, q1, q2); b_n contributes c c_n H_n(nu) to the Hermite part, with
// the monomial coefficients of H_n from the recurrence H_{n+1} = 2 nu H_n - 2 n H_{n-1}. Shell
// records hold c_j of each a_lm. The factors are laid out once per fit (FinPlan).
// Coefficient of nu^q in the physicists' H_n, set on the host from the recurrence
// H_{n+1} = 2 nu H_n - 2 n H_{n-1} (see herm_table).
inline void herm_table(double h[7][7])
{
    for (int n = 0; n < 7; ++n)
        for (int q = 0; q < 7; ++q) h[n][q] = 0.0;
    h[0][0] = 1.0;
    h[1][1] = 2.0;
    for (int n = 1; n < 6; ++n)
        for (int q = 0; q < 7; ++q) h[n + 1][q] = (q > 0 ? 2.0 * h[n][q - 1] : 0.0) - 2.0 * n * h[n - 1][q];
}

// Sets this translation unit's constant table (kExp2j) on the current device.
static inline cudaError_t upload_constants()
{
    double t[32];
    exp2_table(t);
    const cudaError_t e = cudaMemcpyToSymbol(kExp2j, t, sizeof t);
    return e == cudaSuccess ? cudaStreamSynchronize(cudaStreamLegacy) : e;  // for kernels on any stream
}

// ---------------------------------------------------------------- finalize
//
// Run once every block has added its sums, by the last block of the step kernel, by k_finalize or
// between the steps of k_steps: converts the fixed-point sums, renormalises, smooths (eq. myts), forms
// Delta_j, chi^2 (eqs. delta, chi) and the force-of-change coefficients, the prior means on
// update steps, and clears the sums for the next step.

// The sum of v over the block, for any block size (a multiple of 32), to every thread: warp
// shuffles, then the warps' sums from shared memory in warp order (the same order in every
// kernel that ends with the finalize). red: 32 doubles.
__device__ __forceinline__ double fold_block(double v, double *red)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    for (int q = 0; q < int(blockDim.x >> 5); ++q) s += red[q];
    return s;
}

// The self-consistent potential at an update (Sec. 6), in the finalize: the mass-to-light
// ratio follows the chi^2 gradient, d ln Upsilon/dt = -eps_ups sum_j Delta_j/sigma_j D_j over
// the update_every steps to the next update (not at the load); then the interval tables
// TA, TB of scf_field from the new coefficients a_lm,k and Upsilon. red: 32 doubles.
template <int WPS>
__device__ void scf_finalize(const Model &m, const Buffers &b, double s_ren, int init, double *red)
{
    Scalars &sc = *b.sc;
    if (!init && m.n_dups > 0) {
        double part = 0.0;
        for (int j = threadIdx.x; j < m.J; j += blockDim.x) {
            const int kind = b.obs_kind[j];
            const double sj = kind == kKindV2 ? m.fx_v2 : ((kind >= kKindGH0 && kind <= kKindGH0 + 6) ? m.fx_dv : 0.0);
            if (sj == 0.0) continue;
            const double D = fx_read<WPS>(b.hist, m.off_dups + j) / sj * s_ren;
            part += b.delta[j] / b.sig[j] * D;
        }
        const double sum = fold_block(part, red);
        if (threadIdx.x == 0) sc.ups *= exp(-m.eps_ups * double(m.update_every) * m.dt * sum);
        __syncthreads();
    }
    const double ups = sc.ups;
    const int n = m.scf_n, nlm = m.scf_nlm;
    for (int idx = threadIdx.x; idx < nlm; idx += blockDim.x) {
        int l = 0;
        while ((l + 1) * (l + 1) <= idx) ++l;
        const double C = -4.0 * 3.14159265358979323846 * m.G * ups / double(2 * l + 1);
        double A = 0.0;  // sum over the shells inside
        for (int j = 0; j <= n; ++j) {
            m.scf_tab[(size_t(j) * nlm + idx) * 2] = C * A;
            if (j < n) {
                const double a = fx_read<WPS>(b.hist, m.off_scf + j * nlm + idx) / m.fx_gh * s_ren;
                m.scf_coef[size_t(j) * nlm + idx] = a;
                A += a * pow(m.scf_r[j], l);
            }
        }
        double B = 0.0;  // sum over the shells outside
        for (int j = n; j >= 0; --j) {
            if (j < n) {
                const double a = fx_read<WPS>(b.hist, m.off_scf + j * nlm + idx) / m.fx_gh * s_ren;
                B += a * pow(m.scf_r[j], -(l + 1));
            }
            m.scf_tab[(size_t(j) * nlm + idx) * 2 + 1] = C * B;
        }
        for (int j = 0; j <= n; ++j) {
            const size_t q = (size_t(j) * nlm + idx) * 2;
            m.scf_tabf[q] = float(m.scf_tab[q]);
            m.scf_tabf[q + 1] = float(m.scf_tab[q + 1]);
        }
    }
    __syncthreads();
    // the x axis (see scf_circ): R_lm(R, 0, 0) = N_lm T_lm(0, R^2) R^m = c_lm R^l for m >= 0, 0 for m < 0
    const int L = m.scf_lmax;
    double *axis = m.scf_tab + size_t(n + 1) * nlm * 2;
    for (int q = threadIdx.x; q < (n + 1) * (L + 1); q += blockDim.x) {
        const int j = q / (L + 1), l = q % (L + 1);
        double A = 0.0, B = 0.0, dfac = 1.0;
        for (int mm = 0; mm <= l; ++mm) {
            double t0 = 0.0, t1 = dfac;  // T_(q-1), T_q at z = 0, r^2 = 1, from q = mm
            for (int i = mm + 1; i <= l; ++i) {
                const double t2 = -double(i + mm - 1) * t0 / double(i - mm);
                t0 = t1;
                t1 = t2;
            }
            const int idx = l * (l + 1) + mm;
            const double *tab = m.scf_tab + (size_t(j) * nlm + idx) * 2;
            A += tab[0] * m.scf_norm[idx] * t1;
            B += tab[1] * m.scf_norm[idx] * t1;
            dfac *= double(2 * mm + 1);
        }
        axis[2 * q] = A;
        axis[2 * q + 1] = B;
    }
    __syncthreads();
}

// Priors of the grid-less variant (Sec. 7): the mean weight of the particles in the window of
// cells |k' - k| <= pwin_E, |l' - l| <= pwin_x around each cell (k, l), cut at the grid's
// edges. The window sums come from cumulative sums of the cells' integer words, first along
// x (into pwin), then, after the row windows are written back over the cell words, along E,
// so they equal the sums of the particles' own words in any order. q = 0 is the particle
// count, q = 1..WPS the words of the weight sum; all unsigned, wrapping like the deposits.
__device__ __forceinline__ void write_prior(const Buffers &b, int c, double pr)
{
    const double ip = pr > 0.0 ? 1.0 / pr : 0.0;
    b.prior[c] = pr;
    b.iprior[c] = ip;
    if (b.ipriorf) b.ipriorf[c] = float(ip);
    b.lprior[c] = pr > 0.0 ? log(pr) : -HUGE_VAL;
}

template <int WPS>
__device__ void window_priors(const Model &m, const Buffers &b, long long *hist, double s_ren)
{
    constexpr int NQ = WPS + 1;
    const int nE = m.nE, nx = m.nx, nc = m.ncell, hE = m.pwin_E, hx = m.pwin_x;
    unsigned long long *H = reinterpret_cast<unsigned long long *>(hist);
    unsigned long long *cum = b.pwin;
    auto at = [&](int q, int c) -> unsigned long long * {
        return q == 0 ? H + m.off_count + c : H + WPS * (m.J + 1 + c) + (q - 1);
    };
    for (int r = threadIdx.x; r < nE * NQ; r += blockDim.x) {  // cumulative sums along x
        const int k = r / NQ, q = r % NQ;
        unsigned long long acc = 0;
        for (int l = 0; l < nx; ++l) {
            const unsigned long long v = __ldcg(at(q, k * nx + l));
            if (q == 0) b.prior_count[k * nx + l] = (long long)v;
            acc += v;
            cum[size_t(q) * nc + k * nx + l] = acc;
        }
    }
    __syncthreads();
    for (int r = threadIdx.x; r < nc * NQ; r += blockDim.x) {  // row windows over the cell words
        const int q = r / nc, c = r % nc, k = c / nx, l = c % nx;
        const unsigned long long *row = cum + size_t(q) * nc + k * nx;
        *at(q, c) = __ldcg(row + min(l + hx, nx - 1)) - (l - hx - 1 >= 0 ? __ldcg(row + l - hx - 1) : 0ull);
    }
    __syncthreads();
    for (int r = threadIdx.x; r < nx * NQ; r += blockDim.x) {  // cumulative sums along E
        const int l = r / NQ, q = r % NQ;
        unsigned long long acc = 0;
        for (int k = 0; k < nE; ++k) {
            acc += __ldcg(at(q, k * nx + l));
            cum[size_t(q) * nc + k * nx + l] = acc;
        }
    }
    __syncthreads();
    for (int c = threadIdx.x; c < nc; c += blockDim.x) {
        const int k = c / nx, l = c % nx, hi = min(k + hE, nE - 1), lo = k - hE - 1;
        unsigned long long box[NQ];
        for (int q = 0; q < NQ; ++q) {
            const unsigned long long *col = cum + size_t(q) * nc + l;
            box[q] = __ldcg(col + size_t(hi) * nx) - (lo >= 0 ? __ldcg(col + size_t(lo) * nx) : 0ull);
        }
        const long long cnt = (long long)box[0];
        double sum = WPS == 2 ? fx_join((long long)box[1], (long long)box[WPS]) : double((long long)box[1]);
        sum = sum / m.fx_w * s_ren;
        const double pr = cnt > 0 ? sum / double(cnt) : 0.0;
        write_prior(b, c, pr);
    }
}

// The head of step t + 1, from the scalars after step t (one thread).
__device__ __forceinline__ StepHead next_head(const Model &m, long long t, int pending, double s_ren, double what,
                                              int fresh = 1)
{
    StepHead h;
    const bool update = (t % m.update_every) == 0;  // step t + 1 is one of 1, 1 + P, ...
    h.pending = pending;
    h.prior_step = m.mode == 1 && update;
    h.scf_step = m.pot == 3 && update;
    h.wscale = float(s_ren);
    h.iwhat = what > 0.0 ? float(1.0 / what) : 0.f;
    h.fresh = fresh;
    h.lwscale = log(s_ren);
    h.lwhat = what > 0.0 ? log(what) : -HUGE_VAL;
    return h;
}

// The head from the scalars of a restored state.
static __global__ void k_head(const Model m, const Scalars *sc, StepHead *head)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    StepHead h = next_head(m, sc->t, sc->pending, sc->wscale, sc->what_flat);
    h.lwscale = sc->lwscale;
    h.lwhat = sc->lwhat_flat;
    *head = h;
}

// The total weight of a step (stored units) from its fixed-point sum.
template <int WPS>
__device__ __forceinline__ double total_weight(const Model &m, const long long *hist)
{
    return fx_read<WPS>(hist, m.J) * (1.0 / m.fx_w);  // fx_w is a power of two: exact
}

// The scale W0/U that renormalises the weights of this step, in integers: every thread forms it,
// and as FP64 instructions its division would queue for the narrow pipe.
template <int WPS>
__device__ __forceinline__ double renorm_scale(const Model &m, const long long *hist, int init, double W0)
{
    const long long hi = __ldcg(hist + WPS * m.J), lo = WPS == 2 ? __ldcg(hist + WPS * m.J + 1) : 0;
    if (init || !m.renormalize) return 1.0;
    const long long t = hi + (lo >> 32);
    if (t > 0 && big_range(W0) && big_range(m.fx_w)) {
        const int z = __clzll(t);
        const u64 f = u64(lo) << 32;  // the fraction below t
        const Big U{(u64(t) << z) | (z ? f >> (64 - z) : 0), 63 - z - big_of(m.fx_w).e};
        return big_double(big_norm(big_mul_raw(big_rcp(U), big_of(W0))));
    }
    const double U = total_weight<WPS>(m, hist);
    return U > 0.0 ? W0 / U : 1.0;
}

// The observables of chunks [ch0, ch1) from the fixed-point sums: smoothing (eq. myts),
// Delta_j (eq. delta), coefficients c_j into b.c and cs (if given, J doubles of shared memory);
// csum[chunk]: the chunk's sum of Delta_j^2. A warp per chunk. What does not depend on the
// sums is loaded before them. ys: the block's own copy of ytil in shared memory, or null
// (Buffers::ytil); store: whether this block writes the fit's arrays.
template <int WPS>
__device__ __forceinline__ void fin_observables(const Model &m, const Buffers &b, const long long *hist, int ch0, int ch1,
                                                int init, double W0, double *cs, double *csum, double &s_ren,
                                                double *ys = nullptr, bool store = true)
{
    const FinPlan &pl = b.plan;
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    ObsRow r;
    double h = 0.0, old = 0.0;
    auto fetch = [&](int ch) {
        r = pl.rows[32 * ch + lane];
        if (r.j >= 0) {
            h = fx_read<WPS>(hist, r.j);
            old = ys ? ys[r.j] : b.ytil[r.j];
        }
    };
    int ch = ch0 + int(threadIdx.x >> 5);
    if (ch < ch1) fetch(ch);
    s_ren = renorm_scale<WPS>(m, hist, init, W0);
    for (; ch < ch1; ch += nw) {
        double d = 0.0;
        if (r.j >= 0) {
            const double raw = h * r.iscale * s_ren * r.post;
            const double yt = init ? raw : old + m.alpha * (raw - old);
            const double a = yt - r.Y;  // a / sig: the product with 1/sig and its exact residual
            const double q = a * r.isig;
            d = fma(fma(-q, r.sig, a), r.isig, q);
            const double cj = d * r.cw;
            if (ys) ys[r.j] = yt;
            if (cs) cs[r.j] = cj;
            if (store) {
                b.yraw[r.j] = raw;
                b.ytil[r.j] = yt;
                b.delta[r.j] = d;
                b.c[r.j] = cj;
            }
        }
        double d2 = d * d;
        if (ch + nw < ch1) fetch(ch + nw);
        for (int o = 16; o > 0; o >>= 1) d2 += __shfl_xor_sync(0xffffffffu, d2, o);
        if (lane == 0) csum[ch] = d2;
    }
}

// The record elements [e0, e1) from the coefficients c; rs: also into the block's records in
// shared memory, if given.
template <class T = double>
__device__ __forceinline__ void fin_records(const Buffers &b, int e0, int e1, const double *c, T *rs = nullptr,
                                            bool store = true)
{
    const FinPlan &pl = b.plan;
    for (int e = e0 + int(threadIdx.x); e < e1; e += blockDim.x) {
        const RecElem el = pl.elems[e];
        double v = 0.0;
        for (int k = 0; k < el.nk; ++k) v += pl.coef[size_t(k) * pl.n_elems + e] * c[el.j0 + k * el.stride];
        if (rs) rs[el.dst] = T(v);
        if (store) {
            b.rec[el.dst] = v;
            if (b.recf) b.recf[el.dst] = float(v);
        }
    }
}

// chi^2 from the chunk sums, in chunk order over 32 lanes (one warp). L2: the sums are in
// global memory, from several blocks.
template <bool L2>
__device__ __forceinline__ double fin_chi2(const double *csum, int n)
{
    double v = 0.0;
    for (int q = int(threadIdx.x & 31); q < n; q += 32) v += L2 ? __ldcg(csum + q) : csum[q];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The scalars after the step and the head of the next one (one thread).
__device__ __forceinline__ void fin_scalars(const Model &m, const Buffers &b, long long n, int init, int prior_step,
                                            int scf_step, double s_ren, double U)
{
    Scalars &sc = *b.sc;
    const long long t = init ? 0 : __ldcg(&sc.t) + 1;
    const double what = init ? (n > 0 ? U / double(n) : 0.0) : __ldcg(&sc.what_flat);
    // the integer sums wrap beyond their range: the floating-point check sum catches it
    if (!(__ldcg(&sc.Wcheck) <= 0.5 * __ldcg(&sc.Wrange))) atomicOr(&sc.err, kErrOverflow);
    const StepHead h = next_head(m, t, init ? 0 : (t > m.n_relax ? 1 : 0), s_ren, what, scf_step);
    if (init) {
        sc.W0 = U;
        sc.what_flat = what;
        sc.lwhat_flat = h.lwhat;
    }
    sc.Wcheck = 0.0;
    sc.Wsum = U;
    if (!init) sc.t = t;
    sc.wscale = s_ren;
    sc.lwscale = h.lwscale;
    sc.pending = h.pending;
    sc.blocks_done = 0;
    if (prior_step && m.smooth) sc.smooth_pending = 1;
    *b.head = h;
}

// Update steps: the cell means (Sec. 2.3.1) or window means from the cells' sums, by block
// `blk` of `blks` (the windows by the first).
template <int WPS>
__device__ __forceinline__ void fin_priors(const Model &m, const Buffers &b, long long *hist, double s_ren, int blk = 0,
                                           int blks = 1)
{
    if (m.pwin_E > 0 || m.pwin_x > 0) {
        if (blk == 0) window_priors<WPS>(m, b, hist, s_ren);
        return;
    }
    const double ifx = 1.0 / m.fx_w;
    for (int q = blk * blockDim.x + threadIdx.x; q < m.ncell; q += blks * blockDim.x) {
        const long long cnt = __ldcg(hist + m.off_count + q);
        const double sum = fx_read<WPS>(hist, m.J + 1 + q) * ifx * s_ren;
        const double pr = cnt > 0 ? sum / double(cnt) : 0.0;  // mean weight of the cell
        b.prior_count[q] = cnt;
        if (m.smooth) b.prior_raw[q] = pr;  // the smoothing kernels turn the raw means into the priors
        else write_prior(b, q, pr);
    }
}

// The finalize in one block (the last of a block-shared step). The GPU waits for it, so what
// counts is its chain of dependent latencies and the instructions it fetches cold: a warp per
// chunk of observables, one thread per record element with the factors laid out beforehand, no
// unrolled code, the scalars of the next step (two logarithms, a modulo) beside the records.
// Measured on the 60-observable fit: 32,000 cycles with one thread per aperture and the scalars
// before the barrier, 12,000 so.
// cs: the start of the shared memory, J coefficients and one double per chunk.
template <int WPS>
__device__ void finalize_block(const Model &m, const Buffers &b, long long n, int init, int prior_step,
                               double *cs, int scf_step = 0)
{
    const FinPlan &pl = b.plan;
    const double W0 = init ? 0.0 : __ldcg(&b.sc->W0);
    double *csum = cs + m.J;
    double s_ren;
    fin_observables<WPS>(m, b, b.hist, 0, pl.n_chunks, init, W0, cs, csum, s_ren);
    __syncthreads();
    if (int(threadIdx.x) == int(blockDim.x) - 32)
        fin_scalars(m, b, n, init, prior_step, scf_step, s_ren, total_weight<WPS>(m, b.hist));
    if (threadIdx.x < 32) {
        const double chi2 = fin_chi2<false>(csum, pl.n_chunks);
        if (threadIdx.x == 0) b.sc->chi2 = chi2;
    }
    fin_records(b, 0, pl.n_elems, cs);
    if (scf_step) {
        __syncthreads();
        scf_finalize<WPS>(m, b, s_ren, init, cs);
    }
    if (prior_step) fin_priors<WPS>(m, b, b.hist, s_ren);
    __syncthreads();
    const int words = (prior_step || scf_step) ? m.hist_words : m.off_grid;
    for (int q = threadIdx.x; q < words; q += blockDim.x) b.hist[q] = 0;
}

// ---------------------------------------------------------------- step kernel
//
// One M2M step over all particles, one read and one write of the particle state:
// (a) the previous step's force of change at the current position, (b) the
// kick-drift-kick push, (c) the deposit of w K_j into block-shared fixed-point
// sums, (d) on prior-update steps the (E, x) cell of every particle with per-cell
// weight sums and counts. Blocks add their sums to the global sums with integer
// atomics (exact, so order-independent); the last block to finish runs the
// finalize (or k_finalize follows). Nothing waits on another block here; k_steps, which runs
// many steps per launch with the same functions, meets once or twice per step.
//
// GA (global deposit): for observable sets whose block sums or force-of-change
// records do not fit in shared memory (e.g. 64 x 64 pixel maps of five moments),
// every deposit goes straight to the global int64 sums with 64-bit atomics and the
// records are read from global memory (L1/L2 resident). The sums are the same
// integers in either mode, so both give bit-identical results.
template <class T>
__device__ __forceinline__ const T *global_records(const Buffers &b);
template <>
__device__ __forceinline__ const double *global_records<double>(const Buffers &b) { return b.rec; }
template <>
__device__ __forceinline__ const float *global_records<float>(const Buffers &b) { return b.recf; }

// V_p and 1/sigma_p per aperture in global memory (the global-deposit kernel keeps its
// shared memory for the aperture window)
template <class T>
__device__ __forceinline__ const T *global_vp(const Buffers &b);
template <>
__device__ __forceinline__ const double *global_vp<double>(const Buffers &b) { return b.Vp; }
template <>
__device__ __forceinline__ const float *global_vp<float>(const Buffers &b) { return b.Vpf; }
template <class T>
__device__ __forceinline__ const T *global_isp(const Buffers &b);
template <>
__device__ __forceinline__ const double *global_isp<double>(const Buffers &b) { return b.isp; }
template <>
__device__ __forceinline__ const float *global_isp<float>(const Buffers &b) { return b.ispf; }

// One deposit into the global sums (global-deposit mode): the fixed-point words of
// the block-shared path, added directly.
// Adds v to a 64-bit integer sum in global memory, without reading the result back.
__device__ __forceinline__ void red_add(long long *p, long long v)
{
    asm volatile("red.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ void global_add(long long *hist, int slot, double v, double scale)
{
    if (is_zero(v)) return;
    long long hi, lo;
    fx2(v, scale, hi, lo);
    red_add(hist + 2 * slot, hi);
    if (lo) red_add(hist + 2 * slot + 1, lo);
}
__device__ __forceinline__ void global_add(long long *hist, int slot, float v, float scale)
{
    if (v == 0.f) return;
    red_add(hist + slot, __float2ll_rn(v * scale));
}

// Per-step flags of one fit, read from its scalars at the start of the step.
template <class T>
struct StepFlags {
    int pending, prior_step, scf_step, fresh;
    T wscale, lwscale, iwhat_flat;
};

template <class T>
__device__ __forceinline__ StepFlags<T> step_flags(const Model &m, const StepHead *head, int init)
{
    StepFlags<T> f;
    const StepHead h = *head;
    f.pending = init ? 0 : h.pending;
    f.prior_step = init ? 0 : h.prior_step;
    // the self-consistent potential is rebuilt at the load and on the prior schedule
    f.scf_step = init ? m.pot == 3 : h.scf_step;
    f.fresh = h.fresh;
    if constexpr (kLogWeights<T>) {
        f.wscale = T(1);
        f.lwscale = init ? T(0) : T(h.lwscale);
        f.iwhat_flat = T(h.lwhat);
    } else {
        f.wscale = init ? T(1) : T(h.wscale);
        f.lwscale = T(0);
        f.iwhat_flat = T(h.iwhat);
    }
    return f;
}

// Zeroes the block sums (block-shared deposit only).
template <class T, bool GA>
__device__ __forceinline__ void block_zero(const Model &m, const Smem<T> &S)
{
    int4 *z = static_cast<int4 *>(S.h);
    const int nw = int(acc_bytes_padded<T>(m, GA ? 2 : 1) / sizeof(int4));
    for (int q = threadIdx.x; q < nw; q += blockDim.x) z[q] = int4{0, 0, 0, 0};
}

// The per-particle part of one step for particles i0, i0 + stride, ... below i1:
// the pending force of change, the push, the deposit, the prior binning, and the
// write-back of the state.
//
// LATE: the next particle's loads are issued after the force of change instead of before it. Their
// ten values are then not alive across the force of change, where the mixed batched kernel (64
// registers) otherwise spills two or three into local memory and misses the L1 with them (long-scoreboard
// stalls 0.5 -> 2.5 per instruction), and the loads of the mixed global-deposit kernel do not queue before
// its records (3.1 -> 2.1). us per step, before and after: 96 Hernquist + NFW fits of 52M particles
// 934 -> 816, Hernquist 873 -> 794, log halo 873 -> 793; maps of 4M 84 -> 78. The other kernels lose by it
// and load early: FP64 1M 119.2 -> 121.5, the mixed one of five blocks an SM 45.9 -> 46.4 at 2M, many
// mixed steps per launch up to 2 %.
template <class T, bool GA, bool LATE, unsigned M0, unsigned M1, unsigned M2, unsigned M3>
__device__ __forceinline__ void step_particles(const Model &m, const Model &mh, const Cst<T> &k, const State<T> &P,
                                               const Buffers &b,
                                               const Smem<T> &S, const StepFlags<T> &f, int push, long long i0,
                                               long long i1, long long stride, unsigned &err, Total<T> &wtot, T &wdep)
{
    // The block's tables are on their way into shared memory and its sums are being zeroed:
    // the first particles are loaded before the block waits for both.
    // mh: the fields of the per-particle path (observable layout, regularisation and update
    // modes, potential kind). It is the fit's own Model, or in the batched kernel one Model
    // in the parameter space that every fit of the batch equals in those fields. m: the
    // fit's own Model, for the prior binning and the self-consistent potential.
    // the self-consistent potential runs in the generic kernel only (the host picks it)
    constexpr bool kScf = M0 == kDyn;
    const Tables<T> tb{S.esq, S.lut, GA ? global_vp<T>(b) : S.vp, GA ? global_isp<T>(b) : S.isp, S.et, S.ln};
    const T *rec = GA ? global_records<T>(b) : S.c;
    auto deposit = [&](int slot, T v, T scale) {
        if constexpr (GA) global_add(b.hist, slot, v, scale);
        else Acc<T>::add(S.h, slot, v, scale);
    };
    // the next particle's state is loaded while the current one is processed
    const bool need_cell = f.pending && mh.mode == 1;
    const bool cache = mh.ap_cache != 0;
    const bool need_ap = cache && f.pending;
    const bool gxc = sizeof(T) == 8 && P.gx != nullptr;  // FP64, aperture cache, a Gauss-Hermite group
    const bool need_fa = keeps_accel<T>(mh) && push;
    T nx = T(0), ny = T(0), nz = T(0), nvx = T(0), nvy = T(0), nvz = T(0), nw = T(0), ngx = T(0), nfa = T(0);
    int ncell = 0;
    unsigned nap = kApUncached;
    auto fetch = [&](long long j) {
        nx = P.x[j]; ny = P.y[j]; nz = P.z[j];
        nvx = P.vx[j]; nvy = P.vy[j]; nvz = P.vz[j];
        nw = P.w[j];
        if (need_fa) nfa = P.fa[j];
        if (need_cell) ncell = P.cell[j];
        if (need_ap) nap = P.ap[j];
        if (need_ap && gxc) ngx = P.gx[j];
    };
    if (i0 < i1) fetch(i0);
    tables_wait();
    __syncthreads();
    for (long long i = i0; i < i1; i += stride) {
        T x = nx, y = ny, z = nz;
        T vx = nvx, vy = nvy, vz = nvz;
        const T wst = nw;
        const int cell = ncell;
        const unsigned code = nap;
        const T gin = ngx;
        const T fa_in = nfa;
        const T *gp = gxc ? &gin : static_cast<const T *>(nullptr);
        if (!LATE && i + stride < i1) fetch(i + stride);
        T w, u;
        if constexpr (kLogWeights<T>) {
            u = wst + f.lwscale;
            if (f.pending) {
                const T lp = mh.mode == 1 ? S.iprior[cell] : f.iwhat_flat;
                u = foc_update_log<M0, M1, M2, M3>(mh, k, tb, rec, code, gp, lp, u, x, y, z, vy, vz, err);
            }
            w = kexp(tb, u);
        } else {
            w = wst * f.wscale;
            if (f.pending) {
                const T pr = mh.mode == 1 ? S.iprior[cell] : f.iwhat_flat;
                w = foc_update<M0, M1, M2, M3>(mh, k, tb, rec, code, gp, pr, w, x, y, z, vy, vz, err);
            }
            u = w;
        }
        if (LATE && i + stride < i1) fetch(i + stride);
        if (keeps_accel<T>(mh)) {
            T fa;
            if (push) {
                fa = fa_in;
                leapfrog_from(mh, k, x, y, z, vx, vy, vz, fa, tb.ln);
            } else {
                fa = accel_factor(mh, k, x, y, z, tb.ln);
            }
            P.fa[i] = fa;
        } else if (kScf && mh.pot == 3) {
            if (push) {
                T ax, ay, az;
                if (f.fresh) {
                    accel<T, kScf>(mh, k, x, y, z, ax, ay, az);
                } else {
                    ax = P.ax[i];
                    ay = P.ay[i];
                    az = P.az[i];
                }
                leapfrog_scf(mh, k, x, y, z, vx, vy, vz, ax, ay, az);
                P.ax[i] = ax;
                P.ay[i] = ay;
                P.az[i] = az;
            }
        } else {
            if (push) leapfrog<T>(mh, k, x, y, z, vx, vy, vz);
        }
        if (!is_zero(w)) {
            T Y, vlos;
            project(k, y, z, vy, vz, Y, vlos);
            // the fixed-point weight, shared by the total and the surface-mass deposits
            const auto wfx = Acc<T>::fx(w, k.fx_w);
            unsigned code_out = 0;
            T gout = T(0);
            each_group<0, M0, M1, M2, M3>(mh, [&](auto Pl, int g) {
                constexpr unsigned M = decltype(Pl)::mask;
                const GroupDesc &G = mh.g[g];
                if (GP<M>::shells(G)) {  // never cached; never in the global-deposit kernel
                    shell_kernels(mh, g, tb, x, y, z, w, [&](int j, T v, int, int) {
                        if constexpr (GA) global_add(b.hist, j, v, k.fx_gh);
                        else Acc<T>::add(S.h, j, v, k.fx_gh);
                    });
                    return;
                }
                const int p = aperture<M>(G, tb.esq, tb.lut, x, Y);
                if (cache) code_out = ap_encode(mh, code_out, g, p);
                if (p >= 0) {
                    // the v^2 sums' range assumes v^2 <= v2max (energy bound with headroom)
                    const T vv = product(vlos, vlos);
                    if (GP<M>::v2(G) && gt_nonneg(vv, k.v2max)) err |= kErrOverflow;
                    group_kernels<M>(
                        G, tb, p, vlos, vv, w,
                        [&](int j, T v, int cls, int kk) {
                            const T scale = cls == kClassMass ? k.fx_w : (cls == kClassVel ? k.fx_v2 : k.fx_gh);
                            if constexpr (GA) {
                                const unsigned a = unsigned(p - mh.win_lo);
                                if (g == mh.win_group && a < unsigned(mh.win_n))
                                    WinAcc<T>::add(S.h, ga_slots(mh), cell_slots(mh) + kk * mh.win_n + int(a), v, scale);
                                else
                                    global_add(b.hist, j, v, scale);
                            } else if (cls == kClassMass) {  // v is w (the kernel is 1)
                                Acc<T>::put(S.h, j, wfx);
                            } else {
                                Acc<T>::add(S.h, j, v, scale);
                            }
                        },
                        gxc && g == mh.gx_group ? &gout : nullptr);
                    if constexpr (kScf) {
                        if (f.scf_step && m.n_dups > 0)  // derivatives for the mass-to-light ratio (Sec. 6)
                            group_dkernels<M>(G, tb, p, vlos, w, [&](int j, T v, int cls) {
                                deposit(m.off_dups + j, v, cls == kClassVel ? k.fx_v2 : k.fx_dv);
                            });
                    }
                }
            });
            if constexpr (kScf) {
                if (f.scf_step)  // the particle's luminosity in the expansion of the stellar potential
                    scf_deposit(m, x, y, z, w, [&](int slot, T v) { deposit(slot, v, k.fx_gh); });
            }
            if (cache) P.ap[i] = static_cast<uint16_t>(code_out);
            if (gxc) P.gx[i] = gout;
            wtot.add_fx(wfx, w, k.fx_w);
            if constexpr (sizeof(T) == 4) wdep += w;
        }
        if (f.prior_step) {
            const int c = prior_cell<T, kScf>(m, k, lc_table<T>(b), x, y, z, vx, vy, vz, FnTables{tb.et, m.pot < 2 ? tb.ln : nullptr});
            if (GA && m.cells_smem) WinAcc<T>::add(S.h, ga_slots(m), c, w, k.fx_w);
            else deposit(m.J + 1 + c, w, k.fx_w);
            if (GA && !m.cells_smem) red_add(b.hist + m.off_count + c, 1);
            else atomicAdd(acc_counts<T, GA>(S.h, m) + c, 1u);
            P.cell[i] = static_cast<uint16_t>(c);
        }
        P.x[i] = x; P.y[i] = y; P.z[i] = z;
        P.vx[i] = vx; P.vy[i] = vy; P.vz[i] = vz;
        P.w[i] = u;
    }
}

// Adds the block's sums, its total weight and its error bits to the fit's global
// sums and scalars. Called by every thread of the block.
template <class T, int WPS, bool GA>
__device__ __forceinline__ void block_flush(const Model &m, const Cst<T> &k, Scalars *sc, long long *hist, double *wcheck,
                                            const Smem<T> &S, int prior_step, unsigned err, const Total<T> &wtot, T wdep,
                                            int scf_step)
{
    if (err) atomicOr(&sc->err, err);
    // the total weight went into registers: one global atomic per warp and word
#pragma unroll
    for (int q = 0; q < WPS; ++q) {
        long long v = wtot.word(q, k.fx_w);
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0 && v != 0)
            red_add(hist + WPS * m.J + q, v);
    }
    auto chk = wtot.range_sum(wdep);
    for (int o = 16; o > 0; o >>= 1) chk += __shfl_xor_sync(0xffffffffu, chk, o);
    if ((threadIdx.x & 31) == 0 && chk != 0)
        atomicAdd(wcheck, Total<T>::range_value(chk, k.fx_w));
    __syncthreads();
    if (GA) {  // the aperture window's sums go to their observables' global words
        const GroupDesc &G = m.g[m.win_group < 0 ? 0 : m.win_group];
        const int slots = m.win_n > 0 ? G.n_kinds * m.win_n : 0;
        for (int q = threadIdx.x; q < WPS * slots; q += blockDim.x) {
            const int slot = q / WPS, wd = q - slot * WPS;
            const int kk = slot / m.win_n, a = slot - kk * m.win_n;
            const long long v = WinAcc<T>::word(S.h, ga_slots(m), cell_slots(m) + slot, wd);
            const int j = G.obs_off + kk * G.n_ap + m.win_lo + a;
            if (v != 0) red_add(hist + WPS * j + wd, v);
        }
    }
    const bool all = prior_step || scf_step;
    const int words = GA ? 0 : WPS * (all ? m.nslots : m.J);
    for (int q = threadIdx.x; q < words; q += blockDim.x) {
        const int slot = q / WPS;
        if (slot == m.J) continue;  // the total is already global
        const long long v = Acc<T>::word(S.h, slot, q - slot * WPS);
        if (v != 0) red_add(hist + q, v);
    }
    if (GA && all)
        for (int q = threadIdx.x; q < WPS * cell_slots(m); q += blockDim.x) {
            const int slot = q / WPS;
            const long long v = WinAcc<T>::word(S.h, ga_slots(m), slot, q - slot * WPS);
            if (v != 0) red_add(hist + WPS * (m.J + 1) + q, v);
        }
    if ((!GA || m.cells_smem) && all) {
        const unsigned *cnt = acc_counts<T, GA>(S.h, m);
        for (int q = threadIdx.x; q < m.ncell; q += blockDim.x)
            if (cnt[q]) red_add(hist + m.off_count + q, static_cast<long long>(cnt[q]));
    }
    __syncthreads();
}

// Whether this block is the last of `blocks` to arrive at the counter, to every thread. The
// block's reductions come before the counter for every reader: the barrier orders them before
// thread 0, whose fence orders them before its atomic (one fence, not one per thread).
__device__ __forceinline__ bool block_is_last(unsigned *counter, unsigned blocks, bool *flag)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        *flag = atomicAdd(counter, 1u) == blocks - 1;
        __threadfence();
    }
    __syncthreads();
    return *flag;
}

// Threads per block the step kernel is compiled for. The mixed-precision global-deposit
// kernel runs up to 1024 threads in one block per SM, so that one aperture window takes
// the whole shared memory of the SM (DRAM and L2 see the deposits once per block).
template <class T, bool GA>
constexpr int kStepMaxThreads = (GA && sizeof(T) == 4) ? 1024 : 256;

template <class T, int WPS, int MINB, bool GA, unsigned M0, unsigned M1, unsigned M2, unsigned M3>
__global__ void __launch_bounds__(kStepMaxThreads<T, GA>, (GA && sizeof(T) == 4) ? 1 : MINB) k_step(const Model m, const Cst<T> k, const State<T> P,
                                                    const Buffers b, int push, int init)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const Smem<T> S = carve<T>(m, b, smem, GA ? 2 : 1, GA ? 0 : 1);
    __shared__ bool am_last;

    tables_start<T>(b, S);
    const StepFlags<T> f = step_flags<T>(m, b.head, init);
    block_zero<T, GA>(m, S);

    // The particles in whole warps of 32, cut into one contiguous run per block: a small fit
    // then spreads over all SMs instead of filling the first ones.
    const long long units = (P.n + 31) >> 5;
    const long long lo = (units * blockIdx.x / gridDim.x) << 5;
    long long hi = (units * (blockIdx.x + 1) / gridDim.x) << 5;
    if (hi > P.n) hi = P.n;
    unsigned err = 0;
    Total<T> wtot;
    T wdep = T(0);  // floating-point twin of wtot, for the fixed-point range check
    step_particles<T, GA, GA && sizeof(T) == 4, M0, M1, M2, M3>(m, m, k, P, b, S, f, push, lo + threadIdx.x, hi, blockDim.x, err, wtot, wdep);
    block_flush<T, WPS, GA>(m, k, b.sc, b.hist, &b.sc->Wcheck, S, f.prior_step, err, wtot, wdep, f.scf_step);
    if (GA || m.fin_wide || m.shard) return;  // k_finalize follows (a shard's after the exchange of its sums)
    // last block to finish runs the finalize
    if (block_is_last(&b.sc->blocks_done, gridDim.x, &am_last))
        finalize_block<WPS>(m, b, P.n, init, f.prior_step, reinterpret_cast<double *>(smem), f.scf_step);
}

// ---------------------------------------------------------------- shards of one fit
//
// A fit whose particles are split over several processes (contiguous ranges, one per
// shard) runs the per-particle pass of a step on every shard (k_step with Model::shard),
// then the caller adds the shards' integer sums word by word (an all-reduce), and every
// shard runs the same finalize on the same integers (k_finalize): the result is
// bit-identical to the unsplit fit. The exchanged words are the fixed-point sums of
// Model::hist_words, then one range word (the deposited weight in units of
// Wrange 2^-40, for the overflow check) and two words of the total weight that a
// weight read-out renormalises with.
constexpr double kRangeUnit = 1.0 / 1099511627776.0;  // 2^-40

// After a shard's pass: its floating-point deposited weight into the range word.
static __global__ void k_shard_pack(long long *hist, int hist_words, Scalars *sc)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        // up to 2^12 times the range (infinity and NaN too): the words of all shards add up
        hist[hist_words] = llrint(fmin(ceil(sc->Wcheck / (sc->Wrange * kRangeUnit)), 4503599627370496.0));
        sc->Wcheck = 0.0;
    }
}

// The finalize as a kernel of its own, one block per range of 32 apertures: after a global-
// deposit step or one of more than 16 chunks of observables (one block took 430,000 cycles for
// 64 x 64 pixels of five moments, 207 of 604 us; the step takes 360 us with the ranges spread), and for a shard, from the
// exchanged (summed) words. Every block handles its observables and records; the last one to
// arrive adds chi^2, the priors and the scalars. A shard's range word replaces Wcheck first.
template <class T, int WPS>
__global__ void __launch_bounds__(256) k_finalize(const Model m, const Buffers b, long long n, int init)
{
    __shared__ bool am_last;
    __shared__ double red[32];
    const FinPlan &pl = b.plan;
    const StepFlags<T> f = step_flags<T>(m, b.head, init);
    const double W0 = init ? 0.0 : __ldcg(&b.sc->W0);
    const int2 r0 = pl.range[blockIdx.x], r1 = pl.range[blockIdx.x + 1];
    double s_ren;
    fin_observables<WPS>(m, b, b.hist, r0.x, r1.x, init, W0, nullptr, pl.csum, s_ren);
    __syncthreads();
    fin_records(b, r0.y, r1.y, b.c);
    if (!block_is_last(&b.sc->blocks_done, gridDim.x, &am_last)) return;
    if (threadIdx.x < 32) {
        const double chi2 = fin_chi2<true>(pl.csum, pl.n_chunks);
        if (threadIdx.x == 0) {
            b.sc->chi2 = chi2;
            if (m.shard) {
                b.sc->Wcheck = double(b.hist[m.hist_words]) * (b.sc->Wrange * kRangeUnit);
                b.hist[m.hist_words] = 0;
            }
            fin_scalars(m, b, n, init, f.prior_step, f.scf_step, s_ren, total_weight<WPS>(m, b.hist));
        }
    }
    if (f.scf_step) {
        __syncthreads();
        scf_finalize<WPS>(m, b, s_ren, init, red);
    }
    if (f.prior_step) fin_priors<WPS>(m, b, b.hist, s_ren);
    __syncthreads();
    const int words = (f.prior_step || f.scf_step) ? m.hist_words : m.off_grid;
    for (int q = threadIdx.x; q < words; q += blockDim.x) b.hist[q] = 0;
}

// ---------------------------------------------------------------- batched step kernel
//
// Many independent fits (their own potential, targets, priors and particle counts)
// advanced by one launch. The host cuts the fits' particles, taken in model order,
// into equal contiguous shares, one per block, and each share into segments
// (model, begin, end) of at most kMaxParticlesPerBlock particles. A block walks its
// segments: on a new model it loads the model's descriptors and tables into shared
// memory, it runs the per-particle step over the segment, and it flushes its sums
// into the model's global sums. The block that flushes a model's last segment runs
// that model's finalize. The sums are exact integers, so a fit advanced in a batch
// gives bit-identical results to the same fit advanced alone.
struct Segment {
    int model;
    int pad;
    long long begin, end;
};

template <class T>
struct BatchArgs {
    const Model *models;
    const Cst<T> *csts;
    const State<T> *states;
    const Buffers *bufs;
    const Segment *seg;
    const int *seg_off;      // block b walks seg[seg_off[b] .. seg_off[b+1])
    const unsigned *nseg;    // per model: its number of segments
};

// the batched kernel copies Model and Cst<T> into shared memory in 8-byte words
static_assert(sizeof(Model) % 8 == 0 && sizeof(Cst<float>) % 8 == 0 && sizeof(Cst<double>) % 8 == 0,
              "descriptor copies need whole 8-byte words");

// The per-fit constants of a batch in the kernel's parameter space (the constant bank): the
// per-particle loop reads them there, where no store can alias them, instead of from copies
// in shared memory that every shared-memory atomic of the deposit could have changed.
// shape: a Model that every fit of the batch equals in the fields of the per-particle path
// (see step_particles); cst[i]: the constants of fit i. With more fits than the bank holds,
// or fits that differ in those fields, the kernel runs from the shared-memory copies.
template <class T>
constexpr int kBankFits = sizeof(T) == 8 ? 112 : 224;

template <class T>
struct BatchBank {
    Model shape;
    Cst<T> cst[kBankFits<T>];
};
static_assert(sizeof(BatchBank<float>) + sizeof(BatchArgs<float>) <= 32764 &&
                  sizeof(BatchBank<double>) + sizeof(BatchArgs<double>) <= 32764,
              "kernel parameters are limited to 32764 bytes");

template <class T, int WPS, int MINB, bool BANK, unsigned M0, unsigned M1, unsigned M2, unsigned M3>
__global__ void __launch_bounds__(256, MINB) k_step_batch(const BatchArgs<T> a, const __grid_constant__ BatchBank<T> bank)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ __align__(16) unsigned long long mbuf[(sizeof(Model) + 7) / 8];
    __shared__ __align__(16) unsigned long long kbuf[(sizeof(Cst<T>) + 7) / 8];
    __shared__ Buffers sb;
    __shared__ State<T> sP;
    __shared__ bool am_last;
    const Model &m = *reinterpret_cast<const Model *>(mbuf);
    const Cst<T> &k = *reinterpret_cast<const Cst<T> *>(kbuf);

    int cur = -1;
    const int s1 = a.seg_off[blockIdx.x + 1];
    for (int s = a.seg_off[blockIdx.x]; s < s1; ++s) {
        const Segment sg = a.seg[s];
        const bool fresh = sg.model != cur;
        if (fresh) {
            __syncthreads();
            const unsigned long long *src = reinterpret_cast<const unsigned long long *>(a.models + sg.model);
            for (int q = threadIdx.x; q < int(sizeof(mbuf) / 8); q += blockDim.x) mbuf[q] = src[q];
            const unsigned long long *ks = reinterpret_cast<const unsigned long long *>(a.csts + sg.model);
            for (int q = threadIdx.x; q < int(sizeof(kbuf) / 8); q += blockDim.x) kbuf[q] = ks[q];
            if (threadIdx.x == 0) {
                sb = a.bufs[sg.model];
                sP = a.states[sg.model];
            }
            __syncthreads();
            cur = sg.model;
        }
        const Buffers &b = sb;
        const State<T> P = sP;
        const Smem<T> S = carve<T>(m, b, smem, 1, 1);
        if (fresh) tables_start<T>(b, S);
        const StepFlags<T> f = step_flags<T>(m, b.head, 0);
        block_zero<T, false>(m, S);
        unsigned err = 0;
        Total<T> wtot;
        T wdep = T(0);
        if constexpr (BANK)
            step_particles<T, false, sizeof(T) == 4, M0, M1, M2, M3>(m, bank.shape, bank.cst[sg.model], P, b, S, f, 1,
                                                     sg.begin + threadIdx.x, sg.end, blockDim.x, err, wtot, wdep);
        else
            step_particles<T, false, sizeof(T) == 4, M0, M1, M2, M3>(m, m, k, P, b, S, f, 1, sg.begin + threadIdx.x, sg.end,
                                                     blockDim.x, err, wtot, wdep);
        block_flush<T, WPS, false>(m, k, b.sc, b.hist, &b.sc->Wcheck, S, f.prior_step, err, wtot, wdep, f.scf_step);
        if (block_is_last(&b.sc->blocks_done, a.nseg[cur], &am_last)) {
            finalize_block<WPS>(m, b, P.n, 0, f.prior_step, reinterpret_cast<double *>(smem), f.scf_step);
            cur = -1;  // the finalize used the shared memory: reload before the next segment
        }
    }
}

// ---------------------------------------------------------------- helpers

// Weights as of the end of the last step: the pending force of change applied
// (without renormalisation) into out[], and the total added to acc (two words).
template <class T>
__global__ void k_materialize(const Model m, const Cst<T> k, const State<T> P, const Buffers b, double *out,
                              long long *acc)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const Smem<T> S = carve<T>(m, b, smem, 0, 0);
    tables_start<T>(b, S);
    const Scalars sc = *b.sc;
    tables_wait();
    __syncthreads();
    // the force of change takes V_p and 1/sigma_p from the records
    const Tables<T> tb{S.esq, S.lut, nullptr, nullptr, S.et, S.ln};
    unsigned err = 0;
    Total<double> tot;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < P.n; i += stride) {
        T w;
        if constexpr (kLogWeights<T>) {
            T u = P.w[i] + T(sc.lwscale);
            if (sc.pending) {
                const T lp = (m.mode == 1) ? S.iprior[P.cell[i]] : T(sc.lwhat_flat);
                u = foc_update_log<kDyn, kDyn, kDyn, kDyn>(m, k, tb, global_records<T>(b), kApUncached,
                                                           static_cast<const T *>(nullptr), lp, u, P.x[i], P.y[i],
                                                           P.z[i], P.vy[i], P.vz[i], err);
            }
            w = kexp(tb, u);
        } else {
            w = P.w[i] * T(sc.wscale);
            if (sc.pending) {
                const T pr =
                    (m.mode == 1) ? S.iprior[P.cell[i]] : (sc.what_flat > 0.0 ? T(1.0 / sc.what_flat) : T(0));
                w = foc_update<kDyn, kDyn, kDyn, kDyn>(m, k, tb, global_records<T>(b), kApUncached,
                                                       static_cast<const T *>(nullptr), pr, w, P.x[i], P.y[i], P.z[i],
                                                       P.vy[i], P.vz[i], err);
            }
        }
        if (sc.pending && w != T(0)) tot.add(double(w), m.fx_w);
        out[i] = double(w);
    }
    if (err) atomicOr(&b.sc->err, err);
    for (int q = 0; q < 2; ++q) {
        long long s = tot.word(q, m.fx_w);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((threadIdx.x & 31) == 0 && s != 0)
            atomicAdd(reinterpret_cast<unsigned long long *>(acc + q), static_cast<unsigned long long>(s));
    }
}

static __global__ void k_scale(double *out, long long n, const long long *acc, const Model m, const Scalars *sc)
{
    const double U = (double(acc[0]) + double(acc[1]) * (1.0 / 4294967296.0)) / m.fx_w;
    if (!sc->pending || !m.renormalize || !(U > 0.0)) return;
    const double s = sc->W0 / U;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        out[i] *= s;
}

template <class T>
__global__ void k_convert_in(const double *src, T *dst, long long n)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = T(src[i]);
}

// FP64 mode stores ln w (w = 0 gives -inf; load rejects negative weights first).
static __global__ void k_log_in(const double *src, double *dst, long long n)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = log(src[i]);
}

template <class T>
__global__ void k_convert_out(const T *src, double *dst, long long n)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = double(src[i]);
}

// Largest v^2 a particle can reach in the fixed potential (2 (E - phi_min)), and a
// flag for non-finite input or negative weights.
static __global__ void k_load_stats(const Model m, const Cst<double> k, const double *x, const double *y,
                             const double *z, const double *vx, const double *vy, const double *vz,
                             const double *w, long long n, unsigned long long *v2max_bits, unsigned *bad)
{
    double best = 0.0;
    unsigned flag = 0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double v2 = vx[i] * vx[i] + vy[i] * vy[i] + vz[i] * vz[i];
        // the self-consistent potential bounds only its halo here (its stellar well is added
        // on the host)
        const double pmin = m.pot == 3 ? m.v0 * m.v0 * log(m.r0) : m.phi_min;
        const double e = v2 + 2.0 * (potential<double>(m, k, x[i], y[i], z[i]) - pmin);
        const double val = e > v2 ? e : v2;
        if (!isfinite(val) || !isfinite(x[i] + y[i] + z[i]) || !isfinite(w[i]) || w[i] < 0.0) flag = 1;
        else if (val > best) best = val;
    }
    for (int o = 16; o > 0; o >>= 1) best = fmax(best, __shfl_xor_sync(0xffffffffu, best, o));
    flag = __reduce_or_sync(0xffffffffu, flag);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(v2max_bits, static_cast<unsigned long long>(__double_as_longlong(best)));
        if (flag) atomicOr(bad, 1u);
    }
}

}  // namespace m2m
