// Several steps of a fit in one launch.
//
// A step of a small fit is a chain of latencies: the launch, the tables, one particle per
// thread, the sums, the last block's finalize, all with instructions and data fetched cold. Here
// one cooperative launch runs up to kPersistSteps steps: the blocks keep their tables, records,
// priors and smoothed observables in shared memory, meet once per step after adding their sums
// and then form the residuals and the force-of-change records. Either every block does that for
// itself from the same integers, so that nothing is handed back, or each takes its ranges of
// apertures and all meet again: the first costs FP64 instructions in every block (about 20 per
// chunk of observables, 16 cycles each on an SM's pipe), the second a meeting of about 2,500 cycles
// (the line lies at eight chunk-blocks an SM). Steps that update the priors meet a second time in either
// case. The arithmetic and its order are those of k_step, bit for bit.
//
// Measured against one launch per step: 20,000 FP64 particles 18.9 -> 13.5 us per step (the sizes at
// persist_fits).
//
// Three sets of sums take turns: set s % 3 collects step s, is read after that step's meeting,
// and is cleared after the next one, when every block has read it, two meetings before it collects
// again. Waits are bounded: a block that gives up sets kErrTimeout and returns, and so do all
// others in turn.
#include "m2m_ctx.h"
#include "m2m_meet.cuh"

#include <algorithm>
#include <mutex>

using namespace m2m;

namespace {

constexpr int kPersistSteps = 64;
// Most chunk-blocks an SM (chunks of observables times blocks an SM) with which every block
// finalizes for itself (see `spread`): at most so many chunk sums are then in a block's memory.
constexpr int kOwnChunks = 8;

template <class T, int WPS, int MINB, unsigned M0, unsigned M1, unsigned M2, unsigned M3>
__global__ void __launch_bounds__(256, MINB) k_steps(const Model m, const Cst<T> k, const State<T> P, const Buffers b,
                                                     long long *hist2, Meet *g, int nsteps, int own, int spread)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const Smem<T> S = carve<T>(m, b, smem, 1);
    __shared__ bool ok, last;
    __shared__ double lw;
    const TabLayout tl = tab_layout<T>(m);
    // The coefficients of the finalize take the place of the block's sums (J doubles of the 12 bytes
    // each of J + 1 slots or more). own: offset of the block's smoothed observables and, behind them,
    // its chunk sums: up to J of them with single apertures, they do not fit before the tables, which
    // stay for the steps to come.
    double *cs = reinterpret_cast<double *>(smem);
    double *ys = reinterpret_cast<double *>(smem + own), *csum = ys + m.J;
    const FinPlan &pl = b.plan;

    tables_start<T>(b, S);
    StepFlags<T> f = step_flags<T>(m, b.head, 0);
    const long long t0 = b.sc->t;
    const double W0 = b.sc->W0, what = b.sc->what_flat;
    int phase = int(t0 % m.update_every);  // 0: the next step updates the priors
    for (int j = threadIdx.x; j < m.J; j += blockDim.x) ys[j] = b.ytil[j];

    const long long units = (P.n + 31) >> 5;
    const long long lo = (units * blockIdx.x / gridDim.x) << 5;
    long long hi = (units * (blockIdx.x + 1) / gridDim.x) << 5;
    if (hi > P.n) hi = P.n;
    unsigned meetings = 0;
    double s_ren = 1.0;
    bool good = true;
    for (int s = 0; s < nsteps; ++s) {
        const bool end = s + 1 == nsteps, store = end && blockIdx.x == 0;
        const int set = s % 3;
        long long *hist = set ? hist2 + size_t(set - 1) * m.hist_words : b.hist;
        block_zero<T, false>(m, S);
        unsigned err = 0;
        Total<T> wtot;
        T wdep = T(0);
        step_particles<T, false, false, M0, M1, M2, M3>(m, m, k, P, b, S, f, 1, lo + threadIdx.x, hi, blockDim.x, err,
                                                        wtot, wdep);
        block_flush<T, WPS, false>(m, k, b.sc, hist, &g->wcheck[set], S, f.prior_step, err, wtot, wdep, 0);
        good = meet(g, (meetings += gridDim.x), &ok);
        if (!good) break;
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            if (!(__ldcg(&g->wcheck[set]) <= 0.5 * b.sc->Wrange)) atomicOr(&b.sc->err, kErrOverflow);
            g->wcheck[(set + 2) % 3] = 0.0;
        }
        if (spread) {
            s_ren = renorm_scale<WPS>(m, hist, 0, W0);
            for (int r = blockIdx.x; r < pl.n_ranges; r += gridDim.x) {
                const int2 r0 = pl.range[r], r1 = pl.range[r + 1];
                fin_observables<WPS>(m, b, hist, r0.x, r1.x, 0, W0, cs, pl.csum, s_ren);
                __syncthreads();
                fin_records<T>(b, r0.y, r1.y, cs);
            }
        } else {
            fin_observables<WPS>(m, b, hist, 0, pl.n_chunks, 0, W0, cs, csum, s_ren, ys, store);
            __syncthreads();
            fin_records<T>(b, 0, pl.n_elems, cs, S.c, store);
        }
        if (kLogWeights<T> && int(threadIdx.x) == int(blockDim.x) - 32) lw = log(s_ren);
        // clear the set that was read before this meeting, shared out over the blocks
        {
            const int old = (set + 2) % 3;
            long long *h = old ? hist2 + size_t(old - 1) * m.hist_words : b.hist;
            for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < m.hist_words; q += gridDim.x * blockDim.x) h[q] = 0;
        }
        if (f.prior_step) fin_priors<WPS>(m, b, hist, s_ren, blockIdx.x, gridDim.x);
        if (spread || f.prior_step) {
            good = meet(g, (meetings += gridDim.x), &ok);
            if (!good) break;
            // waited for with the first particles
            if (spread) tables_range<T>(b, S, tl.rec, tl.vp);
            if (f.prior_step) tables_range<T>(b, S, tl.prior, tl.esq);
        }
        if (store && threadIdx.x < 32) {
            const double chi2 = spread ? fin_chi2<true>(pl.csum, pl.n_chunks) : fin_chi2<false>(csum, pl.n_chunks);
            if (threadIdx.x == 0) {
                Scalars &sc = *b.sc;
                const long long t = t0 + nsteps;
                const StepHead h = next_head(m, t, t > m.n_relax ? 1 : 0, s_ren, what);
                sc.chi2 = chi2;
                sc.t = t;
                sc.Wsum = total_weight<WPS>(m, hist);
                sc.wscale = s_ren;
                sc.lwscale = h.lwscale;
                sc.pending = h.pending;
                *b.head = h;
            }
        }
        phase = phase + 1 == m.update_every ? 0 : phase + 1;
        __syncthreads();
        f.pending = t0 + s + 1 > m.n_relax ? 1 : 0;
        f.prior_step = m.mode == 1 && phase == 0;
        if constexpr (kLogWeights<T>) f.lwscale = T(lw);
        else f.wscale = T(s_ren);
    }
    if (!good && threadIdx.x == 0) atomicOr(&b.sc->err, kErrTimeout);
    tables_wait();
    // the last block to leave clears what the next launch expects clear
    if (!block_is_last(&g->done, gridDim.x, &last)) return;
    for (int q = threadIdx.x; q < m.hist_words; q += blockDim.x) b.hist[q] = 0;
    for (int q = threadIdx.x; q < 2 * m.hist_words; q += blockDim.x) hist2[q] = 0;
    if (threadIdx.x == 0) *g = Meet{};
}

template <class T>
using StepsFn = void (*)(const Model, const Cst<T>, const State<T>, const Buffers, long long *, Meet *, int, int, int);

template <class T, int WPS>
StepsFn<T> pick_steps(const Model &m)
{
    switch (step_shape(m)) {
    case kShapeKin1: return k_steps<T, WPS, kMinBlocksBatch<T>, kBitMass, kKin1, 0u, 0u>;
    case kShapeKin2: return k_steps<T, WPS, kMinBlocksBatch<T>, kBitMass, kKin2, 0u, 0u>;
    case kShapeMap: return k_steps<T, WPS, kMinBlocksBatch<T>, kMapMask, 0u, 0u, 0u>;
    default: return k_steps<T, WPS, kMinBlocksBatch<T>, kDyn, kDyn, kDyn, kDyn>;
    }
}

// Two sets of sums and the scratch of the meetings (8-byte words both).
size_t scratch_bytes(const m2m_ctx *ctx) { return sizeof(long long) * 2 * size_t(ctx->m.hist_words) + sizeof(Meet); }

template <class T, int WPS>
m2m_status setup(m2m_ctx *ctx)
{
    const Model &m = ctx->m;
    const size_t own = (ctx->smem_step + 15) / 16 * 16;
    const size_t smem = own + sizeof(double) * (size_t(m.J) + std::min(ctx->plan.n_chunks, kOwnChunks));
    int maxsm = 0;
    CU(cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device));
    if (smem > size_t(maxsm)) return M2M_OK;
    StepsFn<T> fn = pick_steps<T, WPS>(m);
    CU(allow_smem(reinterpret_cast<const void *>(fn), smem));
    int occ = 0;
    CU(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, ctx->block, smem));
    if (occ < 1) return M2M_OK;
    ctx->steps_bps = std::min(occ, ctx->bps);
    ctx->ksteps = reinterpret_cast<void *>(fn);
    ctx->smem_steps = smem;
    ctx->steps_own = int(own);
    return M2M_OK;
}

// Launches of this kernel are kept from running side by side (two kernels whose blocks wait for
// their own kind must not share out the SMs between them), and a fit never waits for another's
// stream: where the last launch on the device, on another stream, is not done yet, the fit takes
// the step-by-step route, whose kernels wait for nothing and fill the SMs beside it. Fits whose
// streams hold work at the same time so overlap; the steps are the same bits on either route.
// us per step of all of 1, 2, 4 and 8 fits on streams of their own, and with every launch waiting
// for the one before: 20,000 FP64 particles each 11.9, 20.3, 27.6, 47.6 and 11.9, 23.6, 47.2, 94.5;
// 100,000 mixed 15.6, 23.7, 29.7, 44.4 and 15.6, 30.5, 61.5, 123.
struct Turn {
    std::mutex mu;
    cudaEvent_t ev = nullptr;         // behind the last launch
    cudaStream_t stream = nullptr;    // its stream
};
Turn &turn_of(int device)
{
    static Turn turns[64];
    return turns[device & 63];
}

// Whether the fit may launch now (the caller holds t.mu).
m2m_status my_turn(m2m_ctx *ctx, Turn &t, bool &mine)
{
    mine = true;
    if (!t.ev) {
        CU(cudaEventCreateWithFlags(&t.ev, cudaEventDisableTiming));
        return M2M_OK;
    }
    // ordered by the stream itself (the per-thread handle names a stream of each thread)
    if (t.stream == ctx->stream && ctx->stream != cudaStreamPerThread) return M2M_OK;
    const RelaxedCapture relaxed;
    const cudaError_t e = cudaEventQuery(t.ev);
    if (e == cudaErrorNotReady) {
        cudaGetLastError();
        mine = false;
        return M2M_OK;
    }
    CU(e);
    return M2M_OK;
}

// Queues nsteps steps, unless it is not the fit's turn.
template <class T>
m2m_status run(m2m_ctx *ctx, int nsteps, bool &done)
{
    Model m = ctx->m;
    Cst<T> k = make_cst<T>(m);
    State<T> P = state<T>(ctx);
    Buffers b = buffers(ctx);
    long long *h2 = ctx->d_hist2;
    Meet *g = reinterpret_cast<Meet *>(h2 + 2 * ctx->m.hist_words);
    const int grid = grid_for(ctx, ctx->steps_bps);
    int spread = (grid + ctx->nsm - 1) / ctx->nsm * b.plan.n_chunks > kOwnChunks;
    void *args[] = {&m, &k, &P, &b, &h2, &g, &nsteps, &ctx->steps_own, &spread};
    Turn &t = turn_of(ctx->device);
    std::lock_guard<std::mutex> lock(t.mu);
    const m2m_status s = my_turn(ctx, t, done);
    if (s != M2M_OK || !done) return s;
    CU(cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(ctx->ksteps), dim3(grid), dim3(ctx->block),
                                   args, ctx->smem_steps, ctx->stream));
    t.stream = ctx->stream;
    CU(cudaEventRecord(t.ev, ctx->stream));
    return M2M_OK;
}

}  // namespace

// Which fits can take several steps per launch: block-shared sums, no smoothing kernels or
// self-consistent potential between the steps, not a shard, a device with cooperative launches.
m2m_status persist_setup(m2m_ctx *ctx)
{
    const Model &m = ctx->m;
    if (ctx->global_dep || m.smooth || m.pot == 3 || ctx->internal) return M2M_OK;
    int coop = 0;
    CU(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, ctx->device));
    if (!coop) return M2M_OK;
    return ctx->precision == M2M_PREC_FP64 ? setup<double, 2>(ctx) : setup<float, 1>(ctx);
}

// Whether the fit takes several steps per launch: all blocks resident at once, and in mixed
// precision at most 8,192 particles an SM. The mixed kernel for one step keeps five blocks on an SM,
// this one four (its step loop takes registers); us per step of this one and that one, Hernquist,
// 150 observables: 1,000 particles 8.6 and 13.7, 100,000 16.5 and 18.7, 1M 32.7 and 32.7,
// 2M 49.7 and 45.5. FP64 (two blocks in both): 1,000 12.8 and 17.9, 20,000 13.5 and 18.9, 1M 118.0
// and 117.4.
bool persist_fits(m2m_ctx *ctx)
{
    if (ctx->precision == M2M_PREC_MIXED && ctx->n > 8192ll * ctx->nsm) return false;
    return ctx->ksteps && grid_for(ctx, ctx->steps_bps) <= (long long)ctx->nsm * ctx->steps_bps;
}

void persist_free(m2m_ctx *ctx)
{
    free_dev(ctx->d_hist2);
}

// The scratch of these launches, zeroed, unless the fit has it.
m2m_status persist_alloc(m2m_ctx *ctx)
{
    if (!ctx->ksteps || ctx->d_hist2) return M2M_OK;
    const RelaxedCapture relaxed;
    CU(cudaMalloc(&ctx->d_hist2, scratch_bytes(ctx)));
    return persist_reset(ctx);
}

m2m_status persist_reset(m2m_ctx *ctx)
{
    if (!ctx->d_hist2) return M2M_OK;
    CU(cudaMemsetAsync(ctx->d_hist2, 0, scratch_bytes(ctx), ctx->stream));
    return M2M_OK;
}

// Queues steps in launches of at most kPersistSteps (bounded, so that other streams' work gets
// its turn) while it is the fit's turn; left: the steps that remain for the caller.
m2m_status persist_steps(m2m_ctx *ctx, int64_t &left)
{
    const m2m_status a = persist_alloc(ctx);
    if (a != M2M_OK) return a;
    while (left > 0) {
        const int now = int(std::min<int64_t>(left, kPersistSteps));
        bool done = false;
        const m2m_status s = ctx->precision == M2M_PREC_FP64 ? run<double>(ctx, now, done) : run<float>(ctx, now, done);
        if (s != M2M_OK) return s;
        if (!done) break;
        left -= now;
    }
    return M2M_OK;
}
