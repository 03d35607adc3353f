// pond.cu -- host side of libpond: the C ABI declared in include/pond.h.
//
// A context owns two state buffers of one 32-value record per node (ping-pong), a 6-plane
// FP64 staging buffer for host <-> device field copies, the block partials of the conservation sums and a
// small block of device counters.  Every call enqueues on the context stream; one time
// step is one launch of the fused kernel k_pond_step (pond_step.cuh).
#include "pond.h"

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "pond_kernels.cuh"
#include "pond_step.cuh"
#include "pond_q16.cuh"
#include "pond_q27.cuh"
#include "pond_init.cuh"
#include "pond_state.cuh"

using namespace pond;

cudaEvent_t batch_done_event(pond_batch *b);   // defined with the batches below

struct pond_ctx {
    pond_grid grid{};
    pond_eos eos{};
    pond_opts opts{};
    double kappa = 0.0, tau = 1.0;
    int device = 0;
    size_t N = 0, esize = 0;
    void *state[2] = {nullptr, nullptr};
    int cur = 0;
    double *stage = nullptr;       // 6 planes of double
    double *part = nullptr;        // conservation partials (nblk * 8) + out[4]
    int red_blocks = 0;
    DevStats *dstats = nullptr;
    cudaStream_t stream = nullptr;
    int64_t steps = 0;
    int lanes = 8;                 // work split of the D2Q9 step: 8 = a thread, 16 = nine lanes per node
    bool initialised = false;
    pond_batch *batch = nullptr;   // batch that steps this context, if any
    int nonlocal = 0;              // 1: current-time non-local terms (two passes per step)
    void *pred = nullptr;          // first pass's state (nonlocal = 1)
    DevStats *dstats_pred = nullptr;
    int lattice = POND_D2Q9;       // POND_D2Q16: node records of SLQ values; POND_D3Q27: SL27
    Grid3 g3{1, 0};                // z extent and boundary (D3Q27)
    double *nlbuf = nullptr;       // D2Q16: NL_PLANES FP64 planes of non-local terms
    std::string err;
    size_t bytes = 0;
    DevParams dp{};
    // device counters already reported by a sync point's status (sticky flags: a
    // condition is reported once, by the first sync point after it occurred)
    unsigned long long rep_nonconv = 0, rep_clamped = 0;
};

namespace {

pond_status fail(pond_ctx *c, pond_status st, const std::string &msg)
{
    if (c) c->err = msg;
    return st;
}

pond_status cuda_fail(pond_ctx *c, cudaError_t e, const char *where)
{
    return fail(c, POND_ECUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

#define CK(call, where)                                 \
    do {                                                \
        cudaError_t e_ = (call);                        \
        if (e_ != cudaSuccess) return cuda_fail(c, e_, where); \
    } while (0)

void *dev_alloc(pond_ctx *c, size_t bytes)
{
    void *p = nullptr;
    if (c->opts.dalloc) {
        p = c->opts.dalloc(bytes, c->opts.alloc_ctx);
    } else if (cudaMalloc(&p, bytes) != cudaSuccess) {
        p = nullptr;
    }
    if (p) c->bytes += bytes;
    return p;
}

void dev_free(pond_ctx *c, void *p)
{
    if (!p) return;
    if (c->opts.dfree) c->opts.dfree(p, c->opts.alloc_ctx);
    else cudaFree(p);
}

inline unsigned blocks_for(size_t n, unsigned bs) { return (unsigned)((n + bs - 1) / bs); }

bool mixed(const pond_ctx *c) { return c->opts.precision == POND_MIXED; }

// Tiles of the D2Q9 step kernel over the grid.
int step_tiles(const pond_ctx *c) { return c->dp.tiles_x * ((c->grid.ny + c->dp.tile_y - 1) / c->dp.tile_y); }

bool split(const pond_ctx *c) { return c->lanes == 16; }

template <typename R>
size_t step_smem(const pond_ctx *c)
{
    return step_smem_bytes(c->dp.tile_x, c->dp.tile_y, split(c), Slot<R>::stride, (int)sizeof(R));
}

// Lets the step kernels of type R use more than the default 48 KB of dynamic shared
// memory on the current device (idempotent; not a stream operation).
template <typename R>
cudaError_t allow_step_smem()
{
    size_t m = 0, ms = 0;
    for (int tx = 1; tx <= STEP_NB; tx *= 2)
        m = std::max(m, step_smem_bytes(tx, STEP_NB / tx, false, Slot<R>::stride, (int)sizeof(R)));
    for (int tx = 1; tx <= SPLIT_NB; ++tx)
        ms = std::max(ms, step_smem_bytes(tx, SPLIT_NB / tx, true, Slot<R>::stride, (int)sizeof(R)));
    size_t mq = 0;
    for (int tx = 1; tx <= STEP_NB; tx *= 2) mq = std::max(mq, q16_smem_bytes<R>(tx, STEP_NB / tx));
    cudaError_t e = cudaFuncSetAttribute(k_q16_step<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mq);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_q27_step<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)q27_smem_bytes<R>());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_pond_step<R, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)m);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_pond_step<R, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ms);
    return e;
}

// One launch of the D2Q9 step over `blocks` tiles of `one` or of a batch's work list.  A
// lone simulation's may begin while the stream's previous step drains (programmatic
// dependent launch: the kernel waits for that step's completion before it reads anything),
// which hides most of the launch latency between small steps: 128 x 4 nodes 14.6 -> 12.0 us
// a step, 2048 x 1 14.8 -> 12.6.
template <typename R>
cudaError_t launch_step_kernel(bool use_split, unsigned blocks, size_t smem, cudaStream_t s, const SimDesc<R> &one,
                               const SimDesc<R> *descs, const int2 *work)
{
    if (work) {   // a batch's launch, captured in its graph
        if (use_split) k_pond_step<R, true><<<blocks, STEP_THREADS, smem, s>>>(one, descs, work);
        else k_pond_step<R, false><<<blocks, STEP_THREADS, smem, s>>>(one, descs, work);
        return cudaSuccess;
    }
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(STEP_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return use_split ? cudaLaunchKernelEx(&cfg, k_pond_step<R, true>, one, descs, work)
                     : cudaLaunchKernelEx(&cfg, k_pond_step<R, false>, one, descs, work);
}

// After a step's launches: the state is the buffer they write, unless one of them failed.
pond_status step_launched(pond_ctx *c)
{
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(c, e, "step launch");
    c->cur = 1 - c->cur;
    return POND_OK;
}

// D2Q16: the non-local terms of state `src` into nlbuf, then the node step in -> out.
template <typename R>
void launch_q16_pass(pond_ctx *c, const R *in, const R *src, R *out, DevStats *stats,
                     cudaStream_t strm)
{
    const unsigned nb = blocks_for(c->N, 256);
    using W = typename Wide<R>::type;
    W *nl = reinterpret_cast<W *>(c->nlbuf);
    const dim3 blk = c->grid.ny < 4 ? dim3(256, 1) : dim3(32, 8);
    const unsigned across = blocks_for((size_t)c->grid.nx, blk.x);   // (along y a launch holds 65,535 blocks only)
    k_q16_nonlocal1<R><<<across * blocks_for((size_t)c->grid.ny, blk.y), blk, 0, strm>>>(c->dp, src, nl, (int)across);
    k_q16_nonlocal2<R><<<nb, 256, 0, strm>>>(c->dp, nl);
    k_q16_step<R><<<(unsigned)step_tiles(c), STEP_THREADS, q16_smem_bytes<R>(c->dp.tile_x, c->dp.tile_y), strm>>>(
        c->dp, in, nl, out, stats);
}

template <typename R>
pond_status launch_step_q16(pond_ctx *c, cudaEvent_t *ev)
{
    const R *in = (const R *)c->state[c->cur];
    R *out = (R *)c->state[1 - c->cur];
    if (ev) cudaEventRecord(ev[0], c->stream);
    const R *nl = in;
    if (c->nonlocal) {
        // pass 1 predicts rho, T at t (lagged terms); pass 2 redoes the step with the
        // non-local terms of that prediction
        launch_q16_pass<R>(c, in, in, (R *)c->pred, c->dstats_pred, c->stream);
        nl = (const R *)c->pred;
    }
    launch_q16_pass<R>(c, in, nl, out, c->dstats, c->stream);
    if (ev) cudaEventRecord(ev[1], c->stream);
    return step_launched(c);
}

// D3Q27: the non-local terms of state `src`, then the node step in -> out.
template <typename R>
void launch_q27_pass(pond_ctx *c, const R *in, const R *src, R *out, DevStats *stats)
{
    const unsigned nb = blocks_for(c->N, 256);
    using W = typename Wide<R>::type;
    W *nl = reinterpret_cast<W *>(c->nlbuf);
    k_q27_pi<R><<<nb, 256, 0, c->stream>>>(c->dp, src, nl);
    k_q27_nonlocal1<R><<<nb, 256, 0, c->stream>>>(c->dp, c->g3, src, nl);
    k_q27_nonlocal2<R><<<nb, 256, 0, c->stream>>>(c->dp, c->g3, nl);
    const unsigned nx = blocks_for((size_t)c->grid.nx, T27X), ny = blocks_for((size_t)c->grid.ny, T27Y);
    k_q27_step<R><<<nx * ny * blocks_for((size_t)c->g3.nz, T27Z), Q27_THREADS, q27_smem_bytes<R>(), c->stream>>>(
        c->dp, c->g3, (int)nx, (int)ny, in, nl, out, stats);
}

template <typename R>
pond_status launch_step_q27(pond_ctx *c, cudaEvent_t *ev)
{
    const R *in = (const R *)c->state[c->cur];
    R *out = (R *)c->state[1 - c->cur];
    if (ev) cudaEventRecord(ev[0], c->stream);
    const R *nl = in;
    if (c->nonlocal) {
        launch_q27_pass<R>(c, in, in, (R *)c->pred, c->dstats_pred);
        nl = (const R *)c->pred;
    }
    launch_q27_pass<R>(c, in, nl, out, c->dstats);
    if (ev) cudaEventRecord(ev[1], c->stream);
    return step_launched(c);
}

template <typename R>
pond_status launch_step(pond_ctx *c, cudaEvent_t *ev = nullptr)
{
    if (c->lattice == POND_D2Q16) return launch_step_q16<R>(c, ev);
    if (c->lattice == POND_D3Q27) return launch_step_q27<R>(c, ev);
    const R *in = (const R *)c->state[c->cur];
    R *out = (R *)c->state[1 - c->cur];
    const unsigned nb = (unsigned)step_tiles(c);
    const size_t smem = step_smem<R>(c);
    if (ev) cudaEventRecord(ev[0], c->stream);
    const R *nl = in;
    if (c->nonlocal) {
        // pass 1: the lagged step predicts rho, T at t (its counters kept apart); pass 2
        // redoes the step from the same state with the non-local terms of that prediction
        R *pred = (R *)c->pred;
        const SimDesc<R> first{c->dp, in, pred, c->dstats_pred, in};
        launch_step_kernel<R>(split(c), nb, smem, c->stream, first, nullptr, nullptr);
        nl = pred;
    }
    const SimDesc<R> one{c->dp, in, out, c->dstats, nl};
    launch_step_kernel<R>(split(c), nb, smem, c->stream, one, nullptr, nullptr);
    if (ev) cudaEventRecord(ev[1], c->stream);
    return step_launched(c);
}

template <typename R>
void launch_init(pond_ctx *c, const double *rho, const double *ux, const double *uy, const double *uz,
                 const double *T)
{
    if (c->lattice == POND_D3Q27) {
        k_q27_init<R><<<blocks_for(c->N, 256), 256, 0, c->stream>>>(c->dp, c->g3, rho, ux, uy, uz, T,
                                                                    (R *)c->state[c->cur], c->dstats);
        return;
    }
    if (c->lattice == POND_D2Q16) {
        k_q16_init<R><<<blocks_for(c->N, 256), 256, 0, c->stream>>>(c->dp, rho, ux, uy, T,
                                                                    (R *)c->state[c->cur], c->dstats);
        return;
    }
    k_init<R><<<blocks_for(c->N, 256), 256, 0, c->stream>>>(c->dp, rho, ux, uy, T,
                                                             (R *)c->state[c->cur], c->dstats);
}

template <typename R>
void launch_moments(pond_ctx *c, double *rho, double *ux, double *uy, double *uz, double *T, double *p)
{
    if (c->lattice == POND_D3Q27) {
        k_q27_moments<R><<<blocks_for(c->N, 256), 256, 0, c->stream>>>(c->dp, (const R *)c->state[c->cur],
                                                                       rho, ux, uy, uz, T, p);
        return;
    }
    if (c->lattice == POND_D2Q16) {
        k_q16_moments<R><<<blocks_for(c->N, 256), 256, 0, c->stream>>>(c->dp, (const R *)c->state[c->cur],
                                                                       rho, ux, uy, T, p);
        return;
    }
    k_moments<R><<<blocks_for(c->N, 256), 256, 0, c->stream>>>(c->dp, (const R *)c->state[c->cur],
                                                                rho, ux, uy, T, p);
}

template <typename R>
void launch_conserve(pond_ctx *c)
{
    if (c->lattice == POND_D3Q27)
        k_q27_conserve1<R><<<c->red_blocks, 256, 0, c->stream>>>(c->dp, (const R *)c->state[c->cur], c->part);
    else if (c->lattice == POND_D2Q16)
        k_q16_conserve1<R><<<c->red_blocks, 256, 0, c->stream>>>(c->dp, (const R *)c->state[c->cur], c->part);
    else
        k_conserve1<R><<<c->red_blocks, 256, 0, c->stream>>>(c->dp, (const R *)c->state[c->cur], c->part);
    k_conserve2<<<1, 32, 0, c->stream>>>(c->part, c->red_blocks, c->part + 8 * c->red_blocks);
}

pond_status check_ctx(pond_ctx *c)
{
    if (!c) return POND_EINVAL;
    c->err.clear();
    cudaError_t e = cudaSetDevice(c->device);
    if (e != cudaSuccess) return cuda_fail(c, e, "cudaSetDevice");
    // work of a batch this context belongs to comes first on the context's stream
    if (c->batch) {
        e = cudaStreamWaitEvent(c->stream, batch_done_event(c->batch), 0);
        if (e != cudaSuccess) return cuda_fail(c, e, "cudaStreamWaitEvent");
    }
    return POND_OK;
}

// Status of a sync point from the device counters hs (read after the context stream
// was synchronised): POND_ENAN while the state holds non-finite values; otherwise
// POND_ENONCONV if frame searches hit max_iter since the last report, else POND_ETHETA if
// the pressure floor was hit since the last report, else POND_OK.  A report clears both
// flags (the counts stay readable through pond_stats).
pond_status report_flags(pond_ctx *c, const DevStats &hs)
{
    if (hs.nonfinite)
        return fail(c, POND_ENAN, "non-finite values in the state (" + std::to_string(hs.nonfinite) +
                                      " node updates; see pond_stats)");
    const unsigned long long nc = hs.nonconv - std::min(hs.nonconv, c->rep_nonconv);
    const unsigned long long cl = hs.clamped - std::min(hs.clamped, c->rep_clamped);
    c->rep_nonconv = hs.nonconv;
    c->rep_clamped = hs.clamped;
    if (nc)
        return fail(c, POND_ENONCONV, "frame search hit max_iter at " + std::to_string(nc) +
                                          " node updates since the last report (results are returned)");
    if (cl)
        return fail(c, POND_ETHETA, "pressure floor hit at " + std::to_string(cl) +
                                        " node updates since the last report (results are returned)");
    return POND_OK;
}

// Enqueue the copy of the device counters into hs (read it after synchronising).
cudaError_t fetch_stats(pond_ctx *c, DevStats *hs)
{
    return cudaMemcpyAsync(hs, c->dstats, sizeof(DevStats), cudaMemcpyDeviceToHost, c->stream);
}

// Calls f(R{}, lattice state description{}) for the context's precision and lattice.
template <typename F>
pond_status with_state(const pond_ctx *c, F f)
{
    if (c->lattice == POND_D3Q27) return mixed(c) ? f(0.0f, StateD3Q27{}) : f(0.0, StateD3Q27{});
    if (c->lattice == POND_D2Q16) return mixed(c) ? f(0.0f, StateD2Q16{}) : f(0.0, StateD2Q16{});
    return mixed(c) ? f(0.0f, StateD2Q9{}) : f(0.0, StateD2Q9{});
}

constexpr int STAGE_PLANES = 6;   // planes of the staging buffer

// The state as host planes, a staging buffer's worth at a time.
template <typename R, typename S>
pond_status state_out(pond_ctx *c, double *state)
{
    const unsigned nb = blocks_for(c->N, 256);
    for (int p = 0; p < S::planes; p += STAGE_PLANES) {
        const int k = std::min(STAGE_PLANES, S::planes - p);
        k_state_out<R, S><<<nb, 256, 0, c->stream>>>((const R *)c->state[c->cur], c->N, p, k, c->stage);
        CK(cudaGetLastError(), "k_state_out launch");
        CK(cudaMemcpyAsync(state + (size_t)p * c->N, c->stage, (size_t)k * c->N * sizeof(double),
                           cudaMemcpyDeviceToHost, c->stream), "cudaMemcpyAsync D2H");
    }
    CK(cudaStreamSynchronize(c->stream), "cudaStreamSynchronize");
    return POND_OK;
}

template <typename R, typename S>
pond_status state_in(pond_ctx *c, const double *state)
{
    const unsigned nb = blocks_for(c->N, 256);
    R *st = (R *)c->state[c->cur];
    for (int p = 0; p < S::planes; p += STAGE_PLANES) {
        const int k = std::min(STAGE_PLANES, S::planes - p);
        CK(cudaMemcpyAsync(c->stage, state + (size_t)p * c->N, (size_t)k * c->N * sizeof(double),
                           cudaMemcpyHostToDevice, c->stream), "cudaMemcpyAsync H2D");
        // the non-local scratch (rewritten by every step) holds the remainders' sums
        k_state_in<R, S><<<nb, 256, 0, c->stream>>>(c->stage, c->N, p, k, st, c->nlbuf);
        CK(cudaGetLastError(), "k_state_in launch");
    }
    if constexpr (S::q != 9 && sizeof(R) == 4) {
        k_state_finish<S><<<nb, 256, 0, c->stream>>>(c->N, st, c->nlbuf);
        CK(cudaGetLastError(), "k_state_finish launch");
    }
    CK(cudaStreamSynchronize(c->stream), "cudaStreamSynchronize");
    return POND_OK;
}

pond_status init_common(pond_ctx *c, const double *d_rho, const double *d_ux, const double *d_uy,
                        const double *d_uz, const double *d_T)
{
    CK(cudaMemsetAsync(c->dstats, 0, sizeof(DevStats), c->stream), "cudaMemsetAsync");
    if (mixed(c)) launch_init<float>(c, d_rho, d_ux, d_uy, d_uz, d_T);
    else launch_init<double>(c, d_rho, d_ux, d_uy, d_uz, d_T);
    CK(cudaGetLastError(), "k_init launch");
    DevStats hs{};
    CK(cudaMemcpyAsync(&hs, c->dstats, sizeof(DevStats), cudaMemcpyDeviceToHost, c->stream), "cudaMemcpyAsync");
    CK(cudaStreamSynchronize(c->stream), "cudaStreamSynchronize");
    CK(cudaMemsetAsync(c->dstats, 0, sizeof(DevStats), c->stream), "cudaMemsetAsync");
    if (hs.bad_init)
        return fail(c, POND_EINVAL, "init fields need rho > 0, b*rho < 1 and T > 0 at every node ("
                                        + std::to_string(hs.bad_init) + " nodes violate it)");
    c->initialised = true;
    c->steps = 0;
    c->rep_nonconv = c->rep_clamped = 0;
    return POND_OK;
}

// ---------------------------------------------------------------------------
// Allocation-free conservation sums.  Scratch for the block partials lives in this
// file-scope device array instead of memory the caller or the library allocates: every
// device that loads the library holds these NOALLOC_SCRATCH_DOUBLES doubles until the
// process exits.  Host code may not pass the symbol itself to a kernel (it is a host-side
// stand-in, not a device address); the device address is looked up once per device.
constexpr int NOALLOC_SPAN = 2048;          // nodes summed by one block
constexpr int NOALLOC_MAX_BLOCKS = 4096;    // => at most 8,388,608 nodes per call
constexpr int NOALLOC_SCRATCH_DOUBLES = 8 * NOALLOC_MAX_BLOCKS + 8;
static __device__ __align__(256) double g_noalloc_scratch[NOALLOC_SCRATCH_DOUBLES];

constexpr int NOALLOC_MAX_DEVICES = 64;
std::mutex g_noalloc_mutex;
double *g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {nullptr};

// Device address of g_noalloc_scratch on the current device, looked up on first use.
cudaError_t noalloc_scratch(double **ptr)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        g_noalloc_ptr[dev] = (double *)p;
    }
    *ptr = g_noalloc_ptr[dev];
    return cudaSuccess;
}

}  // namespace

namespace {
// 8 independent chains a = a * m + c per thread (m, c chosen so that values stay finite
// and the compiler cannot fold them); one value per thread is written so that nothing
// is eliminated.
template <typename R>
__global__ void k_fma_chains(R *out, int iters, R m, R c)
{
    R a[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) a[k] = R(threadIdx.x + k) * R(1e-3);
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int k = 0; k < 8; ++k) a[k] = fma(a[k], m, c);
    }
    R s = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += a[k];
    out[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = s;
}

template <typename R>
pond_status fma_peak(int iters, cudaStream_t s, double *tflops)
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return POND_ECUDA;
    const int blocks = 8 * sms, threads = 256;
    R *out = nullptr;
    if (cudaMalloc((void **)&out, (size_t)blocks * threads * sizeof(R)) != cudaSuccess) return POND_ECUDA;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    k_fma_chains<R><<<blocks, threads, 0, s>>>(out, iters / 10 + 1, R(0.999999), R(1e-6));   // warm-up
    cudaEventRecord(e0, s);
    k_fma_chains<R><<<blocks, threads, 0, s>>>(out, iters, R(0.999999), R(1e-6));
    cudaEventRecord(e1, s);
    cudaError_t e = cudaEventSynchronize(e1);
    float ms = 0.0f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    if (e == cudaSuccess) e = cudaGetLastError();
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(out);
    if (e != cudaSuccess || !(ms > 0.0f)) return POND_ECUDA;
    *tflops = 2.0 * 8.0 * (double)iters * blocks * threads / (ms * 1e-3) / 1e12;
    return POND_OK;
}
}  // namespace

extern "C" {

pond_status pond_conservation_noalloc(const double *d_planes, int64_t n_nodes, double out[4],
                                      void *stream)
{
    if (!d_planes || !out || n_nodes < 1) return POND_EINVAL;
    if (n_nodes > (int64_t)NOALLOC_SPAN * NOALLOC_MAX_BLOCKS) return POND_EINVAL;
    double *scratch = nullptr;
    if (noalloc_scratch(&scratch) != cudaSuccess) return POND_ECUDA;
    cudaStream_t s = (cudaStream_t)stream;
    const int nb = (int)((n_nodes + NOALLOC_SPAN - 1) / NOALLOC_SPAN);
    // launch errors are peeked right after each launch (a sticky error left by other work
    // is neither taken nor cleared here); the stream's synchronisation decides the result
    k_conserve_planes1<<<nb, 256, 0, s>>>(d_planes, (long long)n_nodes, NOALLOC_SPAN, scratch);
    if (cudaPeekAtLastError() != cudaSuccess) return POND_ECUDA;
    k_conserve2<<<1, 32, 0, s>>>(scratch, nb, scratch + 8 * NOALLOC_MAX_BLOCKS);
    if (cudaPeekAtLastError() != cudaSuccess) return POND_ECUDA;
    if (cudaMemcpyAsync(out, scratch + 8 * NOALLOC_MAX_BLOCKS, 4 * sizeof(double),
                        cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return POND_ECUDA;
    return cudaStreamSynchronize(s) == cudaSuccess ? POND_OK : POND_ECUDA;
}


const char *pond_version(void) { return "pond-gb300 0.1 (sm_103a)"; }


pond_status pond_fma_peak(int32_t precision, int32_t iters, void *stream, double *tflops_out)
{
    if (!tflops_out || iters < 1 || (precision != POND_MIXED && precision != POND_FP64)) return POND_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    return precision == POND_MIXED ? fma_peak<float>(iters, s, tflops_out)
                                   : fma_peak<double>(iters, s, tflops_out);
}

const char *pond_last_error(const pond_ctx *ctx) { return ctx ? ctx->err.c_str() : "null context"; }

size_t pond_device_bytes(const pond_ctx *ctx) { return ctx ? ctx->bytes : 0; }

pond_status pond_create(const pond_grid *grid, const pond_lattice *lattice, const pond_eos *eos,
                        double kappa, double tau, const pond_opts *opts, pond_ctx **out)
{
    if (!out) return POND_EINVAL;
    *out = nullptr;
    if (!grid || !lattice || !eos || !opts) return POND_EINVAL;
    if (grid->nx < 1 || grid->ny < 1) return POND_EINVAL;
    if ((grid->bc_x != POND_PERIODIC && grid->bc_x != POND_ZEROGRAD) ||
        (grid->bc_y != POND_PERIODIC && grid->bc_y != POND_ZEROGRAD))
        return POND_EINVAL;
    if (lattice->kind != POND_D2Q9 && lattice->kind != POND_D2Q16 && lattice->kind != POND_D3Q27)
        return POND_EINVAL;
    // z extent: 0 or 1 on the two-dimensional lattices; >= 1 on D3Q27
    if (grid->nz < 0 || (lattice->kind != POND_D3Q27 && grid->nz > 1)) return POND_EINVAL;
    if (lattice->kind == POND_D3Q27 && (grid->nz < 1 || (grid->bc_z != POND_PERIODIC && grid->bc_z != POND_ZEROGRAD)))
        return POND_EINVAL;
    if (eos->kind != POND_VDW && eos->kind != POND_IDEAL && eos->kind != POND_DIETERICI &&
        eos->kind != POND_SIMPLIFIED)
        return POND_EINVAL;
    if (eos->kind == POND_SIMPLIFIED &&
        (!eos->isothermal || !(eos->beta > 0.0) || !(eos->rho_v > 0.0) || !(eos->rho_l > eos->rho_v) ||
         !(eos->p0 > 0.0)))
        return POND_EINVAL;
    if (eos->isothermal != 0 && eos->isothermal != 1) return POND_EINVAL;
    if (eos->isothermal && !(eos->T_iso > 0.0 && std::isfinite(eos->T_iso))) return POND_EINVAL;
    if (eos->kind == POND_DIETERICI && (!eos->isothermal || !(eos->a > 0.0) || !(eos->b > 0.0)))
        return POND_EINVAL;
    if (!(eos->R > 0.0) || !(eos->delta > 0.0) || !(eos->delta <= 2.0 / 3.0 + 1e-12)) return POND_EINVAL;
    if (eos->kind == POND_VDW && (!(eos->a >= 0.0) || !(eos->b >= 0.0))) return POND_EINVAL;
    if (!(kappa >= 0.0) || !(tau > 0.5) || !std::isfinite(tau) || !std::isfinite(kappa)) return POND_EINVAL;
    if (opts->precision != POND_FP64 && opts->precision != POND_MIXED) return POND_EINVAL;
    if (!(opts->dt > 0.0) || !(opts->dt <= 1.0)) return POND_EINVAL;
    if (!(opts->tol > 0.0) || opts->max_iter < 1 || opts->max_iter > 1000) return POND_EINVAL;
    if (!(opts->p_floor > 0.0)) return POND_EINVAL;
    if ((opts->dalloc == nullptr) != (opts->dfree == nullptr)) return POND_EINVAL;
    if (opts->lanes_per_node != 0 && opts->lanes_per_node != 8 && opts->lanes_per_node != 16)
        return POND_EINVAL;
    if (opts->nonlocal != POND_NONLOCAL_LAGGED && opts->nonlocal != POND_NONLOCAL_CURRENT)
        return POND_EINVAL;
    if (opts->tile_x != 0 && opts->tile_x != 1 && opts->tile_x != 2 && opts->tile_x != 4 &&
        opts->tile_x != 8 && opts->tile_x != 16)
        return POND_EINVAL;

    pond_ctx *c = new pond_ctx();
    c->grid = *grid;
    c->eos = *eos;
    if (eos->kind == POND_IDEAL) { c->eos.a = 0.0; c->eos.b = 0.0; }
    c->opts = *opts;
    c->lattice = lattice->kind;
    c->kappa = kappa;
    c->tau = tau;
    c->stream = (cudaStream_t)opts->stream;
    c->N = (size_t)grid->nx * (size_t)grid->ny * (size_t)(grid->nz > 1 ? grid->nz : 1);
    if (c->lattice == POND_D3Q27) c->g3 = Grid3{grid->nz, grid->bc_z};
    c->esize = opts->precision == POND_MIXED ? sizeof(float) : sizeof(double);
    cudaError_t e = cudaGetDevice(&c->device);
    int sms = 0;
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
    if (e == cudaSuccess)
        e = opts->precision == POND_MIXED ? allow_step_smem<float>() : allow_step_smem<double>();
    if (e != cudaSuccess) {
        delete c;
        return POND_ECUDA;
    }
    const StepShape shape = step_shape(c->lattice == POND_D2Q9, opts->precision == POND_MIXED, grid->nx, grid->ny,
                                       opts->lanes_per_node, opts->tile_x, sms);
    c->lanes = shape.lanes;
    DevParams &d = c->dp;
    d.nx = grid->nx; d.ny = grid->ny; d.bcx = grid->bc_x; d.bcy = grid->bc_y;
    d.N = (long long)c->N;
    d.a = c->eos.a; d.b = c->eos.b; d.R = c->eos.R; d.delta = c->eos.delta; d.cv = c->eos.R / c->eos.delta;
    d.kappa = kappa; d.tau = tau; d.omega = 1.0 / tau; d.dt = opts->dt; d.k_cond = opts->k_cond;
    d.p_floor = opts->p_floor; d.tol = opts->tol; d.max_iter = opts->max_iter;
    d.tile_x = shape.tx; d.tile_y = shape.ty; d.tiles_x = (grid->nx + shape.tx - 1) / shape.tx;
    d.pd.a = d.a; d.pd.b = d.b; d.pd.R = d.R; d.pd.cv = d.cv; d.pd.inv_cv = 1.0 / d.cv;
    d.pd.kappa = d.kappa; d.pd.p_floor = d.p_floor; d.pd.dt = d.dt; d.pd.omega = d.omega;
    d.pd.mu_coef = (d.tau - 0.5) * d.dt; d.pd.cvR = d.cv + d.R; d.pd.k_cond = d.k_cond;
    d.pf.a = (float)d.pd.a; d.pf.b = (float)d.pd.b; d.pf.R = (float)d.pd.R; d.pf.cv = (float)d.pd.cv;
    d.pf.inv_cv = (float)d.pd.inv_cv; d.pf.kappa = (float)d.pd.kappa; d.pf.p_floor = (float)d.pd.p_floor;
    d.pf.dt = (float)d.pd.dt; d.pf.omega = (float)d.pd.omega; d.pf.mu_coef = (float)d.pd.mu_coef;
    d.pf.cvR = (float)d.pd.cvR; d.pf.k_cond = (float)d.pd.k_cond;
    auto split = [](double x, float out[2]) {
        out[0] = (float)x;
        out[1] = (float)(x - (double)out[0]);
    };
    split(d.a, d.ff_a); split(d.b, d.ff_b); split(d.R, d.ff_R); split(d.pd.inv_cv, d.ff_icv);
    split(d.p_floor, d.ff_pfl); split(d.dt, d.ff_dt);
    split(d.kappa, d.ff_kap); split(d.cv, d.ff_cv); split(d.pd.mu_coef, d.ff_mu); split(d.pd.cvR, d.ff_cvR);
    split(d.k_cond, d.ff_kc);
    d.tol_f = (float)d.tol;
    d.eos_kind = c->eos.kind == POND_DIETERICI ? 2 : (c->eos.kind == POND_SIMPLIFIED ? 3 : 0);
    d.sp[0] = c->eos.beta; d.sp[1] = c->eos.rho_l; d.sp[2] = c->eos.rho_v; d.sp[3] = c->eos.p0;
    for (int k = 0; k < 4; ++k) d.spf[k] = (float)d.sp[k];
    split(d.sp[3], d.ff_p0);
    d.isothermal = c->eos.isothermal;
    d.T_iso = c->eos.isothermal ? c->eos.T_iso : 0.0;
    split(d.T_iso, d.ff_Tiso);

    c->red_blocks = (int)std::min<size_t>(1024, std::max<size_t>(1, (c->N + 255) / 256));
    size_t sb = (size_t)(c->lattice == POND_D2Q16 ? SLQ : (c->lattice == POND_D3Q27 ? SL27 : SL)) * c->N * c->esize;
    c->state[0] = dev_alloc(c, sb);
    c->state[1] = dev_alloc(c, sb);
    c->stage = (double *)dev_alloc(c, STAGE_PLANES * c->N * sizeof(double));
    c->part = (double *)dev_alloc(c, (8 * (size_t)c->red_blocks + 8) * sizeof(double));
    c->dstats = (DevStats *)dev_alloc(c, sizeof(DevStats));
    if (c->lattice == POND_D2Q16) c->nlbuf = (double *)dev_alloc(c, (size_t)NL_PLANES * c->N * sizeof(double));
    if (c->lattice == POND_D3Q27) c->nlbuf = (double *)dev_alloc(c, (size_t)N3_PLANES * c->N * sizeof(double));
    c->nonlocal = opts->nonlocal;
    if (c->nonlocal) {
        c->pred = dev_alloc(c, sb);
        c->dstats_pred = (DevStats *)dev_alloc(c, sizeof(DevStats));
    }
    if (!c->state[0] || !c->state[1] || !c->stage || !c->part || !c->dstats ||
        (c->nonlocal && (!c->pred || !c->dstats_pred)) || (c->lattice != POND_D2Q9 && !c->nlbuf)) {
        pond_destroy(c);
        return POND_ENOMEM;
    }
    if (cudaMemsetAsync(c->dstats, 0, sizeof(DevStats), c->stream) != cudaSuccess) {
        pond_destroy(c);
        return POND_ECUDA;
    }
    *out = c;
    return POND_OK;
}

void pond_destroy(pond_ctx *c)
{
    if (!c) return;
    if (c->batch) pond_batch_remove(c->batch, c);
    cudaSetDevice(c->device);
    if (c->stream) cudaStreamSynchronize(c->stream);
    else cudaDeviceSynchronize();
    dev_free(c, c->state[0]);
    dev_free(c, c->state[1]);
    dev_free(c, c->stage);
    dev_free(c, c->part);
    dev_free(c, c->dstats);
    dev_free(c, c->pred);
    dev_free(c, c->dstats_pred);
    dev_free(c, c->nlbuf);
    delete c;
}

pond_status pond_init_fields(pond_ctx *c, const double *rho, const double *ux, const double *uy,
                             const double *T)
{
    pond_status st = check_ctx(c);
    if (st) return st;
    if (!rho || !ux || !uy || !T) return fail(c, POND_EINVAL, "null field pointer");
    size_t bytes = c->N * sizeof(double);
    const double *src[4] = {rho, ux, uy, T};
    for (int k = 0; k < 4; ++k)
        CK(cudaMemcpyAsync(c->stage + k * c->N, src[k], bytes, cudaMemcpyHostToDevice, c->stream),
           "cudaMemcpyAsync H2D");
    CK(cudaMemsetAsync(c->stage + 4 * c->N, 0, bytes, c->stream), "cudaMemsetAsync");   // u_z = 0
    return init_common(c, c->stage, c->stage + c->N, c->stage + 2 * c->N, c->stage + 4 * c->N,
                       c->stage + 3 * c->N);
}

pond_status pond_init_fields3(pond_ctx *c, const double *rho, const double *ux, const double *uy,
                              const double *uz, const double *T)
{
    pond_status st = check_ctx(c);
    if (st) return st;
    if (!rho || !ux || !uy || !uz || !T) return fail(c, POND_EINVAL, "null field pointer");
    size_t bytes = c->N * sizeof(double);
    const double *src[5] = {rho, ux, uy, T, uz};
    for (int k = 0; k < 5; ++k)
        CK(cudaMemcpyAsync(c->stage + k * c->N, src[k], bytes, cudaMemcpyHostToDevice, c->stream),
           "cudaMemcpyAsync H2D");
    return init_common(c, c->stage, c->stage + c->N, c->stage + 2 * c->N, c->stage + 4 * c->N,
                       c->stage + 3 * c->N);
}

pond_status pond_init_fields_device(pond_ctx *c, const double *d_rho, const double *d_ux,
                                    const double *d_uy, const double *d_T)
{
    pond_status st = check_ctx(c);
    if (st) return st;
    if (!d_rho || !d_ux || !d_uy || !d_T) return fail(c, POND_EINVAL, "null field pointer");
    CK(cudaMemsetAsync(c->stage + 4 * c->N, 0, c->N * sizeof(double), c->stream), "cudaMemsetAsync");
    return init_common(c, d_rho, d_ux, d_uy, c->stage + 4 * c->N, d_T);
}

pond_status pond_step(pond_ctx *c, int64_t n)
{
    pond_status st = check_ctx(c);
    if (st) return st;
    if (n < 0) return fail(c, POND_EINVAL, "negative step count");
    if (!c->initialised) return fail(c, POND_EINVAL, "state not initialised");
    if (c->batch) return fail(c, POND_EINVAL, "context belongs to a batch: step it with pond_batch_step");
    for (int64_t k = 0; k < n; ++k) {
        st = mixed(c) ? launch_step<float>(c) : launch_step<double>(c);
        if (st) return st;
        ++c->steps;
    }
    return POND_OK;
}

pond_status pond_step_timed(pond_ctx *c, double *ms_out)
{
    pond_status st = check_ctx(c);
    if (st) return st;
    if (!ms_out) return fail(c, POND_EINVAL, "null output");
    if (!c->initialised) return fail(c, POND_EINVAL, "state not initialised");
    cudaEvent_t ev[2];
    for (int k = 0; k < 2; ++k) CK(cudaEventCreate(&ev[k]), "cudaEventCreate");
    st = mixed(c) ? launch_step<float>(c, ev) : launch_step<double>(c, ev);
    cudaError_t e = st ? cudaSuccess : cudaEventSynchronize(ev[1]);
    float ms = 0.f;
    if (!st && e == cudaSuccess) e = cudaEventElapsedTime(&ms, ev[0], ev[1]);
    *ms_out = ms;
    for (int k = 0; k < 2; ++k) cudaEventDestroy(ev[k]);
    if (st) return st;
    if (e != cudaSuccess) return cuda_fail(c, e, "pond_step_timed");
    c->steps += 1;
    return POND_OK;
}

pond_status pond_moments_device(pond_ctx *c, double *rho, double *ux, double *uy, double *T, double *p)
{
    pond_status st = check_ctx(c);
    if (st) return st;
    if (!c->initialised) return fail(c, POND_EINVAL, "state not initialised");
    if (mixed(c)) launch_moments<float>(c, rho, ux, uy, nullptr, T, p);
    else launch_moments<double>(c, rho, ux, uy, nullptr, T, p);
    CK(cudaGetLastError(), "k_moments launch");
    return POND_OK;
}

pond_status pond_moments(pond_ctx *c, double *rho, double *ux, double *uy, double *T, double *p)
{
    pond_status st = check_ctx(c);
    if (st) return st;
    if (!c->initialised) return fail(c, POND_EINVAL, "state not initialised");
    double *host[5] = {rho, ux, uy, T, p};
    double *dev[5];
    for (int k = 0; k < 5; ++k) dev[k] = host[k] ? c->stage + k * c->N : nullptr;
    st = pond_moments_device(c, dev[0], dev[1], dev[2], dev[3], dev[4]);
    if (st) return st;
    for (int k = 0; k < 5; ++k)
        if (host[k])
            CK(cudaMemcpyAsync(host[k], dev[k], c->N * sizeof(double), cudaMemcpyDeviceToHost, c->stream),
               "cudaMemcpyAsync D2H");
    DevStats hs{};
    CK(fetch_stats(c, &hs), "cudaMemcpyAsync D2H");
    CK(cudaStreamSynchronize(c->stream), "cudaStreamSynchronize");
    return report_flags(c, hs);
}

pond_status pond_moments3(pond_ctx *c, double *rho, double *ux, double *uy, double *uz, double *T,
                          double *p)
{
    pond_status st = check_ctx(c);
    if (st) return st;
    if (!c->initialised) return fail(c, POND_EINVAL, "state not initialised");
    double *host[6] = {rho, ux, uy, uz, T, p};
    double *dev[6];
    for (int k = 0; k < 6; ++k) dev[k] = host[k] ? c->stage + k * c->N : nullptr;
    if (c->lattice == POND_D3Q27) {
        if (mixed(c)) launch_moments<float>(c, dev[0], dev[1], dev[2], dev[3], dev[4], dev[5]);
        else launch_moments<double>(c, dev[0], dev[1], dev[2], dev[3], dev[4], dev[5]);
    } else {
        // two-dimensional lattices: u_z = 0
        if (mixed(c)) launch_moments<float>(c, dev[0], dev[1], dev[2], nullptr, dev[4], dev[5]);
        else launch_moments<double>(c, dev[0], dev[1], dev[2], nullptr, dev[4], dev[5]);
        if (dev[3]) CK(cudaMemsetAsync(dev[3], 0, c->N * sizeof(double), c->stream), "cudaMemsetAsync");
    }
    CK(cudaGetLastError(), "k_moments launch");
    for (int k = 0; k < 6; ++k)
        if (host[k])
            CK(cudaMemcpyAsync(host[k], dev[k], c->N * sizeof(double), cudaMemcpyDeviceToHost, c->stream),
               "cudaMemcpyAsync D2H");
    DevStats hs{};
    CK(fetch_stats(c, &hs), "cudaMemcpyAsync D2H");
    CK(cudaStreamSynchronize(c->stream), "cudaStreamSynchronize");
    return report_flags(c, hs);
}

pond_status pond_conservation(pond_ctx *c, double out[4])
{
    pond_status st = check_ctx(c);
    if (st) return st;
    if (!out) return fail(c, POND_EINVAL, "null output");
    if (!c->initialised) return fail(c, POND_EINVAL, "state not initialised");
    if (mixed(c)) launch_conserve<float>(c);
    else launch_conserve<double>(c);
    CK(cudaGetLastError(), "conservation launch");
    CK(cudaMemcpyAsync(out, c->part + 8 * c->red_blocks, 4 * sizeof(double), cudaMemcpyDeviceToHost,
                       c->stream), "cudaMemcpyAsync D2H");
    DevStats hs{};
    CK(fetch_stats(c, &hs), "cudaMemcpyAsync D2H");
    CK(cudaStreamSynchronize(c->stream), "cudaStreamSynchronize");
    return report_flags(c, hs);
}

pond_status pond_get_state(pond_ctx *c, double *state)
{
    pond_status st = check_ctx(c);
    if (st) return st;
    if (!state) return fail(c, POND_EINVAL, "null output");
    if (!c->initialised) return fail(c, POND_EINVAL, "state not initialised");
    return with_state(c, [&](auto r, auto lat) { return state_out<decltype(r), decltype(lat)>(c, state); });
}

pond_status pond_set_state(pond_ctx *c, const double *state)
{
    pond_status st = check_ctx(c);
    if (st) return st;
    if (!state) return fail(c, POND_EINVAL, "null input");
    st = with_state(c, [&](auto r, auto lat) { return state_in<decltype(r), decltype(lat)>(c, state); });
    if (st) return st;
    c->initialised = true;
    return POND_OK;
}

pond_status pond_stats(pond_ctx *c, pond_stats_t *out, int32_t reset)
{
    pond_status st = check_ctx(c);
    if (st) return st;
    if (!out) return fail(c, POND_EINVAL, "null output");
    DevStats hs{};
    CK(cudaMemcpyAsync(&hs, c->dstats, sizeof(DevStats), cudaMemcpyDeviceToHost, c->stream),
       "cudaMemcpyAsync D2H");
    if (reset) CK(cudaMemsetAsync(c->dstats, 0, sizeof(DevStats), c->stream), "cudaMemsetAsync");
    CK(cudaStreamSynchronize(c->stream), "cudaStreamSynchronize");
    if (reset) c->rep_nonconv = c->rep_clamped = 0;
    out->steps = c->steps;
    out->node_updates = c->steps * (int64_t)c->N;
    out->streams = (int64_t)hs.streams;
    out->nonconverged = (int64_t)hs.nonconv;
    out->clamped = (int64_t)hs.clamped;
    out->nonfinite = (int64_t)hs.nonfinite;
    out->stalled = (int64_t)hs.stalled;
    out->block_streams = (int64_t)hs.block_streams;
    out->max_streams = (int64_t)hs.max_streams;
    out->timeouts = 0;
    out->region_nodes = (int64_t)hs.region_nodes;
    out->pair_streams = (int64_t)hs.pair_streams;
    return hs.nonfinite ? fail(c, POND_ENAN, "non-finite values in the state") : POND_OK;
}

// ---------------------------------------------------------------------------
// Batches: many simulations stepped by one launch per (precision, lanes) group and step.

}  // extern "C"

struct pond_batch {
    int device = 0;
    cudaStream_t stream = nullptr;
    std::vector<pond_ctx *> sims;
    bool dirty = true;
    int64_t since_build = 0;          // batch steps since the device lists were built
    cudaEvent_t done = nullptr;       // recorded after every batch step call
    std::string err;
    struct Group {
        int precision = 0, lanes = 8;
        std::vector<pond_ctx *> sims;
        void *desc[2] = {nullptr, nullptr};   // SimDesc arrays for even / odd steps
        int2 *work = nullptr;
        size_t desc_cap = 0, work_cap = 0;
        int nwork = 0;
        size_t smem = 0;
    };
    Group g[4];                       // (fp64, mixed) x (8, 16 lanes)
    // D2Q16 contexts: stepped by their own three launches on the batch stream; cur0 is
    // the context's current buffer when the lists were built
    struct Q16 { pond_ctx *c; int cur0; };
    std::vector<Q16> q16;
    // the members' chains of launches run beside each other inside the graph: the first on
    // the batch stream, the others on these
    static constexpr int SIDES = 4;
    cudaStream_t side[SIDES] = {};
    cudaEvent_t fork = nullptr, join[SIDES] = {};
    cudaGraphExec_t graph = nullptr;  // two steps (even, odd) of every group
    bool graph_ok = false;
    size_t budget = 0;                // device bytes the members may hold (0: no limit)
    size_t member_bytes = 0;          // sum of the members' pond_device_bytes
};

cudaEvent_t batch_done_event(pond_batch *b) { return b->done; }

namespace {

pond_status bfail(pond_batch *b, pond_status st, const std::string &m)
{
    b->err = m;
    return st;
}


template <typename R>
cudaError_t build_group(pond_batch *b, pond_batch::Group &G)
{
    const size_t ns = G.sims.size();
    std::vector<SimDesc<R>> d0(ns), d1(ns);
    std::vector<int2> work;
    G.smem = 0;
    for (size_t k = 0; k < ns; ++k) {
        pond_ctx *c = G.sims[k];
        d0[k].p = c->dp; d0[k].in = (const R *)c->state[c->cur]; d0[k].out = (R *)c->state[1 - c->cur];
        d0[k].stats = c->dstats; d0[k].nlsrc = d0[k].in;
        d1[k] = d0[k]; d1[k].in = (const R *)c->state[1 - c->cur]; d1[k].out = (R *)c->state[c->cur];
        d1[k].nlsrc = d1[k].in;
        const int tiles = step_tiles(c);
        for (int t = 0; t < tiles; ++t) work.push_back(make_int2((int)k, t));
        G.smem = std::max(G.smem, step_smem<R>(c));
    }
    G.nwork = (int)work.size();
    cudaError_t e = cudaSuccess;
    if (ns * sizeof(SimDesc<R>) > G.desc_cap) {
        for (int k = 0; k < 2; ++k) { cudaFree(G.desc[k]); G.desc[k] = nullptr; }
        G.desc_cap = 2 * ns * sizeof(SimDesc<R>);
        for (int k = 0; k < 2 && e == cudaSuccess; ++k) e = cudaMalloc(&G.desc[k], G.desc_cap);
        if (e != cudaSuccess) { G.desc_cap = 0; return e; }
    }
    if (work.size() * sizeof(int2) > G.work_cap) {
        cudaFree(G.work); G.work = nullptr;
        G.work_cap = 2 * work.size() * sizeof(int2);
        e = cudaMalloc((void **)&G.work, G.work_cap);
        if (e != cudaSuccess) { G.work_cap = 0; return e; }
    }
    if (ns) {
        e = cudaMemcpyAsync(G.desc[0], d0.data(), ns * sizeof(SimDesc<R>), cudaMemcpyHostToDevice, b->stream);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(G.desc[1], d1.data(), ns * sizeof(SimDesc<R>), cudaMemcpyHostToDevice, b->stream);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(G.work, work.data(), work.size() * sizeof(int2), cudaMemcpyHostToDevice, b->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);   // host vectors go out of scope
    }
    return e;
}

template <typename R>
void launch_group(const pond_batch::Group &G, int parity, cudaStream_t s)
{
    const SimDesc<R> *d = (const SimDesc<R> *)G.desc[parity];
    launch_step_kernel<R>(G.lanes == 16, (unsigned)G.nwork, G.smem, s, SimDesc<R>{}, d, G.work);
}

template <typename R>
void launch_q16_entry(const pond_batch::Q16 &e, int parity, cudaStream_t s)
{
    pond_ctx *c = e.c;
    const int ci = e.cur0 ^ parity;
    const R *in = (const R *)c->state[ci];
    launch_q16_pass<R>(c, in, in, (R *)c->state[1 - ci], c->dstats, s);
}

// The steps `first` .. `first + steps - 1` (parities) of every group and D2Q16 member: chain
// k of launches on the stream on(k).
template <typename On>
void launch_all(pond_batch *b, int first, int steps, On on)
{
    int k = 0;
    for (int g = 0; g < 4; ++g) {
        if (!b->g[g].nwork) continue;
        const cudaStream_t s = on(k++);
        for (int t = first; t < first + steps; ++t) {
            if (b->g[g].precision == POND_MIXED) launch_group<float>(b->g[g], t % 2, s);
            else launch_group<double>(b->g[g], t % 2, s);
        }
    }
    for (const pond_batch::Q16 &e : b->q16) {
        const cudaStream_t s = on(k++);
        for (int t = first; t < first + steps; ++t) {
            if (mixed(e.c)) launch_q16_entry<float>(e, t % 2, s);
            else launch_q16_entry<double>(e, t % 2, s);
        }
    }
}

// Captures two steps (even, then odd) of every member; the members' chains are independent
// until both are done, so that a group of few blocks does not hold up the others.
cudaError_t capture_two_steps(pond_batch *b, cudaGraph_t *graph)
{
    cudaError_t e = cudaSuccess;
    if (!b->fork) e = cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming);
    for (int k = 0; k < pond_batch::SIDES && e == cudaSuccess; ++k) {
        if (!b->side[k]) e = cudaStreamCreateWithFlags(&b->side[k], cudaStreamNonBlocking);
        if (e == cudaSuccess && !b->join[k]) e = cudaEventCreateWithFlags(&b->join[k], cudaEventDisableTiming);
    }
    if (e != cudaSuccess) return e;
    e = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return e;
    bool used[pond_batch::SIDES] = {};
    cudaEventRecord(b->fork, b->stream);
    launch_all(b, 0, 2, [&](int k) -> cudaStream_t {
        const int j = k % (pond_batch::SIDES + 1);
        if (j == 0) return b->stream;
        if (!used[j - 1]) cudaStreamWaitEvent(b->side[j - 1], b->fork, 0);
        used[j - 1] = true;
        return b->side[j - 1];
    });
    for (int k = 0; k < pond_batch::SIDES; ++k)
        if (used[k]) {
            cudaEventRecord(b->join[k], b->side[k]);
            cudaStreamWaitEvent(b->stream, b->join[k], 0);
        }
    return cudaStreamEndCapture(b->stream, graph);
}

pond_status batch_build(pond_batch *b)
{
    for (int k = 0; k < 4; ++k) {
        b->g[k].precision = (k & 1) ? POND_MIXED : POND_FP64;
        b->g[k].lanes = (k & 2) ? 16 : 8;
        b->g[k].sims.clear();
    }
    b->q16.clear();
    for (pond_ctx *c : b->sims) {
        if (c->lattice == POND_D2Q16) {
            b->q16.push_back({c, c->cur});
            continue;
        }
        const int k = (c->opts.precision == POND_MIXED ? 1 : 0) | (c->lanes == 16 ? 2 : 0);
        b->g[k].sims.push_back(c);
    }
    for (int k = 0; k < 4; ++k) {
        cudaError_t e = (k & 1) ? build_group<float>(b, b->g[k]) : build_group<double>(b, b->g[k]);
        if (e != cudaSuccess) return bfail(b, POND_ECUDA, std::string("batch build: ") + cudaGetErrorString(e));
    }
    if (b->graph) { cudaGraphExecDestroy(b->graph); b->graph = nullptr; }
    b->graph_ok = false;
    // capture two steps (even then odd parity) of every group once; replays step the batch
    if (b->stream) {
        cudaGraph_t graph = nullptr;
        if (capture_two_steps(b, &graph) == cudaSuccess && graph &&
            cudaGraphInstantiate(&b->graph, graph, 0) == cudaSuccess)
            b->graph_ok = true;
        if (graph) cudaGraphDestroy(graph);
        cudaGetLastError();   // a failed capture falls back to plain launches
    }
    b->dirty = false;
    b->since_build = 0;
    return POND_OK;
}

}  // namespace

extern "C" {

pond_status pond_batch_create(void *stream, pond_batch **out)
{
    if (!out) return POND_EINVAL;
    *out = nullptr;
    pond_batch *b = new pond_batch();
    b->stream = (cudaStream_t)stream;
    if (cudaGetDevice(&b->device) != cudaSuccess ||
        cudaEventCreateWithFlags(&b->done, cudaEventDisableTiming) != cudaSuccess) {
        delete b;
        return POND_ECUDA;
    }
    *out = b;
    return POND_OK;
}

pond_status pond_batch_add(pond_batch *b, pond_ctx *c)
{
    if (!b || !c) return POND_EINVAL;
    b->err.clear();
    if (c->batch) return bfail(b, POND_EINVAL, "context already belongs to a batch");
    if (!c->initialised) return bfail(b, POND_EINVAL, "context state not initialised");
    if (c->nonlocal) return bfail(b, POND_EINVAL, "two-pass (current-time) contexts are stepped alone");
    if (c->lattice == POND_D3Q27) return bfail(b, POND_EINVAL, "D3Q27 contexts are stepped alone");
    if (c->device != b->device) return bfail(b, POND_EINVAL, "context lives on another device");
    // a lone member may exceed the budget, so that no context is refused for ever
    if (b->budget && !b->sims.empty() && b->member_bytes + c->bytes > b->budget)
        return bfail(b, POND_ENOMEM, "the context's " + std::to_string(c->bytes) + " device bytes exceed the batch budget (" +
                                         std::to_string(b->member_bytes) + " of " + std::to_string(b->budget) + " in use)");
    if (cudaSetDevice(b->device) != cudaSuccess) return bfail(b, POND_ECUDA, "cudaSetDevice");
    // the context's queued work (its initialisation) completes before the batch uses it
    if (cudaStreamSynchronize(c->stream) != cudaSuccess) return bfail(b, POND_ECUDA, "cudaStreamSynchronize");
    b->sims.push_back(c);
    b->member_bytes += c->bytes;
    c->batch = b;
    b->dirty = true;
    return POND_OK;
}

pond_status pond_batch_remove(pond_batch *b, pond_ctx *c)
{
    if (!b || !c) return POND_EINVAL;
    auto it = std::find(b->sims.begin(), b->sims.end(), c);
    if (it == b->sims.end()) return bfail(b, POND_EINVAL, "context is not in this batch");
    cudaSetDevice(b->device);
    if (cudaStreamSynchronize(b->stream) != cudaSuccess) return bfail(b, POND_ECUDA, "cudaStreamSynchronize");
    b->sims.erase(it);
    b->member_bytes -= std::min(b->member_bytes, c->bytes);
    c->batch = nullptr;
    b->dirty = true;
    return POND_OK;
}

int32_t pond_batch_size(const pond_batch *b) { return b ? (int32_t)b->sims.size() : 0; }

pond_status pond_batch_set_budget(pond_batch *b, size_t bytes)
{
    if (!b) return POND_EINVAL;
    b->err.clear();
    if (bytes && bytes < b->member_bytes)
        return bfail(b, POND_EINVAL, "budget below the members' current device bytes");
    b->budget = bytes;
    return POND_OK;
}

size_t pond_batch_bytes(const pond_batch *b) { return b ? b->member_bytes : 0; }

pond_status pond_batch_poll(pond_batch *b, int32_t *done)
{
    if (!b || !done) return POND_EINVAL;
    b->err.clear();
    if (cudaSetDevice(b->device) != cudaSuccess) return bfail(b, POND_ECUDA, "cudaSetDevice");
    const cudaError_t e = cudaEventQuery(b->done);
    if (e == cudaSuccess) { *done = 1; return POND_OK; }
    if (e == cudaErrorNotReady) { *done = 0; return POND_OK; }
    return bfail(b, POND_ECUDA, std::string("batch poll: ") + cudaGetErrorString(e));
}

pond_status pond_batch_step(pond_batch *b, int64_t n)
{
    if (!b) return POND_EINVAL;
    b->err.clear();
    if (n < 0) return bfail(b, POND_EINVAL, "negative step count");
    if (cudaSetDevice(b->device) != cudaSuccess) return bfail(b, POND_ECUDA, "cudaSetDevice");
    if (b->sims.empty() || n == 0) return POND_OK;
    if (b->dirty) {
        pond_status st = batch_build(b);
        if (st) return st;
    }
    int64_t k = 0;
    const auto plain = [&](int64_t at) { launch_all(b, (int)(at % 2), 1, [&](int) { return b->stream; }); };
    // whole graph replays from an even step on
    if (b->graph_ok) {
        if (b->since_build % 2) plain(b->since_build + k++);
        for (; k + 2 <= n; k += 2)
            if (cudaGraphLaunch(b->graph, b->stream) != cudaSuccess)
                return bfail(b, POND_ECUDA, "cudaGraphLaunch");
    }
    for (; k < n; ++k) plain(b->since_build + k);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return bfail(b, POND_ECUDA, std::string("batch step: ") + cudaGetErrorString(e));
    b->since_build += n;
    for (pond_ctx *c : b->sims) {
        if (n % 2) c->cur = 1 - c->cur;
        c->steps += n;
    }
    if (cudaEventRecord(b->done, b->stream) != cudaSuccess) return bfail(b, POND_ECUDA, "cudaEventRecord");
    return POND_OK;
}

const char *pond_batch_last_error(const pond_batch *b) { return b ? b->err.c_str() : "null batch"; }

void pond_batch_destroy(pond_batch *b)
{
    if (!b) return;
    cudaSetDevice(b->device);
    cudaStreamSynchronize(b->stream);
    for (pond_ctx *c : b->sims) c->batch = nullptr;
    for (auto &G : b->g) {
        for (int k = 0; k < 2; ++k) cudaFree(G.desc[k]);
        cudaFree(G.work);
    }
    if (b->graph) cudaGraphExecDestroy(b->graph);
    for (int k = 0; k < pond_batch::SIDES; ++k) {
        if (b->join[k]) cudaEventDestroy(b->join[k]);
        if (b->side[k]) cudaStreamDestroy(b->side[k]);
    }
    if (b->fork) cudaEventDestroy(b->fork);
    cudaEventDestroy(b->done);
    delete b;
}

}  // extern "C"
