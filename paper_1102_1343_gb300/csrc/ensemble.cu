// Batched ensemble of independent fire runs (members of different mesh
// sizes, fuels, winds) advanced together by ONE persistent cooperative
// launch per call: its resident CTAs take (member, strip, step) entries from a
// queue, and an entry waits until its member has finished the step before
// (EnsWork).  Each member is an ordinary fire context (same state layout, same
// strip code as fire_step), so a member advanced here matches the same member
// advanced alone.  The launch (with the reset of the queue) is captured in a
// CUDA graph and replayed while its arguments do not change.
//
// Two forms of the persistent kernel, both with one entry per CTA at a time:
// FP32 ensembles run the strip code of k_fire_warp, FP64 ensembles (or
// refinements above 30) that of k_fire_march.
//
// The waits are bounded: a CTA that waits longer than the spin limit sets the
// status bit TIMEOUT and the abort flag, and every CTA leaves the kernel at its
// next entry, so a lost CTA ends the launch with an error status instead of
// hanging the GPU.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

#include "fire_internal.h"
#include "march_kernel.cuh"
#include "warp_kernel.cuh"

using namespace wf;

namespace {

struct EnsItem {
    int member, x0, y0;
    int count;  // items of the member
};

// the queue of a launch (zeroed before it, but for status): entry q is item
// q mod n_items of step q / n_items
struct EnsQueue {
    int status;               // ensemble-wide status bits (TIMEOUT)
    int abort;
    unsigned long long next;  // the first entry not handed out, less the grid
    unsigned long long done[FIRE_MAX_MEMBERS];  // entries finished, per member
};

// values that change from call to call, read by the kernel from device memory
// so that a captured launch can be replayed
struct EnsRun {
    double t0;
    int parity0;
    int nsteps;
    long long spin_limit;
    int skip_block;  // test hook: this CTA reports nothing done and ends (-1: none)
};

struct EnsembleArgs {
    const StepArgs *margs;  // [2 * n_members]: parity 0 and 1 of each member
    const EnsItem *items;
    int n_items;
    int n_members;
    double dt;
    EnsQueue *queue;
    const EnsRun *run;
};

// Work of the persistent kernels.  A step of a member needs the member's step
// before, and nothing of the other members: entries are taken in order, and one
// waits only until its member's entries of the step before are finished.  So
// no step ends with an emptying device (a grid-wide barrier per step did: 24
// members of 26..130 cells square, 40 steps, 13.7 ms; 13.0 so, and 11.7 with
// the taller strips that this allows).  The lowest
// unfinished entry never waits, so the queue always advances; the wait is
// bounded all the same.  Entries are fetched one ahead.
struct EnsWork {
    unsigned long long q;  // current entry
    unsigned long long ahead;  // thread 0: the next one
    int step;
    double t;

    __device__ void start(const EnsRun &run) {
        q = blockIdx.x;
        step = 0;
        t = run.t0;
    }
    // takes the current entry (all threads): false where the launch must end
    __device__ bool take(const EnsembleArgs &e, const EnsRun &run, EnsItem &it) {
        __shared__ int s_ok;
        const unsigned long long total = (unsigned long long)e.n_items * run.nsteps;
        if (q >= total) return false;
        const int s = (int)(q / e.n_items);
        it = e.items[q - (unsigned long long)s * e.n_items];
        for (; step < s; ++step) t = t + e.dt;
        if (threadIdx.x == 0) {
            ahead = gridDim.x + atomicAdd(&e.queue->next, 1ull);
            volatile EnsQueue *v = e.queue;
            const unsigned long long need = (unsigned long long)s * it.count;
            bool ok = v->abort == 0;
            long long polls = 0;
            while (ok && v->done[it.member] < need) {
                if (v->abort) {
                    ok = false;
                    break;
                }
                if (++polls > run.spin_limit) {
                    atomicOr(&e.queue->status, ST_TIMEOUT);
                    atomicExch(&e.queue->abort, 1);
                    ok = false;
                    break;
                }
                __nanosleep(100);
            }
            __threadfence();
            s_ok = ok;
        }
        __syncthreads();
        return s_ok != 0;
    }
    // the entry is finished (all threads): false where the launch must end
    __device__ bool finish(const EnsembleArgs &e, const EnsRun &run, const EnsItem &it) {
        __shared__ unsigned long long s_next;
        __syncthreads();
        if ((int)blockIdx.x == run.skip_block) return false;
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(&e.queue->done[it.member], 1ull);
            s_next = ahead;
        }
        __syncthreads();
        q = s_next;
        return true;
    }
    // the members' device time after the last step
    __device__ void end(const EnsembleArgs &e, const EnsRun &run) {
        if (blockIdx.x != 0 || q < (unsigned long long)e.n_items * run.nsteps) return;
        for (; step < run.nsteps; ++step) t = t + e.dt;
        const int pf = (run.parity0 + run.nsteps) & 1;
        for (int m = threadIdx.x; m < e.n_members; m += blockDim.x)
            *const_cast<double *>(e.margs[2 * m + pf].t_in) = t;
    }
};

template <typename T, bool NC>
__global__ void __launch_bounds__(kMarchThreads, MarchOccupancy<T>::blocks)
    k_fire_ensemble(const EnsembleArgs e) {
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    const EnsRun run = *e.run;
    EnsWork work;
    EnsItem it;
    for (work.start(run); work.take(e, run, it);) {
        const StepArgs &a = e.margs[2 * it.member + ((run.parity0 + work.step) & 1)];
        MarchSmem<T> sm;
        sm.carve(dyn_smem, a.ky * a.sry, a.ncls);
        MarchStrip<T, NC> strip(a, sm);
        strip.run(it.x0, it.y0, work.t);
        if (strip.st) atomicOr(a.status, strip.st);
        if (!work.finish(e, run, it)) break;
    }
    work.end(e, run);
}

// the warp form: the CTA's warps share one item, its member's arguments in
// shared memory.  One CTA per SM fewer than k_fire_warp: at 80 registers this
// kernel spills 176 bytes (8 at 96, 104 where it holds the row loops of even and
// odd widths): 24 members of 26..130 cells square, 40
// steps, 14.35 ms with six CTAs, 13.69 with five (17.8 with the former kernel)
template <typename T, int MODE, int WIDTH>
__global__ void __launch_bounds__(32 * kRowWarps, (row_ctas<T, MODE>()) - 1)
    k_fire_ensemble_warp(const EnsembleArgs e) {
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    __shared__ StepArgs a;
    RowSmem<T, kRowWarps> sm;
    const EnsRun run = *e.run;
    EnsWork work;
    EnsItem it;
    for (work.start(run); work.take(e, run, it);) {
        const int *src = reinterpret_cast<const int *>(e.margs + 2 * it.member + ((run.parity0 + work.step) & 1));
        for (int q = threadIdx.x; q < (int)(sizeof(StepArgs) / sizeof(int)); q += 32 * kRowWarps)
            reinterpret_cast<int *>(&a)[q] = src[q];
        __syncthreads();
        sm.carve(dyn_smem, a.ky, a.sry, a.ncls);
        RowStrip<T, MODE, kRowWarps, WIDTH> strip(a, sm, dyn_smem);
        strip.run(it.x0, it.y0, work.t);  // ends with a barrier
        const int stw = __reduce_or_sync(0xffffffffu, strip.st);
        if ((threadIdx.x & 31) == 0 && stw) atomicOr(a.status, stw);
        if (!work.finish(e, run, it)) break;
    }
    work.end(e, run);
}

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

// members are ordinary contexts: the accessors below are defined in context.cu
namespace wf {
int ctx_step_args(fire_ctx *c, int parity, const void *u, const void *v, double dt, double *hs,
                  double *hl, StepArgs &a);
int ctx_info(const fire_ctx *c, int *prec, int *variant, int *nx, int *ny, int *srx, int *sry,
             int *kx, int *ky, int *ncls, int *cur, double *t);
int ctx_advance(fire_ctx *c, int nsteps, double dt);
bool ctx_ignition_active(fire_ctx *c, double t);
cudaStream_t ctx_stream(const fire_ctx *c);
int ctx_workspace(fire_ctx *c, size_t bytes, void **out);
int ctx_default_march(fire_ctx *c);
int ctx_default_warp_strips(fire_ctx *c, int rows);
int ctx_ensure_node_coefficients(fire_ctx *c);
bool ctx_has_node_coefficients(const fire_ctx *c);
}  // namespace wf

struct fire_ensemble {
    std::vector<fire_ctx *> members;
    int n = 0;
    int device = 0;  // the device current at fire_ensemble_create (its members')
    int prec = FIRE_FP32;
    cudaStream_t stream = nullptr;
    StepArgs *margs_dev = nullptr;
    StepArgs *margs_host = nullptr;  // pinned
    EnsItem *items_dev = nullptr;
    int n_items = 0;
    EnsQueue *queue = nullptr;
    EnsRun *run_dev = nullptr;
    EnsRun *run_host = nullptr;  // pinned
    cudaEvent_t staged = nullptr;  // the pinned staging buffers may be rewritten
    int grid = 0;
    size_t smem = 0;
    long long spin_limit = 20000000;  // x ~100 ns: about 2 s
    int skip_block = -1;
    cudaGraphExec_t graph = nullptr;
    bool capture_failed = false;
    int variant = FIRE_KERNEL_MARCH;  // member kernel: FIRE_KERNEL_MARCH or FIRE_KERNEL_WARP
    int strip_cols = 0, strip_rows = 0;  // nodes of the members' strips, as set or by default
    bool even = true;  // every member's mesh has an even width
    bool nc = false;  // members carry per-node coefficients (a per-node fuel moisture)
    int g_nsteps = -1;
    double g_dt = 0;
    int g_grid = 0;
    size_t g_smem = 0;
};

namespace {

int ens_cuda_at(cudaError_t e, const char *where) {
    if (e == cudaSuccess) return FIRE_OK;
    record_cuda_error(e, where);
    cudaGetLastError();  // reported here: the next call starts without it
    return e == cudaErrorMemoryAllocation ? FIRE_ERR_OOM : FIRE_ERR_CUDA;
}

#define ens_cuda(call) ens_cuda_at((call), #call)
#define ENS_CHECK(call)                   \
    do {                                  \
        int _r = ens_cuda(call);          \
        if (_r != FIRE_OK) return _r;     \
    } while (0)

void ens_release(fire_ensemble *e) {
    if (!e) return;
    if (e->graph) cudaGraphExecDestroy(e->graph);
    if (e->staged) cudaEventDestroy(e->staged);
    for (fire_ctx *c : e->members) fire_destroy(c);
    if (e->margs_dev) cudaFree(e->margs_dev);
    if (e->items_dev) cudaFree(e->items_dev);
    if (e->queue) cudaFree(e->queue);
    if (e->run_dev) cudaFree(e->run_dev);
    if (e->margs_host) cudaFreeHost(e->margs_host);
    if (e->run_host) cudaFreeHost(e->run_host);
    delete e;
}

// the warp form's kernel (FP32 only)
const void *ens_warp_kernel(const fire_ensemble *e) {
    const bool w = e->even;
    if (e->nc)
        return w ? (const void *)k_fire_ensemble_warp<float, ROW_NC, WIDTH_EVEN>
                 : (const void *)k_fire_ensemble_warp<float, ROW_NC, WIDTH_ANY>;
    return w ? (const void *)k_fire_ensemble_warp<float, ROW_MULT, WIDTH_EVEN>
             : (const void *)k_fire_ensemble_warp<float, ROW_MULT, WIDTH_ANY>;
}

// work list and launch shape for the members' current kernel configuration
int ens_plan(fire_ensemble *e) {
    // a captured launch holds the old work list (pointer and length): drop
    // it, after the stream has finished with it, before the list is replaced
    ENS_CHECK(cudaStreamSynchronize(e->stream));
    if (e->graph) {
        cudaGraphExecDestroy(e->graph);
        e->graph = nullptr;
    }
    // a member's items one after the other, the largest member first
    std::vector<std::vector<EnsItem>> of(e->n);
    size_t smem = 0;
    for (int m = 0; m < e->n; ++m) {
        int prec, variant, nx, ny, srx, sry, kx, ky, ncls, cur;
        double t;
        ctx_info(e->members[m], &prec, &variant, &nx, &ny, &srx, &sry, &kx, &ky, &ncls, &cur, &t);
        if (variant != e->variant) return FIRE_ERR_STATE;
        if (e->variant == FIRE_KERNEL_WARP) ky = row_strip_bands(e->prec == FIRE_FP64, ky, sry);
        const int W = kx * srx, L = ky * sry;
        const int count = ((nx + W - 1) / W) * ((ny + L - 1) / L);
        for (int y0 = 0; y0 < ny; y0 += L)
            for (int x0 = 0; x0 < nx; x0 += W) of[m].push_back(EnsItem{m, x0, y0, count});
        if (e->variant == FIRE_KERNEL_MARCH) {
            const size_t sm = e->prec == FIRE_FP64 ? march_smem_bytes<double>(ky, sry, ncls)
                                                   : march_smem_bytes<float>(ky, sry, ncls);
            smem = std::max(smem, sm);
        } else {
            const size_t sm = e->prec == FIRE_FP64 ? warp_smem_bytes<double>(ky, sry, ncls)
                                                   : warp_smem_bytes<float>(ky, sry, ncls);
            smem = std::max(smem, sm);
        }
    }
    std::stable_sort(of.begin(), of.end(), [](const std::vector<EnsItem> &a, const std::vector<EnsItem> &b) {
        return a.size() > b.size();
    });
    std::vector<EnsItem> items;
    for (const std::vector<EnsItem> &o : of) items.insert(items.end(), o.begin(), o.end());
    if (e->items_dev) cudaFree(e->items_dev);
    e->items_dev = nullptr;
    ENS_CHECK(cudaMalloc(&e->items_dev, sizeof(EnsItem) * items.size()));
    ENS_CHECK(cudaMemcpy(e->items_dev, items.data(), sizeof(EnsItem) * items.size(),
                         cudaMemcpyHostToDevice));
    e->n_items = (int)items.size();
    const void *fn;
    int threads;
    const bool f64 = e->prec == FIRE_FP64;
    if (e->variant == FIRE_KERNEL_WARP) {
        fn = ens_warp_kernel(e);
        threads = 32 * kRowWarps;
    } else {
        fn = e->nc ? (f64 ? (const void *)k_fire_ensemble<double, true>
                          : (const void *)k_fire_ensemble<float, true>)
                   : (f64 ? (const void *)k_fire_ensemble<double, false>
                          : (const void *)k_fire_ensemble<float, false>);
        threads = kMarchThreads;
    }
    {
        // the limit is a property of the kernel function on a device, shared by
        // all ensembles there: one slot per function (the parity of the mesh
        // widths selects one in the warp form alone)
        static std::mutex mu;
        static size_t current[kMaxDevices][16] = {};
        std::lock_guard<std::mutex> lock(mu);
        const int dev = attr_device();
        const bool warp = e->variant == FIRE_KERNEL_WARP;
        const int form = (f64 ? 1 : 0) + (warp ? 2 : 0) + (e->nc ? 4 : 0) + (warp && e->even ? 8 : 0);
        if (dev < 0 || smem > current[dev][form]) {
            ENS_CHECK(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            if (dev >= 0) current[dev][form] = smem;
        }
    }
    int per_sm = 0, dev = 0, sms = 0;
    ENS_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem));
    ENS_CHECK(cudaGetDevice(&dev));
    ENS_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (per_sm < 1) return FIRE_ERR_ARG;
    e->grid = std::min(e->n_items, per_sm * sms);
    e->smem = smem;
    return FIRE_OK;
}

cudaError_t ens_launch(fire_ensemble *e, double dt, cudaStream_t s) {
    EnsembleArgs ea;
    ea.margs = e->margs_dev;
    ea.items = e->items_dev;
    ea.n_items = e->n_items;
    ea.n_members = e->n;
    ea.dt = dt;
    ea.queue = e->queue;
    ea.run = e->run_dev;
    cudaError_t err = cudaMemsetAsync(&e->queue->abort, 0, sizeof(EnsQueue) - offsetof(EnsQueue, abort), s);
    if (err != cudaSuccess) return err;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3(e->grid);
    cfg.blockDim = dim3(e->variant == FIRE_KERNEL_WARP ? 32 * kRowWarps : kMarchThreads);
    cfg.dynamicSmemBytes = e->smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const bool f64 = e->prec == FIRE_FP64;
    if (e->variant == FIRE_KERNEL_WARP) {
        void *args[] = {&ea};
        return cudaLaunchKernelExC(&cfg, ens_warp_kernel(e), args);
    }
    if (e->nc)
        return f64 ? cudaLaunchKernelEx(&cfg, k_fire_ensemble<double, true>, ea)
                   : cudaLaunchKernelEx(&cfg, k_fire_ensemble<float, true>, ea);
    return f64 ? cudaLaunchKernelEx(&cfg, k_fire_ensemble<double, false>, ea)
               : cudaLaunchKernelEx(&cfg, k_fire_ensemble<float, false>, ea);
}

}  // namespace

extern "C" {

int fire_ensemble_create(fire_ensemble **out, int n_members, const fire_member_desc *members,
                         void *cuda_stream) {
    if (!out) return FIRE_ERR_ARG;
    *out = nullptr;
    if (n_members < 1 || n_members > FIRE_MAX_MEMBERS || !members) return FIRE_ERR_ARG;
    const int prec = members[0].grid.precision;
    for (int m = 0; m < n_members; ++m)
        if (members[m].grid.precision != prec) return FIRE_ERR_ARG;
    fire_ensemble *e = new (std::nothrow) fire_ensemble();
    if (!e) return FIRE_ERR_OOM;
    e->n = n_members;
    e->prec = prec;
    if (cudaGetDevice(&e->device) != cudaSuccess) {
        delete e;
        return FIRE_ERR_CUDA;
    }
    e->stream = static_cast<cudaStream_t>(cuda_stream);
    int r = FIRE_OK;
    for (int m = 0; m < n_members && r == FIRE_OK; ++m) {
        const fire_member_desc &d = members[m];
        fire_ctx *c = nullptr;
        r = fire_init(&c, &d.grid, d.classes, d.n_classes, d.fuel_class_dev, d.moisture_dev,
                      d.spread_mult_dev, d.dzdx_dev, d.dzdy_dev, d.ignitions, d.n_ign, cuda_stream);
        if (r == FIRE_OK) e->members.push_back(c);
    }
    // one member with a per-node moisture: every member takes the per-node
    // coefficient form of the kernel (the others' planes from their classes)
    if (r == FIRE_OK) {
        for (fire_ctx *c : e->members) e->nc = e->nc || ctx_has_node_coefficients(c);
        if (e->nc)
            for (fire_ctx *c : e->members)
                if (r == FIRE_OK) r = ctx_ensure_node_coefficients(c);
    }
    // the warp form when every member can take warp strips (FP32, refinement
    // <= 30), else the marching form for all; members start from marching
    // strips of the large-mesh size, or from warp strips whose height suits
    // the whole ensemble.  A step costs its items times L + 23 rows' time over
    // the resident CTAs, and, where the largest member's next step follows
    // within a wave or two, waits of up to 0.8 (L + 20).  Measured, ms per 40
    // steps: 24 members of 26..130 cells square, rows 60: 13.0, 80: 12.4, 120:
    // 11.7 (taken), 160: 11.4; 60 members of 26..40, rows 40: 8.3, 60: 7.6
    // (taken), 80: 7.2, 120: 7.4; 3 members of 100..130, rows 30: 3.4, 40: 3.1
    // (taken), 60: 3.1, 80: 3.5.
    if (r == FIRE_OK) {
        bool warp = prec == FIRE_FP32;
        for (fire_ctx *c : e->members) {
            int prc, variant, nx, ny, srx, sry, kx, ky, ncls, cur;
            double t;
            ctx_info(c, &prc, &variant, &nx, &ny, &srx, &sry, &kx, &ky, &ncls, &cur, &t);
            e->even = e->even && (nx & 1) == 0;
            warp = warp && srx <= kWarpMaxColumns / 2 && (long long)nx * ny <= kWarpMaxNodes;
        }
        e->variant = warp ? FIRE_KERNEL_WARP : FIRE_KERNEL_MARCH;
        int rows = 10, n_sm = 1;
        double least = 0;
        r = ens_cuda(cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, e->device));
        const double slots = (double)n_sm * (kRowCtasPerSmF32 - 1);
        for (int L = 10; L <= 160; L += 10) {
            double all = 0, most = 0;
            for (fire_ctx *c : e->members) {
                int nx = 0, ny = 0;
                fire_mesh_size(c, &nx, &ny);
                const double own =
                    (double)((nx + kWarpMaxColumns - 1) / kWarpMaxColumns) * ((ny + L - 1) / L);
                all += own;
                most = std::max(most, own);
            }
            const double between = (all - most) / slots;  // waves from a member's step to its next
            const double wait = std::min(0.8, std::max(0.0, 0.8 - 0.4 * (between - 1.0)));
            const double t = all * (L + 23) / slots + wait * (L + 20);
            if (L == 10 || t < least) {
                least = t;
                rows = L;
            }
        }
        e->strip_cols = warp ? kWarpMaxColumns : kMarchMaxColumns;
        e->strip_rows = warp ? rows : 60;
        for (fire_ctx *c : e->members)
            if (r == FIRE_OK && (warp ? ctx_default_warp_strips(c, rows) : ctx_default_march(c)) != FIRE_OK)
                r = FIRE_ERR_ARG;
    }
#define ENS_TRY(call)                 \
    do {                              \
        if (r == FIRE_OK) r = ens_cuda(call); \
    } while (0)
    ENS_TRY(cudaMalloc(&e->margs_dev, sizeof(StepArgs) * 2 * n_members));
    ENS_TRY(cudaMallocHost(&e->margs_host, sizeof(StepArgs) * 2 * n_members));
    ENS_TRY(cudaMalloc(&e->queue, sizeof(EnsQueue)));
    ENS_TRY(cudaMalloc(&e->run_dev, sizeof(EnsRun)));
    ENS_TRY(cudaMallocHost(&e->run_host, sizeof(EnsRun)));
    ENS_TRY(cudaEventCreateWithFlags(&e->staged, cudaEventDisableTiming));
    ENS_TRY(cudaMemsetAsync(e->queue, 0, sizeof(EnsQueue), e->stream));
#undef ENS_TRY
    if (r == FIRE_OK) r = ens_plan(e);
    if (r == FIRE_OK) r = ens_cuda(cudaStreamSynchronize(e->stream));
    if (r != FIRE_OK) {
        ens_release(e);
        return r;
    }
    *out = e;
    return FIRE_OK;
}

int fire_ensemble_step(fire_ensemble *e, int nsteps, double dt, const void *const *wind_u_dev,
                       const void *const *wind_v_dev, double *const *heat_sens_dev,
                       double *const *heat_lat_dev) {
    if (!e || nsteps < 0 || !isfinite(dt) || !(dt > 0) || !wind_u_dev || !wind_v_dev)
        return FIRE_ERR_ARG;
    for (int m = 0; m < e->n; ++m)
        if (!wind_u_dev[m] || !wind_v_dev[m]) return FIRE_ERR_ARG;
    DeviceGuard dg(e->device);
    int done = 0;
    while (done < nsteps) {
        // an active ignition window needs its own step (fire_step applies it)
        bool ign = false;
        for (int m = 0; m < e->n; ++m) {
            int prec, variant, nx, ny, srx, sry, kx, ky, ncls, cur;
            double t;
            ctx_info(e->members[m], &prec, &variant, &nx, &ny, &srx, &sry, &kx, &ky, &ncls, &cur, &t);
            if (ctx_ignition_active(e->members[m], t)) ign = true;
        }
        if (ign) {
            for (int m = 0; m < e->n; ++m) {
                int r = fire_step(e->members[m], wind_u_dev[m], wind_v_dev[m], dt,
                                  heat_sens_dev ? heat_sens_dev[m] : nullptr,
                                  heat_lat_dev ? heat_lat_dev[m] : nullptr);
                if (r) return r;
            }
            ++done;
            continue;
        }
        // the rest (up to the next ignition window) in one persistent launch
        int chunk = 0;
        {
            int prec, variant, nx, ny, srx, sry, kx, ky, ncls, cur;
            double t0;
            ctx_info(e->members[0], &prec, &variant, &nx, &ny, &srx, &sry, &kx, &ky, &ncls, &cur, &t0);
            double t = t0;
            while (done + chunk < nsteps) {
                bool any = false;
                for (int m = 0; m < e->n && !any; ++m) any = ctx_ignition_active(e->members[m], t);
                if (any) break;
                t = t + dt;
                ++chunk;
            }
            ENS_CHECK(cudaEventSynchronize(e->staged));
            for (int m = 0; m < e->n; ++m) {
                for (int p = 0; p < 2; ++p) {
                    int r = ctx_step_args(e->members[m], p, wind_u_dev[m], wind_v_dev[m], dt,
                                          heat_sens_dev ? heat_sens_dev[m] : nullptr,
                                          heat_lat_dev ? heat_lat_dev[m] : nullptr,
                                          e->margs_host[2 * m + p]);
                    if (r) return r;
                    StepArgs &ma = e->margs_host[2 * m + p];
                    if (e->variant == FIRE_KERNEL_WARP) ma.ky = row_strip_bands(e->prec == FIRE_FP64, ma.ky, ma.sry);
                }
            }
            e->run_host->t0 = t0;
            e->run_host->parity0 = cur;
            e->run_host->nsteps = chunk;
            e->run_host->spin_limit = e->spin_limit;
            e->run_host->skip_block = e->skip_block;
        }
        ENS_CHECK(cudaMemcpyAsync(e->margs_dev, e->margs_host, sizeof(StepArgs) * 2 * e->n,
                                  cudaMemcpyHostToDevice, e->stream));
        ENS_CHECK(cudaMemcpyAsync(e->run_dev, e->run_host, sizeof(EnsRun), cudaMemcpyHostToDevice,
                                  e->stream));
        ENS_CHECK(cudaEventRecord(e->staged, e->stream));
        // replay the captured launch when its shape is unchanged
        if (!e->capture_failed && (!e->graph || e->g_nsteps != chunk || e->g_dt != dt ||
                                   e->g_grid != e->grid || e->g_smem != e->smem)) {
            if (e->graph) {
                ENS_CHECK(cudaStreamSynchronize(e->stream));  // the old graph may be in flight
                cudaGraphExecDestroy(e->graph);
                e->graph = nullptr;
            }
            cudaStream_t cs;
            ENS_CHECK(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
            cudaGraph_t gr = nullptr;
            cudaError_t err = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
            if (err == cudaSuccess) {
                err = ens_launch(e, dt, cs);
                cudaError_t e2 = cudaStreamEndCapture(cs, &gr);
                if (err == cudaSuccess) err = e2;
            }
            if (err == cudaSuccess) err = cudaGraphInstantiate(&e->graph, gr, 0);
            if (gr) cudaGraphDestroy(gr);
            cudaStreamDestroy(cs);
            if (err != cudaSuccess) {
                // capture of the cooperative launch refused: launch directly
                record_cuda_error(err, "capture of the ensemble launch");
                cudaGetLastError();
                e->graph = nullptr;
                e->capture_failed = true;
            } else {
                e->g_nsteps = chunk;
                e->g_dt = dt;
                e->g_grid = e->grid;
                e->g_smem = e->smem;
            }
        }
        if (e->graph) ENS_CHECK(cudaGraphLaunch(e->graph, e->stream));
        else ENS_CHECK(ens_launch(e, dt, e->stream));
        for (int m = 0; m < e->n; ++m) ctx_advance(e->members[m], chunk, dt);
        done += chunk;
    }
    return FIRE_OK;
}

int fire_ensemble_member(fire_ensemble *e, int member, fire_ctx **ctx) {
    if (!e || !ctx || member < 0 || member >= e->n) return FIRE_ERR_ARG;
    *ctx = e->members[member];
    return FIRE_OK;
}

int fire_ensemble_status(fire_ensemble *e, int *member_status) {
    if (!e) return FIRE_ERR_ARG;
    DeviceGuard dg(e->device);
    ENS_CHECK(cudaStreamSynchronize(e->stream));
    int ens_status = 0;
    ENS_CHECK(cudaMemcpy(&ens_status, &e->queue->status, sizeof ens_status, cudaMemcpyDeviceToHost));
    int worst = FIRE_OK;
    for (int m = 0; m < e->n; ++m) {
        const int s = fire_status(e->members[m]);
        if (member_status) member_status[m] = s;
        if (s != FIRE_OK && worst != FIRE_ERR_BOUNDS &&
            (worst == FIRE_OK || s == FIRE_ERR_NONFINITE || s == FIRE_ERR_BOUNDS))
            worst = s;
    }
    if (ens_status & ST_TIMEOUT) return FIRE_ERR_TIMEOUT;
    return worst;
}

int fire_ensemble_clear_status(fire_ensemble *e) {
    if (!e) return FIRE_ERR_ARG;
    for (fire_ctx *c : e->members) {
        int r = fire_clear_status(c);
        if (r) return r;
    }
    ENS_CHECK(cudaMemsetAsync(e->queue, 0, sizeof(EnsQueue), e->stream));
    return FIRE_OK;
}

int fire_ensemble_set_kernel(fire_ensemble *e, int strip_columns, int strip_rows) {
    if (!e || strip_columns < 2 || strip_rows < 1) return FIRE_ERR_ARG;
    DeviceGuard dg(e->device);
    for (fire_ctx *c : e->members) {
        int prec, variant, nx, ny, srx, sry, kx, ky, ncls, cur;
        double t;
        ctx_info(c, &prec, &variant, &nx, &ny, &srx, &sry, &kx, &ky, &ncls, &cur, &t);
        const int maxw = e->variant == FIRE_KERNEL_WARP ? kWarpMaxColumns : kMarchMaxColumns;
        int kxn = std::max(1, std::min(strip_columns, maxw) / srx);
        int kyn = std::max(1, strip_rows / sry);
        if ((kxn * srx) & 1) kxn = kxn > 1 ? kxn - 1 : 2;
        if (e->variant == FIRE_KERNEL_WARP && kyn * sry > kWarpMaxRows) kyn = kWarpMaxRows / sry;
        int r = fire_set_kernel(c, e->variant, kxn, kyn);
        if (r) return r;
    }
    e->strip_cols = strip_columns;
    e->strip_rows = strip_rows;
    return ens_plan(e);
}

// Times strip shapes (columns x rows of fire nodes) of the persistent
// launch: every candidate starts from the members' saved states, runs one
// untimed call (which also captures its graph) and one timed call of
// probe_steps steps; the fastest is kept and the states are put back.
int fire_ensemble_autotune(fire_ensemble *e, int probe_steps, double dt,
                           const void *const *wind_u_dev, const void *const *wind_v_dev,
                           int *strip_columns, int *strip_rows) {
    if (!e || probe_steps < 1 || !isfinite(dt) || !(dt > 0) || !wind_u_dev || !wind_v_dev)
        return FIRE_ERR_ARG;
    DeviceGuard dg(e->device);
    // the probe must not cross an ignition window (it would apply it)
    std::vector<double> t0(e->n);
    for (int m = 0; m < e->n; ++m) {
        int prec, variant, nx, ny, srx, sry, kx, ky, ncls, cur;
        ctx_info(e->members[m], &prec, &variant, &nx, &ny, &srx, &sry, &kx, &ky, &ncls, &cur,
                 &t0[m]);
        double t = t0[m];
        for (int k = 0; k <= 2 * probe_steps; ++k) {
            if (ctx_ignition_active(e->members[m], t)) return FIRE_ERR_STATE;
            t = t + dt;
        }
    }
    // save the states in the members' workspaces
    const size_t E = e->prec == FIRE_FP64 ? 8 : 4;
    std::vector<unsigned char *> saved(e->n);
    std::vector<size_t> nn(e->n);
    for (int m = 0; m < e->n; ++m) {
        int nx = 0, ny = 0;
        fire_mesh_size(e->members[m], &nx, &ny);
        nn[m] = (size_t)nx * ny;
        void *w = nullptr;
        int r = ctx_workspace(e->members[m], nn[m] * (2 * E + sizeof(double)), &w);
        if (r) return r;
        saved[m] = static_cast<unsigned char *>(w);
        r = fire_get_state(e->members[m], saved[m], reinterpret_cast<double *>(saved[m] + 2 * nn[m] * E),
                           saved[m] + nn[m] * E, nullptr);
        if (r) return r;
    }
    auto restore = [&]() {
        for (int m = 0; m < e->n; ++m) {
            int r = fire_set_state(e->members[m], saved[m],
                                   reinterpret_cast<double *>(saved[m] + 2 * nn[m] * E),
                                   saved[m] + nn[m] * E, t0[m]);
            if (r) return r;
        }
        return (int)FIRE_OK;
    };
    const int cols_m[] = {40, 80, 120, 160, 200, 240}, rows_m[] = {20, 40, 80, 160, 320};
    const int cols_w[] = {20, 30, 40, 50, 60, 60}, rows_w[] = {20, 40, 80, 160, 320};
    const bool wv = e->variant == FIRE_KERNEL_WARP;
    const int *cols = wv ? cols_w : cols_m, *rows = wv ? rows_w : rows_m;
    // the strips in place first (20 rows where they are shorter, the least that
    // is reported)
    std::vector<std::pair<int, int>> cands = {{std::min(e->strip_cols, 240), std::max(e->strip_rows, 20)}};
    for (int ci = 0; ci < 6; ++ci)
        for (int ri = 0; ri < 5; ++ri) {
            const std::pair<int, int> q{cols[ci], rows[ri]};
            if (std::find(cands.begin(), cands.end(), q) == cands.end()) cands.push_back(q);
        }
    cudaEvent_t a, b;
    ENS_CHECK(cudaEventCreate(&a));
    ENS_CHECK(cudaEventCreate(&b));
    float best = 0.f;
    int bc = 0, br = 0;
    int r = FIRE_OK;
    for (const std::pair<int, int> &q : cands) {
        if (fire_ensemble_set_kernel(e, q.first, q.second) != FIRE_OK) continue;
        if ((r = restore())) break;
        if ((r = fire_ensemble_step(e, probe_steps, dt, wind_u_dev, wind_v_dev, nullptr, nullptr))) break;
        if ((r = restore())) break;
        if ((r = ens_cuda(cudaEventRecord(a, e->stream)))) break;
        if ((r = fire_ensemble_step(e, probe_steps, dt, wind_u_dev, wind_v_dev, nullptr, nullptr))) break;
        if ((r = ens_cuda(cudaEventRecord(b, e->stream)))) break;
        if ((r = ens_cuda(cudaEventSynchronize(b)))) break;
        float ms = 0.f;
        if ((r = ens_cuda(cudaEventElapsedTime(&ms, a, b)))) break;
        if (bc == 0 || ms < best) {
            best = ms;
            bc = q.first;
            br = q.second;
        }
    }
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    if (r) return r;
    if (bc == 0) return FIRE_ERR_ARG;
    r = fire_ensemble_set_kernel(e, bc, br);
    if (r) return r;
    r = restore();
    if (r) return r;
    if (strip_columns) *strip_columns = bc;
    if (strip_rows) *strip_rows = br;
    return FIRE_OK;
}

int fire_ensemble_get_kernel(const fire_ensemble *e, int *grid_ctas, int *work_items) {
    if (!e) return FIRE_ERR_ARG;
    if (grid_ctas) *grid_ctas = e->grid;
    if (work_items) *work_items = e->n_items;
    return FIRE_OK;
}

int fire_ensemble_set_barrier_test(fire_ensemble *e, int skip_block, long long spin_limit) {
    if (!e || spin_limit < 1) return FIRE_ERR_ARG;
    e->skip_block = skip_block;
    e->spin_limit = spin_limit;
    return FIRE_OK;
}

void fire_ensemble_destroy(fire_ensemble *e) {
    if (!e) return;
    DeviceGuard dg(e->device);
    cudaStreamSynchronize(e->stream);
    ens_release(e);
}

}  // extern "C"
