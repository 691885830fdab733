// Host-side declarations shared by the translation units of the library.
// (CUDA path only; nothing here is shared with the CPU oracle.)
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "../../include/wrffire.h"

namespace wf {

// sticky device status bits (ST_BOUNDS only in libraries built with
// FIRE_BOUNDS_CHECK)
enum { ST_BOUNDARY = 1, ST_NONFINITE = 2, ST_TIMEOUT = 4, ST_BOUNDS = 8 };

// per-class coefficient slots: eq. (spread-WRF-Fire) + T_f + heat factors
enum { K_S0 = 0, K_R0, K_B, K_C, K_D, K_E, K_TF, K_HS, K_HQ, K_N };

// Function attributes (the dynamic shared-memory limit of a kernel) are
// per device: the caches that avoid setting them again are indexed by it.
constexpr int kMaxDevices = 64;

// The device of a context for the length of an entry point: switched to on
// entry when another one is current, switched back on exit (a context's
// stream and buffers belong to the device current at its fire_init).
struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev) {
        int cur = -1;
        if (cudaGetDevice(&cur) == cudaSuccess && cur != dev && cudaSetDevice(dev) == cudaSuccess)
            prev = cur;
    }
    ~DeviceGuard() {
        if (prev >= 0) cudaSetDevice(prev);
    }
    DeviceGuard(const DeviceGuard &) = delete;
    DeviceGuard &operator=(const DeviceGuard &) = delete;
};

// the device a context was created on (context.cu)
int ctx_device(const fire_ctx *c);

// the current device as an index of the attribute caches (-1: none of them)
inline int attr_device() {
    int d = -1;
    if (cudaGetDevice(&d) != cudaSuccess || d < 0 || d >= kMaxDevices) return -1;
    return d;
}

constexpr int kThreadsX = 32;
constexpr int kThreadsY = 8;
constexpr int kThreads = kThreadsX * kThreadsY;
constexpr int kMaxSegPerLaunch = 64;

// Arguments of the fused step kernel.  Element type of the void pointers is
// the path precision T.
struct StepArgs {
    const void *psi_in;
    void *psi_out;
    const void *F_in;
    void *F_out;  // null (warp and tile kernels): psi alone, without F, t_i and heat
    double *tign;
    const uint8_t *fuel;
    const void *dzdx, *dzdy, *mult;
    const void *u, *v;
    const double *coef;  // [ncls][K_N]
    int ncls;
    double *heat_s, *heat_l;  // nullable
    int *status;
    const double *t_in;  // model time at the step start (device scalar)
    double *t_out;       // receives t_in + dt (written by one thread)
    int nx, ny, nxa, nya, srx, sry;
    int kx, ky;  // tile = kx*srx by ky*sry nodes
    int band;
    double dx, dy, eps, dt;
    // per-node coefficients of a per-node fuel moisture, or all null: R0, c,
    // d, H_s, H_q, each [ny][nx] in the path precision (S0, b, e and T_f
    // stay per class)
    const void *nco[5];
    // fuel fraction: 0 the subcell scheme of Sect. 3.3, 1 the scheme exact
    // for linear psi and t_i (2-D tile kernel only)
    int scheme;
    // (host) the launch before on the stream is a kernel whose dependents may
    // start early (launch_chained)
    int chained;
};

// A launch that may start while the kernel before it on the stream still runs
// (programmatic dependent launch): each of these kernels lets its dependents
// start at once (chain_go) and waits for what it depends on itself before it
// touches what a step writes (chain_wait), so that one kernel's launch, its tables
// and the filling of the SMs overlap the end of the one before.  Only for chains of the library's own
// kernels (chained); after anything else the launch is an ordinary one.
template <typename... P, typename... A>
cudaError_t launch_chained(bool chained, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                           cudaStream_t s, const A &...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = chained ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
    if (e != cudaSuccess) cudaGetLastError();  // (the caller reports it; the next call starts without)
    return e;
}

struct IgnSeg {
    double ax, ay, bx, by;
    double rho;      // current radius term: r_g (instantaneous) or S_g (t - t_g)
    double tg, sg;   // start time and growth speed (sg <= 0: instantaneous)
    // drip torch: the step start t and min{t, t_end}; the nearest point at
    // parameter u of [a, b] was laid at tg + u (tlay - tg)
    int drip;
    double tnow, tlay;
    // b - a, and 1/|b - a|^2 (0 for a point); set by apply_ignitions
    double dx, dy, il2;
};

struct IgniteArgs {
    void *psi;
    double *tign;
    int nx, ny;
    double dx, dy;
    int nseg;
    IgnSeg seg[kMaxSegPerLaunch];
};

template <typename T>
size_t step_smem_bytes(int kx, int ky, int srx, int sry, int ncls);

// shared memory of the tile kernel's form with wind tables, 0: a tile too
// large for it
template <typename T>
size_t step_table_bytes(int kx, int ky, int srx, int sry, int ncls);

template <typename T>
cudaError_t launch_step(const StepArgs &a, cudaStream_t s);

template <typename T>
cudaError_t launch_ignite(const IgniteArgs &a, cudaStream_t s);

template <typename T>
cudaError_t launch_fill(void *psi, double *tign, void *frac, size_t n, double psi_far,
                        cudaStream_t s);

template <typename T>
cudaError_t prepare_step_kernel(size_t smem_bytes);

template <typename T>
size_t march_smem_bytes(int ky, int sry, int ncls);

template <typename T>
cudaError_t launch_march(const StepArgs &a, cudaStream_t s);

template <typename T>
cudaError_t prepare_march_kernel(size_t smem_bytes);

constexpr int kMarchMaxColumns = 248;  // output columns of one marching strip (even)

template <typename T>
size_t warp_smem_bytes(int ky, int sry, int ncls);

template <typename T>
cudaError_t launch_warp(const StepArgs &a, cudaStream_t s);

// four columns per lane (FP32 only): strips of <= 120 output columns
constexpr int kWarp4MaxColumns = 120;
cudaError_t launch_warp4(const StepArgs &a, cudaStream_t s);

constexpr int kRowWarps = 4;         // warps of a CTA of the warp kernel, one row each at a time
constexpr int kRowCtasPerSmF32 = 6;  // its resident CTAs per SM that the registers allow
constexpr int kRowCtasPerSmF64 = 2;
constexpr int kTileCtasPerSmF32 = 4;  // and of the tile kernel
constexpr int kTileCtasPerSmF64 = 2;
// atmospheric rows of one CTA of it at most (the wind table of a CTA: at
// refinement 1, where 16 are few, 28 keep the five CTAs per SM of 16 in FP32;
// 8000^2 nodes there, six steps 11.2 ms with 16, 9.8 with 28)
constexpr int row_max_bands(bool fp64, int sry) { return !fp64 && sry == 1 ? 28 : 16; }
// a taller strip is cut into CTAs of that many (the results do not depend on it)
constexpr int row_strip_bands(bool fp64, int ky, int sry) {
    return ky < row_max_bands(fp64, sry) ? ky : row_max_bands(fp64, sry);
}
constexpr int kWarpStrips = 4;       // warps (strips) per CTA of the four-column warp kernel
constexpr int kWarpMaxColumns = 60;  // output columns of one warp strip (even)
constexpr int kWarpMaxRows = 512;    // output rows of one warp strip
// the warp kernel indexes the mesh with 32-bit offsets: nx * ny below 2^31
constexpr long long kWarpMaxNodes = 2147483647LL;

// resident CTAs per SM that default_shape counts on: of the warp strips (four
// strips to a CTA; the rule's own unit, the launch takes warp_launch_rows),
// and of the marching strips (the minimum blocks of their __launch_bounds__,
// checked where the kernels are defined)
constexpr int kWarpCtasPerSmF32 = 3;
constexpr int kMarchCtasPerSmF32 = 5;
constexpr int kMarchCtasPerSmF64 = 2;

// Default launch shape of a single run's step (fire_init and
// fire_step_noalloc).  Strips (warp strips of <= 60 columns in FP32 when the
// refinement allows, else marching strips of <= 248 columns) of the largest
// height up to ~160 rows (warp) / ~60 rows (march) that still gives 3.5
// (warp) / 2.5 (march) waves of resident CTAs on n_sm SMs, else strips one
// atmospheric cell high; where even those fill under a quarter of one wave,
// 2-D tiles of one atmospheric cell; for refinements too large for either
// strip kernel, tiles of ~80x40 (FP32) / 40x40 (FP64) nodes.  The caller
// checks the shape's shared memory and halves tiles that do not fit.
struct DefaultShape {
    int variant, kx, ky;
    bool operator==(const DefaultShape &o) const {
        return variant == o.variant && kx == o.kx && ky == o.ky;
    }
    bool operator!=(const DefaultShape &o) const { return !(*this == o); }
};
DefaultShape default_shape(bool fp64, int nx_atm, int ny_atm, int srx, int sry, int n_sm);

// Atmospheric rows of one CTA of the warp kernel where the caller did not set
// them (fire_init's default and fire_step_noalloc): a CTA of L rows takes
// about L + 10 rows' time (halo rows, tables, the run-in of its stages), and
// the last CTAs to finish leave about 0.8 (L + 20) rows' time of an emptying
// device.  The sum of both over kRowCtasPerSmF32 CTAs per SM is least near
// the measured best: 2000^2 nodes 30 rows (10: 100 us, 30: 64, 60: 69, 160:
// 100), 1000^2 20 rows (10: 32 us, 20: 27, 30: 30), 510^2 10 rows (10: 14.5,
// 20: 20).
// FP64 (two CTAs per SM): 2000^2 nodes 40 rows (10: 1613 us, 20: 1376, 30: 1327,
// 40: 1309, 60: 1350), 1000^2 20 rows (10: 449, 20: 423, 40: 490), 510^2 10
// rows (10: 195, 20: 185, 40: 248).
int warp_launch_rows(bool fp64, int nx, int ny, int W, int sry, int n_sm);

// What launches take in place of the default shape d (fire_init,
// fire_step_noalloc; d is what fire_get_kernel reports, and the results are
// the same bits):
// - warp strips: the rows of warp_launch_rows;
// - FP64 marching strips: the warp kernel's strips, where they are at least
//   kRowMinColumns wide (below, its lanes that hang over cost more than it
//   gains: the time goes with 64 over the width).  us per step, marching and
//   now: 2000^2 nodes 1611 and 1309, 1000^2 565 and 423, 510^2 322 and 185;
// - tiles: of several cells, with tables, where they come out in fewer waves
//   of resident CTAs.  FP64 370x290: 1x1 119 us, 1x2 98, 2x2 94; 200^2: 1x1 64,
//   1x2 49, 2x2 65; 100^2: 1x1 30, 1x2 46.  FP32 370x290: 1x1 21.6, 2x1 14.4,
//   2x2 13.5; 200^2: 1x1 11.4, 2x2 12.4.
DefaultShape launch_shape(bool fp64, const DefaultShape &d, int nx_atm, int ny_atm, int srx, int sry,
                          int ncls, int n_sm, size_t smem_max);
constexpr int kRowMinColumns = 50;

cudaError_t launch_coefficients(const fire_fuel_class *classes_dev, int n, double *coef_dev,
                                cudaStream_t s);
// d(coefficients)/d(M_f) per class at the class moisture (forward-mode dual
// numbers through the same chain)
cudaError_t launch_coefficients_dMf(const fire_fuel_class *classes_dev, int n, double *dcoef_dev,
                                    cudaStream_t s);

// per-node coefficients at a per-node moisture (null: class moisture):
// planes is a host array of device pointers, each [n] in the path precision:
// R0, c, d, H_s, H_q, or (deriv) d/d(M_f) of R0, c, d
template <typename T>
cudaError_t launch_node_coefficients(const fire_fuel_class *classes_dev, int ncls,
                                     const uint8_t *fuel, const void *moist, size_t n,
                                     T *const *planes, bool deriv, cudaStream_t s);

// a fuel class fire_init accepts: a positive weight (burn time), and for a
// Rothermel class with fuel (Table 2) a positive surface-area-to-volume
// ratio, depth, particle density, moisture of extinction and effective
// mineral content (the chain divides by or takes powers of each)
inline bool valid_fuel_class(const fire_fuel_class &f) {
    if (!(f.weight > 0)) return false;
    if (f.fgi > 0 && !f.chaparral &&
        !(f.savr > 0 && f.fueldepthm > 0 && f.fueldens > 0 && f.fuelmce > 0 && f.se > 0))
        return false;
    return true;
}

// remembers the last CUDA error an entry point saw on this host thread
// (read back through fire_last_cuda_error)
void record_cuda_error(cudaError_t e, const char *where);
const char *g_last_error_ptr();

}  // namespace wf
