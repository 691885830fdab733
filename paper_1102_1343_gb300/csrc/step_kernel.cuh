// Fused fire-step kernel (Sect. 5 items 2-6 of the paper) and the
// element-wise ignition / initialisation kernels, templated on the path
// precision T (float or double).  Included by step_f32.cu and step_f64.cu.
//
// One CTA owns a tile of kx x ky atmospheric cells = TX x TY fire nodes
// (TX = kx*srx, TY = ky*sry), so every atmospheric cell's heat average is
// reduced inside one CTA, deterministically.  The CTA stages the level-set
// function psi^n of its tile plus a 3-node halo in shared memory and runs
// the whole step there:
//   stage 1 (eq. Heun, first line)  on the tile + 2 halo -> psi*
//   stage 2 (eq. Heun, second line) on the tile + 1 halo -> psi^{n+1}
//   ignition-time crossing (eq. set-ignition-time) on the tile + 1 halo
//   fuel-fraction quadrature (Sect. 3.3) on the tile, which needs psi^{n+1}
//   and the compatible ignition time on the 3x3 neighbourhood
//   heat fluxes (eqs. sensible-/latent-heat-flux) and their average over the
//   tile's atmospheric cells (Sect. 5, item 6)
// The halo is recomputed redundantly by neighbouring CTAs, so one step costs
// one pass over the state in HBM.  Ghost nodes beyond the domain follow the
// extrapolation of Sect. 3.1 (x first, then y), recomputed for each stage.
#pragma once

#include <cuda_runtime.h>
#include <mutex>
#include <math.h>
#include <stdint.h>

#include "fire_device.cuh"
#include "fire_internal.h"

namespace wf {

// Fill the ghost ring of a staged field whose local (0,0) is the global node
// (ox, oy): x-ghost columns for the domain rows, then y-ghost rows over the
// extended columns (corners).  Block-uniform: all threads must call it.
template <typename T>
__device__ void fill_ghosts(T *B, int BW, int BH, int ox, int oy, int nx, int ny, int tid) {
    const int lxl = -1 - ox, lxr = nx - ox;
    const bool hasL = lxl >= 0 && lxl + 2 < BW, hasR = lxr - 2 >= 0 && lxr < BW;
    for (int ly = tid; ly < BH; ly += kThreads) {
        int gy = oy + ly;
        if (gy < 0 || gy >= ny) continue;
        T *row = B + ly * BW;
        if (hasL) row[lxl] = ghost_value<T>(row[lxl + 1], row[lxl + 2]);
        if (hasR) row[lxr] = ghost_value<T>(row[lxr - 1], row[lxr - 2]);
    }
    __syncthreads();
    const int lyb = -1 - oy, lyt = ny - oy;
    const bool hasB = lyb >= 0 && lyb + 2 < BH, hasT = lyt - 2 >= 0 && lyt < BH;
    for (int lx = tid; lx < BW; lx += kThreads) {
        int gx = ox + lx;
        if (gx < -1 || gx > nx) continue;
        if (hasB) B[lyb * BW + lx] = ghost_value<T>(B[(lyb + 1) * BW + lx], B[(lyb + 2) * BW + lx]);
        if (hasT) B[lyt * BW + lx] = ghost_value<T>(B[(lyt - 1) * BW + lx], B[(lyt - 2) * BW + lx]);
    }
    __syncthreads();
}

// Ghosts of psi^{n+1} (as fill_ghosts) and of Dl = t - t_i (compatible
// ignition time): a ghost copies its inner neighbour's value, then is 0
// where the ghost psi >= 0 (eq. ti-comp).
template <typename T>
__device__ void fill_ghosts_pd(T *P, T *Dl, int BW, int BH, int ox, int oy, int nx, int ny,
                               int tid) {
    const int lxl = -1 - ox, lxr = nx - ox;
    const bool hasL = lxl >= 0 && lxl + 2 < BW, hasR = lxr - 2 >= 0 && lxr < BW;
    for (int ly = tid; ly < BH; ly += kThreads) {
        int gy = oy + ly;
        if (gy < 0 || gy >= ny) continue;
        T *row = P + ly * BW;
        T *drow = Dl + ly * BW;
        if (hasL) {
            T g = ghost_value<T>(row[lxl + 1], row[lxl + 2]);
            row[lxl] = g;
            drow[lxl] = g >= T(0) ? T(0) : drow[lxl + 1];
        }
        if (hasR) {
            T g = ghost_value<T>(row[lxr - 1], row[lxr - 2]);
            row[lxr] = g;
            drow[lxr] = g >= T(0) ? T(0) : drow[lxr - 1];
        }
    }
    __syncthreads();
    const int lyb = -1 - oy, lyt = ny - oy;
    const bool hasB = lyb >= 0 && lyb + 2 < BH, hasT = lyt - 2 >= 0 && lyt < BH;
    for (int lx = tid; lx < BW; lx += kThreads) {
        int gx = ox + lx;
        if (gx < -1 || gx > nx) continue;
        if (hasB) {
            T g = ghost_value<T>(P[(lyb + 1) * BW + lx], P[(lyb + 2) * BW + lx]);
            P[lyb * BW + lx] = g;
            Dl[lyb * BW + lx] = g >= T(0) ? T(0) : Dl[(lyb + 1) * BW + lx];
        }
        if (hasT) {
            T g = ghost_value<T>(P[(lyt - 1) * BW + lx], P[(lyt - 2) * BW + lx]);
            P[lyt * BW + lx] = g;
            Dl[lyt * BW + lx] = g >= T(0) ? T(0) : Dl[(lyt - 1) * BW + lx];
        }
    }
    __syncthreads();
}

// Fuel fraction of the cell at index c of the staged psi^{n+1} (P) and
// Dl = t - t_i (row pitch W).
template <typename T>
__device__ __forceinline__ T cell_fraction(const T *P, const T *Dl, int c, int W, T Tf) {
    return cell_fraction_vals<T>(P[c - W - 1], P[c - W], P[c - W + 1], P[c - 1], P[c], P[c + 1],
                                 P[c + W - 1], P[c + W], P[c + W + 1], Dl[c - W - 1], Dl[c - W],
                                 Dl[c - W + 1], Dl[c - 1], Dl[c], Dl[c + 1], Dl[c + W - 1],
                                 Dl[c + W], Dl[c + W + 1], Tf);
}

template <typename T>
__host__ __device__ inline int lut_slots(int ncls) {
    int n = ncls * K_N;
    return (n + 3) & ~3;
}

// largest shared memory of the tile kernel's form with wind tables
constexpr size_t kTileTabBytes = 56 * 1024;

// wind rows of a tile's table: its atmospheric rows and those around them
__host__ __device__ inline int tile_wind_rows(int ky) { return ky + 5; }

// shared memory of a tile of TX x TY nodes, in elements of T: the class
// table, psi^n (halo 3), psi* (halo 2), F(psi^n), psi^{n+1} and t - t_i
// (halo 1)
template <typename T>
__host__ __device__ inline size_t tile_elems(int TX, int TY, int ncls) {
    return (size_t)lut_slots<T>(ncls) + (size_t)(TX + 6) * (TY + 6) + (size_t)(TX + 4) * (TY + 4) +
           3 * (size_t)(TX + 2) * (TY + 2);
}
// and of the form with wind tables: the node wind u, v (halo 2), the wind
// interpolated in x on the tile's columns, and per fire row its wind row and
// weight (u, then v)
template <typename T>
__host__ __device__ inline size_t tile_wind_elems(int TX, int TY, int ky) {
    return 2 * (size_t)(TX + 4) * (TY + 4) + 2 * (size_t)tile_wind_rows(ky) * (TX + 4) + 4 * (size_t)(TY + 4);
}

// ---------------------------------------------------------------------------
// the fused step kernel.  Each stage runs over its frame with consecutive
// threads on consecutive nodes of the frame (a 14x14 frame fills seven warps;
// a warp per row left 18 of 32 lanes idle).  TAB: the wind is interpolated
// once per node, from rows interpolated in x, with the weights and quotients
// formed once per column and row of the tile (per node and stage they cost
// more FP64 than the right-hand side); otherwise per node and stage, and the
// launch is an ordinary one (the code of a chained one alone cost such tiles,
// which nothing waits for, 10 to 20 %: 1000^2 nodes in FP32, tiles of 80x40, 12
// steps 0.92 ms with it, 0.88 without; 510^2 in FP64, tiles of 40x40, 4.6 and
// 4.3, with the linear fuel fraction 8.3 and 6.7).  Small
// meshes, where this kernel is the default, are bound by the latency of its
// chain of stages.  Measured, us per step (GB300), before and now: 100^2 nodes
// in FP64 53.7 and 24.3 (30.0 with the steps not chained, see launch_chained,
// and the quadrature of a node by one lane).
// ---------------------------------------------------------------------------
template <typename T, bool TAB>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 8 ? kTileCtasPerSmF64 : kTileCtasPerSmF32)
    k_fire_step(const StepArgs a) {
    if (TAB) chain_go();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_status;
    const int tid = threadIdx.x;
    const int srx = a.srx, sry = a.sry, nx = a.nx, ny = a.ny;
    const int TX = a.kx * srx, TY = a.ky * sry;
    const int BW3 = TX + 6, BH3 = TY + 6;
    const int BW2 = TX + 4, BH2 = TY + 4;
    const int BW1 = TX + 2, BH1 = TY + 2;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int TXa = min(TX, nx - x0), TYa = min(TY, ny - y0);
    const int WR = TAB ? tile_wind_rows(a.ky) : 0;
    // psi alone (states recomputed for the adjoint): no ignition times, no
    // fuel fraction, no heat
    const bool full = a.F_out != nullptr;

    T *lut = reinterpret_cast<T *>(smem_raw);
    T *P0 = lut + lut_slots<T>(a.ncls);
    T *P1 = P0 + BW3 * BH3;
    T *F1 = P1 + BW2 * BH2;
    T *P2 = F1 + BW1 * BH1;
    T *Dl = P2 + BW1 * BH1;
    T *un_s = Dl + BW1 * BH1;
    T *vn_s = un_s + BW2 * BH2;
    T *wux = vn_s + BW2 * BH2;  // [WR][BW2]
    T *wvx = wux + WR * BW2;
    T *rowt = wvx + WR * BW2;   // [4][BH2]: wind row and weight of u, of v

    const T *psi_in = static_cast<const T *>(a.psi_in);
    T *psi_out = static_cast<T *>(a.psi_out);
    const T *F_in = static_cast<const T *>(a.F_in);
    T *F_out = static_cast<T *>(a.F_out);
    const T *__restrict__ dzdx = static_cast<const T *>(a.dzdx);
    const T *__restrict__ dzdy = static_cast<const T *>(a.dzdy);
    const T *__restrict__ mult = static_cast<const T *>(a.mult);
    const T *__restrict__ wu = static_cast<const T *>(a.u);
    const T *__restrict__ wv = static_cast<const T *>(a.v);
    const uint8_t *__restrict__ fuel = a.fuel;
    // per-node R0, c, d, H_s, H_q of a per-node fuel moisture (all null
    // otherwise): they replace the class values
    const T *__restrict__ nR0 = static_cast<const T *>(a.nco[0]);
    const T *__restrict__ nc = static_cast<const T *>(a.nco[1]);
    const T *__restrict__ nd = static_cast<const T *>(a.nco[2]);
    const T *__restrict__ nhs = static_cast<const T *>(a.nco[3]);
    const T *__restrict__ nhq = static_cast<const T *>(a.nco[4]);
    auto node_coef = [&](int cls, size_t g, T *cn) {
#pragma unroll
        for (int q = 0; q < 6; ++q) cn[q] = lut[cls * K_N + q];
        if (nR0) {
            cn[K_R0] = nR0[g];
            cn[K_C] = nc[g];
            cn[K_D] = nd[g];
        }
    };
    // frame position e of a frame bw columns wide -> its column, row
    auto split = [](int e, int bw, int &lx, int &ly) {
        ly = e / bw;
        lx = e - ly * bw;
    };

    const T dt = T(a.dt);
    const T idx = T(1) / T(a.dx), idy = T(1) / T(a.dy);
    const T i2dx = T(1) / (T(2) * T(a.dx)), i2dy = T(1) / (T(2) * T(a.dy));
    const T eps = T(a.eps);
    const int ncm1 = a.ncls - 1;

    if (tid == 0) s_status = 0;
    int st = 0;
    // ---- A: psi^n on the tile + 3 halo (0 outside the domain), the tables, the
    // node wind.  In a chained launch psi comes last: the rest does not wait
    // for the step before.
    auto load_psi = [&]() {
        for (int e = tid; e < BW3 * BH3; e += kThreads) {
            int lx, ly;
            split(e, BW3, lx, ly);
            const int gy = y0 - 3 + ly, gx = x0 - 3 + lx;
            T val = T(0);
            if (gy >= 0 && gy < ny && gx >= 0 && gx < nx)
                val = psi_in[WF_CHK((size_t)gy * nx + gx, (long long)nx * ny, st)];
            P0[e] = val;
        }
    };
    const bool chained = TAB && a.chained;
    if (!chained) load_psi();
    for (int k = tid; k < a.ncls * K_N; k += kThreads) lut[k] = T(a.coef[k]);
    const int jb = max(y0 / sry - 2, 0);  // first wind row of the table
    for (int e = tid; e < WR * BW2; e += kThreads) {
        int c, j;
        split(e, BW2, c, j);
        const int gx = min(max(x0 - 2 + c, 0), nx - 1);
        const T xa = (T(gx) + T(0.5)) / T(srx);
        int i0, i1;
        T wx;
        lin_idx<T>(xa, a.nxa + 1, i0, i1, wx);
        const int Ju = min(jb + j, a.nya - 1), Jv = min(jb + j, a.nya);
        const size_t bu = (size_t)Ju * (a.nxa + 1);
        const long long nu = (long long)a.nya * (a.nxa + 1), nv = (long long)(a.nya + 1) * a.nxa;
        wux[e] = (T(1) - wx) * __ldg(wu + WF_CHK(bu + i0, nu, st)) + wx * __ldg(wu + WF_CHK(bu + i1, nu, st));
        lin_idx<T>(xa - T(0.5), a.nxa, i0, i1, wx);
        const size_t bv = (size_t)Jv * a.nxa;
        wvx[e] = (T(1) - wx) * __ldg(wv + WF_CHK(bv + i0, nv, st)) + wx * __ldg(wv + WF_CHK(bv + i1, nv, st));
    }
    for (int ly = tid; TAB && ly < BH2; ly += kThreads) {
        const int gy = min(max(y0 - 2 + ly, 0), ny - 1);
        const T ya = (T(gy) + T(0.5)) / T(sry);
        int j0, j1;
        T wy;
        lin_idx<T>(ya - T(0.5), a.nya, j0, j1, wy);
        rowt[ly] = T(j0 - jb);
        rowt[BH2 + ly] = wy;
        lin_idx<T>(ya, a.nya + 1, j0, j1, wy);
        rowt[2 * BH2 + ly] = T(j0 - jb);
        rowt[3 * BH2 + ly] = wy;
    }
    if constexpr (TAB) {
        __syncthreads();
        for (int e = tid; e < BW2 * BH2; e += kThreads) {
            int lx, ly;
            split(e, BW2, lx, ly);
            // (rows past the last of u repeat it, with weight 0; frame nodes
            // outside the mesh take the wind of its edge)
            const T wyu = rowt[BH2 + ly], wyv = rowt[3 * BH2 + ly];
            const T *u0 = wux + (int)rowt[ly] * BW2 + lx, *v0 = wvx + (int)rowt[2 * BH2 + ly] * BW2 + lx;
            const T un = (T(1) - wyu) * u0[0] + wyu * u0[BW2];
            const T vn = (T(1) - wyv) * v0[0] + wyv * v0[BW2];
            if (!finite_val(un) || !finite_val(vn)) st |= ST_NONFINITE;
            un_s[e] = un;
            vn_s[e] = vn;
        }
    }
    if (chained) {
        chain_wait();
        load_psi();
    }
    const double tstart = *a.t_in;
    const double t1 = tstart + a.dt;
    if (tid == 0 && blockIdx.x == 0 && blockIdx.y == 0) *a.t_out = t1;
    __syncthreads();
    const bool edge_tile = (x0 - 3 < 0) || (y0 - 3 < 0) || (x0 + TX + 3 > nx) || (y0 + TY + 3 > ny);
    if (edge_tile) fill_ghosts<T>(P0, BW3, BH3, x0 - 3, y0 - 3, nx, ny, tid);

    // ---- C: stage 1 on the tile + 2 halo: F1 = F(psi^n), psi* = psi^n + dt F1
    for (int e = tid; e < BW2 * BH2; e += kThreads) {
        int lx, ly;
        split(e, BW2, lx, ly);
        const int gy = y0 - 2 + ly, gx = x0 - 2 + lx;
        if (gy < 0 || gy >= ny || gx < 0 || gx >= nx) {
            P1[e] = T(0);
            continue;
        }
        const size_t g = WF_CHK((size_t)gy * nx + gx, (long long)nx * ny, st);
        int cls = fuel[g];
        cls = cls > ncm1 ? ncm1 : cls;
        T un, vn;
        if constexpr (TAB) {
            un = un_s[e];
            vn = vn_s[e];
        } else {
            wind_at<T>(wu, wv, a.nxa, a.nya, srx, sry, gx, gy, un, vn, st);
            if (!finite_val(un) || !finite_val(vn)) st |= ST_NONFINITE;
        }
        const T m = mult ? mult[g] : T(1);
        const int c = (ly + 1) * BW3 + (lx + 1);
        T cn[6];
        node_coef(cls, g, cn);
        const T F = rhs_at<T>(P0, c, BW3, idx, idy, i2dx, i2dy, eps, cn, m, un, vn, dzdx[g], dzdy[g]);
        P1[e] = P0[c] + dt * F;
        if (lx >= 1 && lx < BW2 - 1 && ly >= 1 && ly < BH2 - 1) F1[(ly - 1) * BW1 + (lx - 1)] = F;
    }
    __syncthreads();
    if (edge_tile) fill_ghosts<T>(P1, BW2, BH2, x0 - 2, y0 - 2, nx, ny, tid);

    // ---- E: stage 2 on the tile + 1 halo, ignition-time crossing, Dl = t1 - t_i
    for (int l1 = tid; l1 < BW1 * BH1; l1 += kThreads) {
        int lx, ly;
        split(l1, BW1, lx, ly);
        const int gy = y0 - 1 + ly, gx = x0 - 1 + lx;
        if (gy < 0 || gy >= ny || gx < 0 || gx >= nx) {
            P2[l1] = T(0);
            Dl[l1] = T(0);
            continue;
        }
        const size_t g = WF_CHK((size_t)gy * nx + gx, (long long)nx * ny, st);
        const T p0 = P0[(ly + 2) * BW3 + (lx + 2)];
        // t_i where the node burns already, read ahead of the arithmetic (in the
        // small tiles, bound by latency)
        double ti = 0.0;
        if (TAB && full && le0(p0)) ti = a.tign[g];
        int cls = fuel[g];
        cls = cls > ncm1 ? ncm1 : cls;
        const int c2 = (ly + 1) * BW2 + (lx + 1);
        T un, vn;
        if constexpr (TAB) {
            un = un_s[c2];
            vn = vn_s[c2];
        } else {
            wind_at<T>(wu, wv, a.nxa, a.nya, srx, sry, gx, gy, un, vn, st);
        }
        const T m = mult ? mult[g] : T(1);
        T cn[6];
        node_coef(cls, g, cn);
        const T F2 = rhs_at<T>(P1, c2, BW2, idx, idy, i2dx, i2dy, eps, cn, m, un, vn, dzdx[g], dzdy[g]);
        const T pn = p0 + dt * (T(0.5) * F1[l1] + T(0.5) * F2);
        P2[l1] = pn;
        const bool own = lx >= 1 && lx <= TXa && ly >= 1 && ly <= TYa;
        T d = T(0);
        if (full && le0(pn)) {
            const bool cross = p0 > T(0) && pn <= T(0);
            if (cross || pn < T(0)) {
                if (!TAB || !le0(p0)) ti = a.tign[g];
                if (cross && isinf(ti)) {
                    const double q0 = (double)p0, q1 = (double)pn;
                    ti = tstart + q0 * a.dt / (q0 - q1);
                    if (own) a.tign[g] = ti;
                }
                if (pn < T(0)) d = T(t1 - ti);
            }
        }
        Dl[l1] = d;
        if (own) {
            psi_out[g] = pn;
            if (!finite_val(pn)) st |= ST_NONFINITE;
            const bool band = gx < a.band || gy < a.band || gx >= nx - a.band || gy >= ny - a.band;
            if (band && pn < T(0)) st |= ST_BOUNDARY;
        }
    }
    if (!full) {
        if (st) atomicOr(a.status, st);
        return;
    }
    __syncthreads();
    if (edge_tile) fill_ghosts_pd<T>(P2, Dl, BW1, BH1, x0 - 1, y0 - 1, nx, ny, tid);

    // ---- G: fuel fraction on the tile, heat contributions dF * H per node
    T *Q = P0;  // P0/P1 are dead: 2 values per tile node
    // FP64: a node's four subcells by two lanes, the lower two and the upper
    // two, where the tile's threads suffice: the quadrature is the longest chain
    // of the kernel (100^2 nodes with a fire, tiles of 100 nodes: 25.7 us per
    // step by one lane, 24.3 by two; tiles of 200 nodes 2 % slower by two).  In
    // FP32 the chain is short, and the sum of the four keeps the form (and the
    // rounding) that the other kernels give it.
    const int lanes = sizeof(T) == 8 && 2 * TX * TY <= kThreads && a.scheme != 1 ? 2 : 1;
    for (int e0 = 0; e0 < lanes * TX * TY; e0 += kThreads) {
        const int e = lanes == 2 ? (e0 + tid) >> 1 : e0 + tid, side = lanes == 2 ? tid & 1 : 0;
        int lx, ly;
        split(e, TX, lx, ly);
        const int gy = y0 + ly, gx = x0 + lx;
        const bool in = e < TX * TY && lx < TXa && ly < TYa;
        const size_t g = in ? WF_CHK((size_t)gy * nx + gx, (long long)nx * ny, st) : 0;
        const int cc = (ly + 1) * BW1 + (lx + 1);
        T Fo = T(0), Fn = T(1);
        const T *co = lut;
        if (in) {
            Fo = F_in[g];
            int cls = fuel[g];
            cls = cls > ncm1 ? ncm1 : cls;
            co = lut + cls * K_N;
        }
        if (a.scheme == 1) {
            if (in) {
                T p9[9], d9[9];
#pragma unroll
                for (int b = 0; b < 3; ++b)
#pragma unroll
                    for (int h = 0; h < 3; ++h) {
                        p9[b * 3 + h] = P2[cc + (b - 1) * BW1 + (h - 1)];
                        d9[b * 3 + h] = Dl[cc + (b - 1) * BW1 + (h - 1)];
                    }
                Fn = cell_fraction_linear_vals<T>(p9, d9, co[K_TF]);
            }
        } else if constexpr (sizeof(T) == 8) {
            T bW = T(0), bE = T(0), uW = T(0), uE = T(0);
            if (in) cell_fraction_half<T>(P2, Dl, cc, BW1, side, co[K_TF], bW, bE);
            if (lanes == 2) {
                uW = __shfl_down_sync(0xffffffffu, bW, 1);
                uE = __shfl_down_sync(0xffffffffu, bE, 1);
            } else if (in) {
                cell_fraction_half<T>(P2, Dl, cc, BW1, 1, co[K_TF], uW, uE);
            }
            // (added without contraction: the same bits by one lane and by two)
            Fn = fma(T(-0.25), __dadd_rn(__dadd_rn(__dadd_rn(bW, bE), uW), uE), T(1));
        } else {
            if (in) Fn = cell_fraction<T>(P2, Dl, cc, BW1, co[K_TF]);
        }
        if (side || e >= TX * TY) continue;
        T hs = T(0), hq = T(0);
        if (in) {
            F_out[g] = Fn;
            const T dF = Fo - Fn;
            hs = dF * (nhs ? nhs[g] : co[K_HS]);
            hq = dF * (nhq ? nhq[g] : co[K_HQ]);
        }
        Q[2 * e] = hs;
        Q[2 * e + 1] = hq;
    }
    if (st) atomicOr(&s_status, st);
    __syncthreads();

    // ---- H: average over the atmospheric cells of the tile (Sect. 5, item 6)
    T *Sg = P2;  // P2/Dl are dead: 2 values per row segment of srx nodes
    const int nseg = TY * a.kx;
    for (int sgi = tid; sgi < nseg; sgi += kThreads) {
        const int row = sgi / a.kx, I = sgi - row * a.kx;
        const T *qr = Q + 2 * (row * TX + I * srx);
        T s0 = T(0), s1 = T(0);
        for (int k = 0; k < srx; ++k) {
            s0 += qr[2 * k];
            s1 += qr[2 * k + 1];
        }
        Sg[2 * sgi] = s0;
        Sg[2 * sgi + 1] = s1;
    }
    __syncthreads();
    const int kxa = TXa / srx, kya = TYa / sry;
    const double scale = 1.0 / (a.dt * (double)srx * (double)sry);
    for (int cell = tid; cell < a.kx * a.ky; cell += kThreads) {
        const int J = cell / a.kx, I = cell - J * a.kx;
        if (I >= kxa || J >= kya) continue;
        double h0 = 0.0, h1 = 0.0;
        for (int rr = 0; rr < sry; ++rr) {
            const T *s = Sg + 2 * ((J * sry + rr) * a.kx + I);
            if (s[0] != T(0)) h0 += (double)s[0];
            if (s[1] != T(0)) h1 += (double)s[1];
        }
        int sth = 0;
        const size_t ga = WF_CHK((size_t)(y0 / sry + J) * a.nxa + (x0 / srx + I),
                                 (long long)a.nxa * a.nya, sth);
        if (a.heat_s) a.heat_s[ga] = h0 * scale;
        if (a.heat_l) a.heat_l[ga] = h1 * scale;
        if (sth) atomicOr(a.status, sth);
    }
    if (tid == 0 && s_status) atomicOr(a.status, s_status);
}

// ---------------------------------------------------------------------------
// ignition (Sect. 3.4): psi := min(psi, dist - rho) for each segment in
// order; newly ignited nodes (psi > 0 >= psi_g, no ignition time yet) get
// the arrival time.
//
// A CTA owns a tile of 64 x 16 nodes.  Its threads read the tile's psi,
// and one thread per segment bounds dist - rho over the tile (the distance of
// the tile's centre to the segment, less or plus the tile's radius).  A
// segment can change a node of the tile only where it may lie below the
// tile's largest psi and below the least upper bound of any segment (the
// minimum does not depend on the order of the segments), or where it may
// cover a node (then it may set the ignition time, which does): the others
// are left out for the whole tile, and a tile with none left is done without
// a look at its ignition times.  The exact test in double runs only where one
// in float, with its rounding bounded, cannot exclude it: near a moving torch
// that is every node it is the nearest fire of, and their FP64 operations (some
// 18, with the quotient by |b - a|^2 a product, the limits on the bits and the
// root of sqrt64) bound the kernel; elsewhere reading psi does.  On a 1400x1000 mesh with four drip torches the
// kernel took 163 us when every node tested every segment in double, 59 with
// the exact test's IEEE quotient and root; a step with it takes 69 us (210, 94).
// ---------------------------------------------------------------------------
constexpr int kIgnX = 64, kIgnThreads = 256, kIgnRows = kIgnThreads / kIgnX;
static_assert(kMaxSegPerLaunch <= kIgnThreads, "one thread bounds each segment of a launch");

// the exact test of segment s at a node (x, y): its distance less the radius,
// and the parameter of the segment's nearest point (contracted one way only: the
// same bits in both forms of the kernel)
__device__ __forceinline__ double ignition_distance(const IgnSeg &s, double x, double y, double &u, double &d) {
    const double qx = x - s.ax, qy = y - s.ay;
    u = fma(qx, s.dx, qy * s.dy) * s.il2;
    // u limited to [0, 1] on its bits
    if (__double_as_longlong(u) <= 0) u = 0.0;
    else if (__double2hiint(u) >= 0x3ff00000) u = 1.0;
    const double rx = fma(-u, s.dx, qx), ry = fma(-u, s.dy, qy);
    d = sqrt64(fma(rx, rx, ry * ry));
    return d - s.rho;
}

// PER: nodes of a thread, one above the other.  TILES false: every segment is
// tested at every node.
template <typename T, int PER, bool TILES>
__global__ void __launch_bounds__(kIgnThreads) k_ignite(const IgniteArgs a) {
    constexpr int kIgnY = kIgnRows * PER;
    __shared__ float s_lo[kMaxSegPerLaunch], s_qx[kMaxSegPerLaunch], s_qy[kMaxSegPerLaunch];
    __shared__ int s_list[kMaxSegPerLaunch];
    __shared__ int s_n;
    __shared__ float s_pmax[kIgnThreads / 32];
    __shared__ float s_up;
    T *psi = static_cast<T *>(a.psi);
    const int tid = threadIdx.x, lx = tid % kIgnX, ly = tid / kIgnX;
    const int tx = (a.nx + kIgnX - 1) / kIgnX;
    const int x0 = (int)(blockIdx.x % tx) * kIgnX, y0 = (int)(blockIdx.x / tx) * kIgnY;
    const int i = x0 + lx;
    // the tile's psi, and its largest value rounded up
    T p[PER];
    float pm = -INFINITY;
#pragma unroll
    for (int e = 0; e < PER; ++e) {
        const int j = y0 + ly + e * kIgnRows;
        const bool in = i < a.nx && j < a.ny;
        p[e] = in ? psi[(size_t)j * a.nx + i] : T(0);
        if (in) {
            const float f = sizeof(T) == 8 ? __double2float_ru((double)p[e]) : (float)p[e];
            pm = f == f ? fmaxf(pm, f) : INFINITY;
        }
    }
    int n = a.nseg;
    if constexpr (TILES) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) pm = fmaxf(pm, __shfl_xor_sync(0xffffffffu, pm, o));
        if ((tid & 31) == 0) s_pmax[tid >> 5] = pm;
        // bounds of dist - rho over the tile (float with a margin above its
        // rounding error: coordinates within 1e-6 of their size)
        float lo = 0.0f, up = INFINITY;
        const double xc = ((double)x0 + 0.5 * kIgnX) * a.dx, yc = ((double)y0 + 0.5 * kIgnY) * a.dy;
        if (tid < a.nseg) {
            const IgnSeg &s = a.seg[tid];
            const float qx = (float)(xc - s.ax), qy = (float)(yc - s.ay);
            const float sx = (float)s.dx, sy = (float)s.dy;
            const float L2 = sx * sx + sy * sy;
            float u = L2 > 0.0f ? (qx * sx + qy * sy) / L2 : 0.0f;
            u = fminf(fmaxf(u, 0.0f), 1.0f);
            const float rx = qx - u * sx, ry = qy - u * sy;
            const float d = sqrtf(rx * rx + ry * ry);
            const float rad = 0.5f * hypotf(kIgnX * (float)a.dx, kIgnY * (float)a.dy);
            const float eps = 4e-6f * (fabsf(qx) + fabsf(qy) + fabsf(sx) + fabsf(sy) + rad + fabsf((float)s.rho)) + 1e-6f;
            lo = d - rad - (float)s.rho - eps;
            up = d + rad - (float)s.rho + eps;
            s_lo[tid] = lo;
            s_qx[tid] = qx;
            s_qy[tid] = qy;
        }
        __syncthreads();
        if (tid < 32) {
            float m = -INFINITY;
            for (int k = 0; k < kIgnThreads / 32; ++k) m = fmaxf(m, s_pmax[k]);
            if (m == -INFINITY) m = INFINITY;  // (no node of the tile is a number below infinity)
            if (tid == 0) s_up = m;
        }
        __syncthreads();
        if (tid < kMaxSegPerLaunch) {  // warps 0 and 1
            float m = up;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) m = fminf(m, __shfl_xor_sync(0xffffffffu, m, o));
            if ((tid & 31) == 0) s_pmax[tid >> 5] = m;
        }
        __syncthreads();
        if (tid < 32) {
            const float lim = fminf(s_up, fminf(s_pmax[0], s_pmax[1]));
            int n = 0;
            for (int k0 = 0; k0 < a.nseg; k0 += 32) {
                const int k = k0 + tid;
                const bool take = k < a.nseg && (!(s_lo[k] > lim) || !(s_lo[k] > 0.0f));
                const unsigned v = __ballot_sync(0xffffffffu, take);
                if (take) s_list[n + __popc(v & ((1u << tid) - 1))] = k;
                n += __popc(v);
            }
            if (tid == 0) s_n = n;
        }
        __syncthreads();
        n = s_n;
    }
    if (n == 0 || i >= a.nx) return;
    const double x = ((double)i + 0.5) * a.dx;
#pragma unroll
    for (int e = 0; e < PER; ++e) {
        const int jl = ly + e * kIgnRows, j = y0 + jl;
        if (j >= a.ny) continue;
        const float ox = ((float)lx + 0.5f - 0.5f * kIgnX) * (float)a.dx, oy = ((float)jl + 0.5f - 0.5f * kIgnY) * (float)a.dy;
        const size_t g = (size_t)j * a.nx + i;
        T pe = p[e];
        const double y = ((double)j + 0.5) * a.dy;
        double ti = 0.0;
        bool read = false, changed = false, tchanged = false;
        for (int q = 0; q < n; ++q) {
            const int k = TILES ? s_list[q] : q;
            const IgnSeg &s = a.seg[k];
            // skip the segment only when the exact test below can change
            // neither psi (needs dist < psi + rho) nor, psi then being above
            // dist - rho too, the ignition time; delta bounds the error of the
            // distance in float
            if constexpr (TILES) {
                const float qx = s_qx[k] + ox, qy = s_qy[k] + oy;
                const float sx = (float)s.dx, sy = (float)s.dy;
                const float L2f = sx * sx + sy * sy;
                float u = L2f > 0.0f ? (qx * sx + qy * sy) / L2f : 0.0f;
                u = fminf(fmaxf(u, 0.0f), 1.0f);
                const float rx = qx - u * sx, ry = qy - u * sy;
                const float d2 = rx * rx + ry * ry;
                const float delta = 1e-6f * (fabsf(s_qx[k]) + fabsf(s_qy[k]) + fabsf(ox) + fabsf(oy) + fabsf(sx) + fabsf(sy)) + 1e-6f;
                const float lim = (float)((double)pe + s.rho);
                const float dl = lim + delta + 1e-6f * fabsf(lim);
                if (!(dl > 0.0f && !(d2 > dl * dl))) continue;
            }
            double u, d;
            const double pg = ignition_distance(s, x, y, u, d);
            if (pe > T(0) && __double_as_longlong(pg) <= 0) {  // (pg is a number: at most 0)
                if (!read) {
                    ti = a.tign[g];
                    read = true;
                }
                if (isinf(ti)) {
                    if (s.drip) {
                        // the fire starts at the nearest point when the torch
                        // lays it and reaches the node at S_g, by t at the latest
                        const double ta = fma(u, s.tlay - s.tg, s.tg) + d / s.sg;
                        ti = ta < s.tnow ? ta : s.tnow;
                    } else {
                        ti = s.sg > 0.0 ? s.tg + d / s.sg : s.tg;
                    }
                    tchanged = true;
                }
            }
            // (pg < psi where the rounded pg is: an equal one changes nothing)
            const T pt = T(pg);
            if (pt < pe) {
                pe = pt;
                changed = true;
            }
        }
        if (changed) psi[g] = pe;
        if (tchanged) a.tign[g] = ti;
    }
}

template <typename T>
__global__ void k_fill(T *psi, double *tign, T *frac, size_t n, T psi_far) {
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n;
         k += (size_t)gridDim.x * blockDim.x) {
        psi[k] = psi_far;
        tign[k] = __longlong_as_double(0x7ff0000000000000ULL);  // +inf
        frac[k] = T(1);
    }
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
template <typename T>
size_t step_smem_bytes(int kx, int ky, int srx, int sry, int ncls) {
    return tile_elems<T>(kx * srx, ky * sry, ncls) * sizeof(T);
}

// bytes of the form with wind tables, or 0 where they would cost a resident
// CTA: past a quarter of the SM's shared memory the wind is interpolated per
// node instead
template <typename T>
size_t step_table_bytes(int kx, int ky, int srx, int sry, int ncls) {
    const size_t n = tile_elems<T>(kx * srx, ky * sry, ncls) + tile_wind_elems<T>(kx * srx, ky * sry, ky);
    return n * sizeof(T) <= kTileTabBytes ? n * sizeof(T) : 0;
}

// raised monotonically: the limit is shared by every context in the process
// (the form with tables needs at most kTileTabBytes, set with it)
template <typename T>
cudaError_t prepare_step_kernel(size_t smem_bytes) {
    static std::mutex mu;
    static size_t current[kMaxDevices] = {};  // per device (the attribute is)
    std::lock_guard<std::mutex> lock(mu);
    const int dev = attr_device();
    if (dev >= 0 && smem_bytes <= current[dev]) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k_fire_step<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem_bytes);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_fire_step<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kTileTabBytes);
    if (e == cudaSuccess && dev >= 0) current[dev] = smem_bytes;
    return e;
}

template <typename T>
cudaError_t launch_step(const StepArgs &a, cudaStream_t s) {
    const int TX = a.kx * a.srx, TY = a.ky * a.sry;
    dim3 grid((a.nx + TX - 1) / TX, (a.ny + TY - 1) / TY);
    const size_t smem = step_smem_bytes<T>(a.kx, a.ky, a.srx, a.sry, a.ncls);
    const size_t tab = step_table_bytes<T>(a.kx, a.ky, a.srx, a.sry, a.ncls);
    cudaError_t e = prepare_step_kernel<T>(smem);
    if (e != cudaSuccess) return e;
    return tab ? launch_chained(a.chained, k_fire_step<T, true>, grid, kThreads, tab, s, a)
               : launch_chained(false, k_fire_step<T, false>, grid, kThreads, smem, s, a);
}

template <typename T>
cudaError_t launch_ignite(const IgniteArgs &a, cudaStream_t s) {
    // few nodes, or few tests in all: the bounds of a tile, behind four
    // barriers, and four nodes to a thread take longer than the tests that
    // they save.  us per FP32 step with it, every segment at every node and by
    // tiles: 100^2 nodes, 4 segments 19 and 35, 64 segments 87 and 179; 200^2,
    // 16 segments 54 and 61, 64 segments 163 and 141; 400^2, 4 segments 46 and
    // 44, 16 segments 115 and 69; 800^2, 1 segment 54 and 61, 4 segments 112
    // and 72.
    const double nodes = (double)a.nx * a.ny;
    const bool plain = nodes <= 3e4 || nodes * a.nseg <= 7e5;
    const int rows = kIgnRows * (plain ? 1 : 4);
    const long long tiles = (long long)((a.nx + kIgnX - 1) / kIgnX) * ((a.ny + rows - 1) / rows);
    if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;  // (beyond 2^41 nodes)
    (plain ? k_ignite<T, 1, false> : k_ignite<T, 4, true>)<<<(unsigned)tiles, kIgnThreads, 0, s>>>(a);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_fill(void *psi, double *tign, void *frac, size_t n, double psi_far,
                        cudaStream_t s) {
    int blocks = (int)((n + 255) / 256);
    if (blocks > 152 * 32) blocks = 152 * 32;
    if (blocks < 1) blocks = 1;
    k_fill<T><<<blocks, 256, 0, s>>>(static_cast<T *>(psi), tign, static_cast<T *>(frac), n,
                                     T(psi_far));
    return cudaGetLastError();
}

#define WF_INSTANTIATE(T)                                                                     \
    template size_t step_smem_bytes<T>(int, int, int, int, int);                              \
    template size_t step_table_bytes<T>(int, int, int, int, int);                             \
    template cudaError_t prepare_step_kernel<T>(size_t);                                      \
    template cudaError_t launch_step<T>(const StepArgs &, cudaStream_t);                      \
    template cudaError_t launch_ignite<T>(const IgniteArgs &, cudaStream_t);                  \
    template cudaError_t launch_fill<T>(void *, double *, void *, size_t, double, cudaStream_t);

}  // namespace wf
