// Warp-row fire-step kernel: the whole step of Sect. 5 (items 2-6) in one
// pass over the state, a CTA of NW warps marching down a strip NW rows at a
// time, each warp handling one row of every stage per iteration.
//
// A strip is W <= 60 output columns (W = kx*srx, even) and L = ky*sry output
// rows; lane l of every warp holds the two columns x0 - 2 + 2l and
// x0 - 1 + 2l, so a row is 64 columns: the strip, two halo columns on the
// left and up to two on the right (the outermost are garbage nobody reads).
// Horizontal neighbours come from the adjacent lane by shuffle, vertical
// ones from rings of rows in shared memory.  In iteration i warp w takes
//   stage 1  (eq. Heun, first line) on row y0 - 2 + i NW + w
//   stage 2  (eq. Heun, second line), ignition-time crossing
//            (eq. set-ignition-time) and t - t_i on row y0 - 3 + (i-1) NW + w
//   stage 3  fuel-fraction quadrature (Sect. 3.3) and the burnt fuel of row
//            y0 - 4 + (i-2) NW + w
//   stage 4  the heat of iteration i-1's rows added to the columns' sums, and
//   stage 5  the average per atmospheric cell (Sect. 5, item 6) of the bands
//            of sry rows that stage 4 ended in iteration i-1.
// Every row a stage reads from another warp was written in an earlier
// iteration, so one barrier per NW rows suffices and the stages of one
// iteration are independent of one another.  No row is computed twice but
// the strip's 4 (stage 1) and 2 (stage 2) halo rows.
//
// The two columns of a lane are one float2 and the FP32 arithmetic of the
// right-hand side uses the packed f32x2 instructions.  The quadrature, the
// ignition-time arithmetic (double) and the domain-boundary ghosts
// (Sect. 3.1) run only in warps that need them.  Mesh offsets are 32-bit
// (meshes below 2^31 nodes).
//
// What bounds it: instruction issue.  A row of a warp takes 485 warp
// instructions, 160 of them the method's arithmetic, at 60 % issue with 21 of 24
// warps active per SM (DRAM at 25 % of its rate; 4000^2 nodes, strips of 100
// rows).  The form before it, a warp
// marching alone with its rows in registers, took 515 at 58 % with the 12
// warps its 159 registers allowed, and one strip's rows ran one after the
// other.  Measured, us per FP32 step, before and now (GB300): 8200^2 nodes,
// 50 small fires 808 and 663; the same 42 % burnt 1166 (its dense variant) and
// 940; 2000^2 88 and 64; 510^2 27.7 and 14.5.  What made the difference on
// the way, on the first of these: rings addressed by 32-bit shared addresses
// at constant offsets 926 -> 865; the warp number made warp-uniform by a warp
// reduction, so that rows, ranges and branches live in uniform registers 865
// -> 687; one body without clamps and ghosts for strips inside the mesh 1304
// -> 926.  Tried and slower: two rows per warp and iteration (417 instructions
// a row, but 12 warps: 976), 8 warps per CTA, one straight body for the
// iterations in which every stage has a row (809).
#pragma once

#include <mutex>

#include "fire_device.cuh"
#include "fire_internal.h"
#include "pair_math.cuh"

namespace wf {

template <typename T>
struct WRow {  // y-interpolation of the wind for one fire row
    int ju0, jv0;
    T wyu, wyv;
};

// warps per CTA (rows per iteration) and resident CTAs the registers are
// allotted for: 80 registers and 6 CTAs measured best in FP32 (8200^2 nodes,
// 663 us; 5 CTAs 675, 4 CTAs 919, 7 spill, 948); the per-node coefficients
// need 96
template <typename T, int MODE>
constexpr int row_ctas() {
    return sizeof(T) == 8 ? kRowCtasPerSmF64 : MODE == 2 ? 5 : kRowCtasPerSmF32;
}

// wind rows of a strip's table: its atmospheric rows and those around them
__host__ __device__ constexpr int row_wind_rows(int ky) { return ky + 5; }
// bands that one iteration can end, twice (stage 4 fills one set while stage
// 5 reads the other)
__host__ __device__ constexpr int row_bands(int nw, int sry) { return 2 * ((nw - 1) / sry + 1); }

// Dynamic shared memory of a strip: byte offsets of its parts.  The rings
// (rows of 32 pairs, in the order of the lanes) come first, at offsets the
// compiler knows.
//   Q   [4 NW]  psi*
//   UN, VN [4 NW]  node wind
//   FN  [4 NW]  -F(psi^n), then psi^{n+1}
//   PD  [4 NW]  psi^n, then t - t_i where the row burns
//   DF  [2 NW]  fuel burnt in the step (rows of two iterations)
//   FLAG [2][NW] bytes of two iterations: bit 0, the warp's row of stage 2
//               holds a node with psi^{n+1} <= 0; bit 1, its row of stage 3
//               burnt fuel
template <typename T, int NW>
struct RowSmem {
    using V = typename PairT<T>::t;
    static constexpr int kRow = 32 * sizeof(V);
    static constexpr int Q = 0, UN = Q + 4 * NW * kRow, VN = UN + 4 * NW * kRow,
                         FN = VN + 4 * NW * kRow, PD = FN + 4 * NW * kRow, DF = PD + 4 * NW * kRow,
                         FLAG = DF + 2 * NW * kRow, REST = FLAG + 16;
    static_assert(NW == 4, "the flags of an iteration are the bytes of one word");
    T *wu, *wv;     // [ky + 5][64] wind interpolated in x
    T *hw;          // [bands][2][64] heat sums of ended bands per column
    WRow<T> *rows;  // [L + 4]
    T *lut;         // [ncls][8] S0 R0 b c d e Tf Hs
    T *lut2;        // [ncls][12] S0 S0 R0 R0 b b c c d d e e
    T *lutq;        // [ncls] Hq

    static __host__ __device__ size_t bytes(int ky, int sry, int ncls) {
        size_t b = REST + (size_t)2 * row_wind_rows(ky) * 64 * sizeof(T);
        b += (size_t)row_bands(NW, sry) * 128 * sizeof(T);
        b += (size_t)(ky * sry + 4) * sizeof(WRow<T>);
        b = (b + 15) & ~(size_t)15;
        return b + (size_t)((ncls + 1) & ~1) * 21 * sizeof(T);
    }
    __device__ __forceinline__ void carve(unsigned char *p, int ky, int sry, int ncls) {
        wu = reinterpret_cast<T *>(p + REST);
        wv = wu + row_wind_rows(ky) * 64;
        hw = wv + row_wind_rows(ky) * 64;
        rows = reinterpret_cast<WRow<T> *>(hw + row_bands(NW, sry) * 128);
        unsigned char *q = reinterpret_cast<unsigned char *>(rows + ky * sry + 4);
        const int nc = (ncls + 1) & ~1;
        lut2 = reinterpret_cast<T *>(p + ((size_t)(q - p + 15) & ~(size_t)15));
        lut = lut2 + nc * 12;
        lutq = lut + nc * 8;
    }
};

// shared memory by 32-bit address: the ring addresses of a thread are a few
// registers and an immediate, with nothing rebuilt from the generic window
__device__ __forceinline__ unsigned smem_addr(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void lds_pair(unsigned a, float2 &v) {
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
}
__device__ __forceinline__ void lds_pair(unsigned a, double2 &v) {
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a));
}
template <typename V>
__device__ __forceinline__ V lds(unsigned a) {
    V v;
    lds_pair(a, v);
    return v;
}
__device__ __forceinline__ void sts(unsigned a, float2 v) {
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void sts(unsigned a, double2 v) {
    asm volatile("st.shared.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(v.x), "d"(v.y) : "memory");
}
__device__ __forceinline__ unsigned lds_u32(unsigned a) {
    unsigned v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts_u32(unsigned a, unsigned v) {
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void sts_u8(unsigned a, int v) {
    asm volatile("st.shared.u8 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void lds_wrow(unsigned a, WRow<float> &r) {
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r.ju0), "=r"(r.jv0), "=f"(r.wyu), "=f"(r.wyv)
                 : "r"(a));
}
__device__ __forceinline__ void lds_wrow(unsigned a, WRow<double> &r) {
    asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(r.ju0), "=r"(r.jv0) : "r"(a));
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(r.wyu) : "r"(a + 8));
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(r.wyv) : "r"(a + 16));
}
// a row of the doubled class table: both columns' coefficients for one class
__device__ __forceinline__ void lds_coef(unsigned a, WCoef<float> &co) {
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(co.S0.x), "=f"(co.S0.y), "=f"(co.R0.x), "=f"(co.R0.y)
                 : "r"(a));
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(co.b.x), "=f"(co.b.y), "=f"(co.c.x), "=f"(co.c.y)
                 : "r"(a + 16));
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(co.d.x), "=f"(co.d.y), "=f"(co.e.x), "=f"(co.e.y)
                 : "r"(a + 32));
}
__device__ __forceinline__ void lds_coef(unsigned a, WCoef<double> &co) {
    lds_pair(a, co.S0);
    lds_pair(a + 16, co.R0);
    lds_pair(a + 32, co.b);
    lds_pair(a + 48, co.c);
    lds_pair(a + 64, co.d);
    lds_pair(a + 80, co.e);
}
// max(m, |v.x|, |v.y|), NaN if one of them is
__device__ __forceinline__ float absmax_nan(float m, float2 v) {
    float r;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(m), "f"(v.x), "f"(v.y));
    return r;
}
__device__ __forceinline__ double absmax_nan(double m, double2 v) {
    return fma(v.x, 0.0, fma(v.y, 0.0, m));
}
// lane 0's copy of a value that all lanes hold: the compiler cannot form it
// again from where it came (in the row loop it otherwise converts the double
// arguments anew in every iteration, on the narrow FP64 pipe)
template <typename U>
__device__ __forceinline__ U keep(U x) {
    return __shfl_sync(0xffffffffu, x, 0);
}

// a mesh row's environment as loaded: raw fuel bytes (decoded at use),
// terrain gradient, multiplier, and with ROW_NC the per-node coefficients
template <typename T>
struct RowEnv {
    using V = typename PairT<T>::t;
    int c;  // the two fuel bytes
    V zx, zy, m, R0, cc, d;
};

// What the nodes carry besides fuel class and slope: nothing; a spread
// multiplier or none; or per-node R0, c, d and heat factors (a per-node fuel
// moisture, the planes of StepArgs::nco) with a multiplier or none.
enum { ROW_PLAIN = 0, ROW_MULT = 1, ROW_NC = 2 };

// how a strip lies in the mesh: any; or inside, on a mesh of even or odd width
enum { EDGE = 0, PAIR = 1, SINGLE = 2 };
// the mesh widths a kernel is compiled for: even, odd, or either (an ensemble
// of both).  (With the bodies of both widths in one kernel the even one's
// registers came out worse: 8200^2 nodes 663 -> 740 us.)
enum { WIDTH_EVEN = 0, WIDTH_ODD = 1, WIDTH_ANY = 2 };

// FULL: false for a step of psi alone (no F_out: states recomputed for the
// adjoint), without stages 3 to 5 and the ignition times
template <typename T, int MODE, int NW, int WIDTH, bool FULL = true>
struct RowStrip {
    using V = typename PairT<T>::t;
    using S = RowSmem<T, NW>;
    static constexpr int kRow = S::kRow, kN = 4 * NW * kRow;  // bytes of a ring row, a ring
    static constexpr int E = sizeof(T);
    const StepArgs &a;
    const S &sm;
    unsigned char *smem;
    unsigned sl;     // shared address of the lane's pair in ring row 0
    unsigned swu, swv;  // the same in the wind tables
    unsigned slut;   // shared address of the doubled class table
    int lane, w, x0, y0, La, Wa, nx, ny, srx, sry, ncm1;
    int xa;          // global column of the lane's first column
    bool outA, outB; // output columns of the strip
    // general form only
    bool vec;        // paired vector access (nx even)
    bool inA, inB;   // columns inside the domain
    bool pst;        // both columns are output columns and stored as a pair
    bool slow;       // some lane of the warp stores single columns (warp-uniform)
    bool xedge;      // the strip touches the left or right domain boundary
    bool bedge;      // the strip touches the boundary band in x
    V idx2, idy2, i2dx2, i2dy2, eps2, ndt2, ndth2;
    double tstart, t1;
    mutable int st;  // status bits (also set by the const loaders' index checks)
    T poison;  // the largest |psi^{n+1}| of the lane, NaN once one was

    __device__ __forceinline__ RowStrip(const StepArgs &args, const S &s, unsigned char *p)
        : a(args), sm(s), smem(p) {}

    // The mesh fields.  Inner strips (PAIR, SINGLE): the lane's columns of row
    // r lie at node off = r nx + xa, read and written as pairs where the mesh
    // width is even.  Others (EDGE) form their own offsets: rows and columns
    // outside the domain are read from the nearest inside ones (their values
    // are never used).
    template <int FORM>
    __device__ __forceinline__ V ld(const void *f_, int r, int off) const {
        const T *f = static_cast<const T *>(f_);
        if (FORM == PAIR) return *reinterpret_cast<const V *>(f + WF_CHK(off, nx * ny - 1, st));
        if (FORM == SINGLE) return mk2(f[WF_CHK(off, nx * ny, st)], f[WF_CHK(off + 1, nx * ny, st)]);
        const int rowb = min(max(r, 0), ny - 1) * nx;
        if (vec) return *reinterpret_cast<const V *>(f + WF_CHK(rowb + min(max(xa, 0), nx - 2), nx * ny - 1, st));
        return mk2(f[WF_CHK(rowb + min(max(xa, 0), nx - 1), nx * ny, st)],
                   f[WF_CHK(rowb + min(max(xa + 1, 0), nx - 1), nx * ny, st)]);
    }
    // the column beyond the row on the side of lanes 0 and 31 (x0 - 3,
    // x0 + 62)
    template <int FORM>
    __device__ __forceinline__ T ld_halo(const void *f_, int r, int off) const {
        const T *f = static_cast<const T *>(f_);
        const int d = lane == 0 ? -1 : 2;
        if (FORM != EDGE) return f[WF_CHK(off + d, nx * ny, st)];
        const int rowb = min(max(r, 0), ny - 1) * nx;
        return f[WF_CHK(rowb + min(max(xa + d, 0), nx - 1), nx * ny, st)];
    }
    template <int FORM>
    __device__ __forceinline__ int ld_fuel(int r, int off) const {
        const uint8_t *f = a.fuel;
        if (FORM == PAIR) return *reinterpret_cast<const uint16_t *>(f + WF_CHK(off, nx * ny - 1, st));
        if (FORM == SINGLE) return f[WF_CHK(off, nx * ny, st)] | f[WF_CHK(off + 1, nx * ny, st)] << 8;
        const int rowb = min(max(r, 0), ny - 1) * nx;
        if (vec) return *reinterpret_cast<const uint16_t *>(f + WF_CHK(rowb + min(max(xa, 0), nx - 2), nx * ny - 1, st));
        return f[WF_CHK(rowb + min(max(xa, 0), nx - 1), nx * ny, st)] |
               f[WF_CHK(rowb + min(max(xa + 1, 0), nx - 1), nx * ny, st)] << 8;
    }
    template <int FORM>
    __device__ __forceinline__ void load_env(int r, int off, RowEnv<T> &e) const {
        e.c = ld_fuel<FORM>(r, off);
        e.zx = ld<FORM>(a.dzdx, r, off);
        e.zy = ld<FORM>(a.dzdy, r, off);
        if (MODE != ROW_PLAIN && a.mult) e.m = ld<FORM>(a.mult, r, off);
        if constexpr (MODE == ROW_NC) {
            e.R0 = ld<FORM>(a.nco[0], r, off);
            e.cc = ld<FORM>(a.nco[1], r, off);
            e.d = ld<FORM>(a.nco[2], r, off);
        }
    }
    __device__ __forceinline__ void coef(const RowEnv<T> &e, WCoef<T> &co) const {
        lds_coef(slut + min(e.c & 0xff, ncm1) * (12 * E), co);
        const bool two = (e.c >> 8) != (e.c & 0xff);
        if (__any_sync(0xffffffffu, two)) {  // a fuel boundary
            if (two) {
                const T *l1 = sm.lut2 + min(e.c >> 8, ncm1) * 12;
                co.S0.y = l1[0];
                co.R0.y = l1[2];
                co.b.y = l1[4];
                co.c.y = l1[6];
                co.d.y = l1[8];
                co.e.y = l1[10];
            }
        }
        if constexpr (MODE == ROW_NC) {
            co.R0 = e.R0;
            co.c = e.cc;
            co.d = e.d;
        }
    }

    // horizontal neighbours of a row of pairs: left of .x, right of .y
    __device__ __forceinline__ void sides(V v, T &l, T &r) const {
        l = __shfl_up_sync(0xffffffffu, v.y, 1);
        r = __shfl_down_sync(0xffffffffu, v.x, 1);
    }

    // 5-point values of the lane's two columns at row r from the rows below
    // (D), at (c) and above (U), with the ghosts of Sect. 3.1 at the domain
    // boundary; l, rr the values left of c.x and right of c.y
    template <int FORM>
    __device__ __forceinline__ void stencil(V &D, V c, V &U, T l, T rr, int r, V &L, V &R) const {
        L = mk2(l, c.x);
        R = mk2(c.y, rr);
        if (FORM != EDGE) return;
        if (xedge) {
            if (xa == 0) L.x = ghost_value<T>(c.x, c.y);
            if (xa + 1 == nx - 1) R.y = ghost_value<T>(c.y, c.x);
            if (xa == nx - 1) R.x = ghost_value<T>(c.x, L.x);
        }
        const V d0 = D, u0 = U;
        if (r == 0) D = mk2(ghost_value<T>(c.x, u0.x), ghost_value<T>(c.y, u0.y));
        if (r == ny - 1) U = mk2(ghost_value<T>(c.x, d0.x), ghost_value<T>(c.y, d0.y));
    }

    // tables of the strip: class coefficients, wind-row weights, x-interpolated
    // wind rows.  Called by all threads of the CTA, which then synchronise.
    __device__ __forceinline__ void tables() {
        const int tid = threadIdx.x;
        for (int k = tid; k < a.ncls; k += 32 * NW) {
            const double *co = a.coef + (size_t)k * K_N;
            T *l = sm.lut + k * 8;
            l[0] = T(co[K_S0]);
            l[1] = T(co[K_R0]);
            l[2] = T(co[K_B]);
            l[3] = T(co[K_C]);
            l[4] = T(co[K_D]);
            l[5] = T(co[K_E]);
            l[6] = T(co[K_TF]);
            l[7] = T(co[K_HS]);
            sm.lutq[k] = T(co[K_HQ]);
            T *l2 = sm.lut2 + k * 12;
            for (int j = 0; j < 6; ++j) l2[2 * j] = l2[2 * j + 1] = l[j];
        }
        const int nxa = a.nxa, nya = a.nya;
        const int jb = max(y0 / sry - 2, 0);  // first wind row of the table
        for (int i = tid; i < La + 4; i += 32 * NW) {
            const int r = y0 - 2 + i;
            WRow<T> wr;
            wr.ju0 = wr.jv0 = 0;
            wr.wyu = wr.wyv = T(0);
            if (r >= 0 && r < ny) {
                int j1;
                const T yr = (T(r) + T(0.5)) / T(sry);
                lin_idx<T>(yr - T(0.5), nya, wr.ju0, j1, wr.wyu);
                lin_idx<T>(yr, nya + 1, wr.jv0, j1, wr.wyv);
                wr.ju0 = (wr.ju0 - jb) * 64 * E;  // byte offsets in the table
                wr.jv0 = (wr.jv0 - jb) * 64 * E;
            }
            sm.rows[i] = wr;
        }
        // thread: one of the 64 columns, every (NW / 2)-th row
        const int c = tid & 63;
        const int x = min(max(x0 - 2 + c, 0), nx - 1);
        int iu0, iu1, iv0, iv1;
        T wxu, wxv;
        const T xr = (T(x) + T(0.5)) / T(srx);
        lin_idx<T>(xr, nxa + 1, iu0, iu1, wxu);
        lin_idx<T>(xr - T(0.5), nxa, iv0, iv1, wxv);
        const int nr = row_wind_rows((La + sry - 1) / sry);
        T bad = T(0);
        for (int j = tid >> 6; j < nr; j += NW / 2) {
            const int Ju = min(jb + j, nya - 1), Jv = min(jb + j, nya);
            const T *u = static_cast<const T *>(a.u) + (size_t)Ju * (nxa + 1);
            const T *v = static_cast<const T *>(a.v) + (size_t)Jv * nxa;
            const int bu = Ju * (nxa + 1), nu = nya * (nxa + 1);  // (index checks only)
            const int bv = Jv * nxa, nv = (nya + 1) * nxa;
            const T wu = (T(1) - wxu) * __ldg(u + WF_CHK_AT(bu, iu0, nu, st)) +
                         wxu * __ldg(u + WF_CHK_AT(bu, iu1, nu, st));
            const T wv = (T(1) - wxv) * __ldg(v + WF_CHK_AT(bv, iv0, nv, st)) +
                         wxv * __ldg(v + WF_CHK_AT(bv, iv1, nv, st));
            sm.wu[j * 64 + c] = wu;
            sm.wv[j * 64 + c] = wv;
            // a non-finite wind value poisons the status
            bad = fma(wu, T(0), fma(wv, T(0), bad));
        }
        if (!finite_val(bad)) st |= ST_NONFINITE;
    }

    // bilinear wind (Sect. 5) of the fire row whose weights lie at address r
    __device__ __forceinline__ void wind(unsigned r, V &un, V &vn) const {
        WRow<T> k;
        lds_wrow(r, k);
        const V UA = lds<V>(swu + k.ju0), UB = lds<V>(swu + k.ju0 + 64 * E);
        const V VA = lds<V>(swv + k.jv0), VB = lds<V>(swv + k.jv0 + 64 * E);
        const V dU = sub2(UB, UA), dV = sub2(VB, VA);
        un = mk2(fma(k.wyu, dU.x, UA.x), fma(k.wyu, dU.y, UA.y));
        vn = mk2(fma(k.wyv, dV.x, VA.x), fma(k.wyv, dV.y, VA.y));
    }

    // One step of the strip with output origin (x0_, y0_), rows [y0_, y0_ +
    // La); all threads of the CTA.  Ends with a barrier.
    __device__ __forceinline__ void run(int x0_, int y0_, double tstart_) {
        const int tid = threadIdx.x;
        lane = __shfl_xor_sync(0xffffffffu, tid & 31, 0);  // (not read anew from its special register)
        // warp-uniform values by a warp reduction, so that they and what
        // depends on them live in uniform registers
        w = __reduce_min_sync(0xffffffffu, tid >> 5);
        srx = a.srx;
        sry = a.sry;
        nx = a.nx;
        ny = a.ny;
        x0 = __reduce_min_sync(0xffffffffu, x0_);
        y0 = __reduce_min_sync(0xffffffffu, y0_);
        La = min(a.ky * sry, ny - y0);
        Wa = min(a.kx * srx, nx - x0);
        xa = x0 - 2 + 2 * lane;
        outA = xa >= x0 && xa < x0 + Wa;
        outB = xa + 1 >= x0 && xa + 1 < x0 + Wa;
        ncm1 = a.ncls - 1;
        auto both = [](T x) { return splat<V>(keep(x)); };
        idx2 = both(T(1) / T(a.dx));
        idy2 = both(T(1) / T(a.dy));
        i2dx2 = both(T(1) / (T(2) * T(a.dx)));
        i2dy2 = both(T(1) / (T(2) * T(a.dy)));
        eps2 = both(T(a.eps));
        ndt2 = both(-T(a.dt));
        ndth2 = both(-(T(0.5) * T(a.dt)));
        tstart = tstart_;
        t1 = tstart + a.dt;
        st = 0;
        poison = T(0);
        sl = smem_addr(smem) + lane * (int)sizeof(V);
        swu = smem_addr(sm.wu) + lane * (int)sizeof(V);
        swv = smem_addr(sm.wv) + lane * (int)sizeof(V);
        slut = smem_addr(sm.lut2);
        // inner strips: the 64 columns, the halo columns and rows all lie
        // inside the domain, away from the boundary band: no clamp, ghost or
        // boundary case can arise
        const int band = a.band;
        // (FP32: its operations are spelled out one by one.  In FP64 the
        // compiler contracts products and sums as it likes, in two bodies
        // perhaps not alike, so there is one.)
        const bool inner = sizeof(T) == 4 && x0 >= 4 && x0 + 63 < nx && y0 >= 3 &&
                           y0 + La + 3 <= ny && x0 >= band && x0 + Wa <= nx - band && y0 >= band &&
                           y0 + La <= ny - band;
        if (inner) {
            if constexpr (sizeof(T) == 4) {
                if constexpr (WIDTH == WIDTH_EVEN) loop<PAIR>();
                else if constexpr (WIDTH == WIDTH_ODD) loop<SINGLE>();
                else if ((nx & 1) == 0) loop<PAIR>();
                else loop<SINGLE>();
            }
        } else {
            vec = WIDTH == WIDTH_EVEN || (WIDTH == WIDTH_ANY && (nx & 1) == 0);
            inA = xa >= 0 && xa < nx;
            inB = xa + 1 >= 0 && xa + 1 < nx;
            pst = vec && outA && outB;
            slow = __any_sync(0xffffffffu, !pst && (outA || outB));
            xedge = x0 - 2 <= 0 || x0 + 62 >= nx - 1;
            bedge = x0 < band || x0 + Wa > nx - band;
            loop<EDGE>();
        }
        if (!finite_val(poison)) st |= ST_NONFINITE;
    }

    template <int FORM>
    __device__ __forceinline__ void loop() {
        const bool hlane = lane == 0 || lane == 31;
        // stage 1's row relative to y0, and its node; the rows of stages 2
        // and 3 follow at k - NW - 1 and k - 2 NW - 2
        int k = w - 2;
        int o1 = (y0 + k) * nx + xa;
        V Pd, Pc, Pu, Fn;
        T ph = T(0);
        RowEnv<T> e1, e2;
        e1.m = e2.m = splat<V>(T(1));
        auto load1 = [&](int r, int o) {
            Pd = ld<FORM>(a.psi_in, r - 1, o - nx);
            Pc = ld<FORM>(a.psi_in, r, o);
            Pu = ld<FORM>(a.psi_in, r + 1, o + nx);
            if (hlane) ph = ld_halo<FORM>(a.psi_in, r, o);
            load_env<FORM>(r, o, e1);
        };
        // the first row of stage 1, in flight while the tables are built
        if (k <= La + 1) load1(y0 + k, o1);
        Fn = splat<V>(T(1));
        e2 = e1;
        tables();
        const unsigned sflag = smem_addr(smem) + S::FLAG;
        if (threadIdx.x < 2) sts_u32(sflag + 4 * threadIdx.x, 0u);
        __syncthreads();

        T acc = T(0);      // stage 4: the heat sum of one column and quantity
        bool bhot = false; // the rows of the current band so far burnt fuel
        int d4 = 0;        // rows stage 4 has taken
        int bend = sry;    // end of its current band
        unsigned hotbits = 0;  // bit b: the band ended b bands ago burnt fuel
        int bdone = 0;     // bands ended by stage 4 before this iteration
        int bavg = 0;      // bands averaged by stage 5
        unsigned f1 = 0;   // flags of iteration i - 2
        // iterations left (psi alone: until stage 2 has taken row La - 1)
        int left = FULL ? (La + 3) / NW + 5 : (La + 3 + NW - 1) / NW + 1;
        unsigned n1 = w * kRow;        // ring offset of stage 1's row
        unsigned aw = smem_addr(sm.rows + w);  // wind weights of stage 1's row
        // bytes w + 2 .. w + 4 of two iterations' flags: rows k3 - 1 .. k3 + 1
        const unsigned sel = 0x432u + 0x111u * w;
        unsigned af = sflag, ad = S::DF;  // flags, dF rows of iteration i (two sets in turn)
#pragma unroll 1
        for (; left > 0; --left) {
            const unsigned f0 = FULL ? lds_u32(af ^ 4) : 0u;  // flags of iteration i - 1
            int flag = 0;
            const unsigned n2 = (n1 - (NW + 1) * kRow) & (kN - 1);
            // ---- stage 3 on row k3
            const int k3 = k - 2 * NW - 2;
            if (FULL && (unsigned)k3 < (unsigned)La) {
                // flags of rows k3 - 1, k3, k3 + 1: warps w - 2, w - 1, w of
                // iteration i - 1, counted on from those of i - 2
                const unsigned burn = __byte_perm(f1, f0, sel);
                if (stage3<FORM>(y0 + k3, o1 - (2 * NW + 2) * nx, (n2 - (NW + 1) * kRow) & (kN - 1), burn, Fn,
                                 ad + w * kRow))
                    flag |= 2;
            }
            // ---- stage 2 on row k2; stage 3's next F^n row (each load goes into
            // the registers whose last use is just behind, so that nothing
            // waits for it before the next iteration)
            const int k2 = k - NW - 1;
            if (FULL ? (unsigned)(k2 + 1) <= (unsigned)(La + 1) : (unsigned)k2 < (unsigned)La) {
                if (FORM != EDGE || (y0 + k2 >= 0 && y0 + k2 < ny))
                    flag |= stage2<FORM>(y0 + k2, o1 - (NW + 1) * nx, n2, e2) ? 1 : 0;
                if (FULL) Fn = ld<FORM>(a.F_in, y0 + k2 - 1, o1 - (NW + 2) * nx);
            }
            // ---- stage 1 on row k; loads of its next row
            if (k <= La + 1) {
                load_env<FORM>(y0 + k - 1, o1 - nx, e2);
                if (FORM != EDGE || (y0 + k >= 0 && y0 + k < ny)) {
                    V un, vn;
                    wind(aw, un, vn);
                    T l, rr;
                    sides(Pc, l, rr);
                    if (lane == 0) l = ph;
                    if (lane == 31) rr = ph;
                    V L, R;
                    V D = Pd, U = Pu;
                    stencil<FORM>(D, Pc, U, l, rr, y0 + k, L, R);
                    WCoef<T> co;
                    coef(e1, co);
                    const V G = neg_rhs2<T, MODE != ROW_PLAIN, true>(Pc, L, R, D, U, idx2, idy2, i2dx2, i2dy2,
                                                               eps2, co, e1.m, un, vn, e1.zx, e1.zy);
                    const unsigned s1 = sl + n1;
                    sts(s1 + S::Q, fma2(ndt2, G, Pc));
                    sts(s1 + S::UN, un);
                    sts(s1 + S::VN, vn);
                    sts(s1 + S::FN, G);
                    sts(s1 + S::PD, Pc);
                }
                if (k + NW <= La + 1) load1(y0 + k + NW, o1 + NW * nx);
            }
            if constexpr (FULL) {
                f1 = f0;
                if (lane == 0) sts_u8(af + w, flag);
                // ---- stage 5: averages of the bands ended in iteration i - 1
                for (; bavg < bdone; ++bavg) average(bavg, (hotbits >> (bdone - 1 - bavg)) & 1u);
                // ---- stage 4: heat of the rows stage 3 took in iteration i - 1
                const int e4 = min(k3 - w, La);  // one past the last of them
                if (e4 >= bend || (f0 & 0x02020202u)) {
                    const int rf = k3 - w - NW;  // the first (negative: none yet)
                    for (int r = max(d4, 0); r < e4; ++r) {
                        if ((f0 >> (8 * (r - rf))) & 2u) {
                            bhot = true;
                            add_heat(y0 + r, (2 * S::DF + NW * kRow - ad) + (r - rf) * kRow, acc);
                        }
                        if (r + 1 == bend) {
                            bend += sry;
                            if (bhot) {
                                sm.hw[(bdone % row_bands(NW, sry)) * 128 + (w < 2 ? 0 : 64) + (w & 1) * 32 + lane] = acc;
                                acc = T(0);
                            }
                            hotbits = (hotbits << 1) | (bhot ? 1u : 0u);
                            bhot = false;
                            ++bdone;
                        }
                    }
                }
                d4 = e4;
            }
            k += NW;
            o1 += NW * nx;
            n1 = (n1 + NW * kRow) & (kN - 1);
            aw += NW * sizeof(WRow<T>);
            af ^= 4;
            ad = 2 * S::DF + NW * kRow - ad;
            __syncthreads();
        }
    }

    // stage 4: the fuel burnt in row r added to the heat sum of the thread's
    // column and quantity (warps 0, 1 sensible, 2, 3 latent)
    __device__ __forceinline__ void add_heat(int r, int dF, T &acc) {
        const int c = (w & 1) * 32 + lane;
        const T d = reinterpret_cast<const T *>(smem + dF)[c];
        if (d == T(0)) return;
        const int g = r * nx + x0 - 2 + c;
        T H;
        if constexpr (MODE == ROW_NC) {
            H = static_cast<const T *>(a.nco[w < 2 ? 3 : 4])[WF_CHK(g, nx * ny, st)];
        } else {
            const int cls = min((int)a.fuel[WF_CHK(g, nx * ny, st)], ncm1);
            H = w < 2 ? sm.lut[cls * 8 + 7] : sm.lutq[cls];
        }
        acc = fma(d, H, acc);
    }

    // stage 5: the averages of band b (zero where nothing of it burnt); one
    // warp per quantity, a lane per atmospheric cell
    __device__ __forceinline__ void average(int b, bool burnt) {
        if (w < NW - 2) return;
        double *out = w == NW - 1 ? a.heat_l : a.heat_s;
        if (!out) return;
        const T *h = sm.hw + (b % row_bands(NW, sry)) * 128 + (w == NW - 1 ? 64 : 0);
        const double hscale = 1.0 / (a.dt * (double)srx * (double)sry);
        for (int c = lane; c * srx < Wa; c += 32) {
            T s = T(0);
            if (burnt)
                for (int e = 0; e < srx; ++e) s += h[2 + c * srx + e];
            const size_t ga = WF_CHK((size_t)(y0 / sry + b) * a.nxa + (x0 / srx + c), a.nxa * a.nya, st);
            out[ga] = burnt ? (double)s * hscale : 0.0;
        }
    }

    // stage 2 of row r at offset off, ring offset n2; returns whether
    // some node of the row has psi^{n+1} <= 0 (t - t_i is then in PD)
    template <int FORM>
    __device__ __forceinline__ bool stage2(int r, int off, unsigned n2, const RowEnv<T> &e) {
        const bool own_row = r >= y0 && r < y0 + La;
        const unsigned s2 = sl + n2;
        const V P0 = lds<V>(s2 + S::PD), Qc = lds<V>(s2 + S::Q);
        V D = lds<V>(sl + ((n2 - kRow) & (kN - 1)) + S::Q);
        V U = lds<V>(sl + ((n2 + kRow) & (kN - 1)) + S::Q);
        const V un = lds<V>(s2 + S::UN), vn = lds<V>(s2 + S::VN);
        // t_i where psi^n <= 0, read ahead of the arithmetic (such nodes get
        // no new t_i in this step, so no other warp writes them)
        const bool fa = lane > 0 && (FORM != EDGE || inA), fb = lane < 31 && (FORM != EDGE || inB);
        double tiA = 0.0, tiB = 0.0;
        if (FULL && __any_sync(0xffffffffu, min_val(P0.x, P0.y) <= T(0))) {
            const int g = r * nx + xa;
            if (fa && P0.x <= T(0)) tiA = a.tign[WF_CHK(g, nx * ny, st)];
            if (fb && P0.y <= T(0)) tiB = a.tign[WF_CHK(g + 1, nx * ny, st)];
        }
        T l, rr;
        sides(Qc, l, rr);
        V L, R;
        stencil<FORM>(D, Qc, U, l, rr, r, L, R);
        WCoef<T> co;
        coef(e, co);
        const V G2 = neg_rhs2<T, MODE != ROW_PLAIN, true>(Qc, L, R, D, U, idx2, idy2, i2dx2, i2dy2, eps2, co, e.m,
                                                    un, vn, e.zx, e.zy);
        // P0 + dt (F0/2 + F2/2) = P0 - dt/2 (G0 + G2), the halving exact
        const V N0 = fma2(ndth2, add2(lds<V>(s2 + S::FN), G2), P0);
        sts(s2 + S::FN, N0);
        // every column of the row is computed from in-domain values, so a
        // non-finite value anywhere in it comes from one of the step
        poison = absmax_nan(poison, N0);
        if (own_row) {
            if (FORM == EDGE) {
                const int band = a.band;
                if (bedge || r < band || r >= ny - band) {
                    const bool ea = xa < band || xa >= nx - band || r < band || r >= ny - band;
                    const bool eb = xa + 1 < band || xa + 1 >= nx - band || r < band || r >= ny - band;
                    if ((outA && ea && N0.x < T(0)) || (outB && eb && N0.y < T(0))) st |= ST_BOUNDARY;
                }
            }
            store<FORM>(a.psi_out, r, off, N0);
        }
        if constexpr (!FULL) return false;
        // ignition time and t - t_i, only where a node is burning
        const bool burn = __any_sync(0xffffffffu, min_val(N0.x, N0.y) <= T(0));
        if (burn) {
            const bool na = fa && N0.x <= T(0), nb = fb && N0.y <= T(0);
            const int g = r * nx + xa;
            V D0 = splat<V>(T(0));
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                if (!(j == 0 ? na : nb)) continue;
                const T p0 = j == 0 ? P0.x : P0.y, pn = j == 0 ? N0.x : N0.y;
                double ti = j == 0 ? tiA : tiB;
                if (p0 > T(0)) {
                    ti = a.tign[WF_CHK(g + j, nx * ny, st)];
                    if (tign_unset(ti)) {
                        const double q0 = (double)p0, q1 = (double)pn;
                        ti = tstart + q0 * a.dt / (q0 - q1);
                        if (own_row && (j == 0 ? outA : outB)) a.tign[WF_CHK(g + j, nx * ny, st)] = ti;
                    }
                }
                if (pn < T(0)) {
                    if (j == 0) D0.x = T(t1 - ti);
                    else D0.y = T(t1 - ti);
                }
            }
            sts(s2 + S::PD, D0);
        }
        return burn;
    }

    // the output columns of the pair v at row r
    template <int FORM>
    __device__ __forceinline__ void store(void *f_, int r, int off, V v) const {
        T *f = static_cast<T *>(f_);
        if (FORM == PAIR) {
            if (outA) *reinterpret_cast<V *>(f + WF_CHK(off, nx * ny - 1, st)) = v;
            return;
        }
        if (FORM == SINGLE) {
            if (outA) f[WF_CHK(off, nx * ny, st)] = v.x;
            if (outB) f[WF_CHK(off + 1, nx * ny, st)] = v.y;
            return;
        }
        const int g = r * nx + xa;
        if (pst) *reinterpret_cast<V *>(f + WF_CHK(g, nx * ny - 1, st)) = v;
        if (slow) {
            if (!pst && outA) f[WF_CHK(g, nx * ny, st)] = v.x;
            if (!pst && outB) f[WF_CHK(g + 1, nx * ny, st)] = v.y;
        }
    }

    // fuel fraction of row r (ring offset n; bits 0, 8, 16 of `burn`:
    // rows r - 1, r, r + 1 hold a node with psi^{n+1} <= 0); returns whether fuel
    // burnt in the row, its amount per output column then at dF
    template <int FORM>
    __device__ __forceinline__ bool stage3(int r, int off, unsigned n, unsigned burn, V Fn, unsigned dF_) {
        V F1 = splat<V>(T(1));
        if (FORM == EDGE && r == 0) burn &= ~1u;
        if (FORM == EDGE && r == ny - 1) burn &= ~0x10000u;
        // no node of the three rows had psi^{n+1} <= 0 (the votes of stage 2
        // cover every column the quadrature reads): every fraction is 1
        if (burn & 0x010101u) {
            const V zero = splat<V>(T(0));
            const unsigned ra = sl + ((n - kRow) & (kN - 1)), rb = sl + n, rc = sl + ((n + kRow) & (kN - 1));
            const V Da = (burn & 1u) ? lds<V>(ra + S::PD) : zero, Db = (burn & 0x100u) ? lds<V>(rb + S::PD) : zero,
                    Dc = (burn & 0x10000u) ? lds<V>(rc + S::PD) : zero;
            gate<FORM>(r, lds<V>(ra + S::FN), lds<V>(rb + S::FN), lds<V>(rc + S::FN), Da, Db, Dc, F1);
        }
        store<FORM>(a.F_out, r, off, F1);
        V dF = sub2(Fn, F1);
        if (!__any_sync(0xffffffffu, dF.x != T(0) || dF.y != T(0))) return false;
        dF.x = outA ? dF.x : T(0);
        dF.y = outB ? dF.y : T(0);
        sts(sl + dF_, dF);
        return true;
    }

    // minimum of psi^{n+1} over the 3x3 neighbourhood of each output column
    // (in-domain values only; ghosts are never below them), and the full
    // quadrature where it is negative
    template <int FORM>
    __device__ __forceinline__ void gate(int rD, V Na, V Nb, V Nc, V Da, V Db, V Dc, V &F1) {
        const T big = T(1e30);
        T va = min_val(min_val(Na.x, Nb.x), Nc.x), vb = min_val(min_val(Na.y, Nb.y), Nc.y);
        if (FORM != EDGE) {
        } else if (rD == 0) {
            va = min_val(Nb.x, Nc.x);
            vb = min_val(Nb.y, Nc.y);
        } else if (rD == ny - 1) {
            va = min_val(Na.x, Nb.x);
            vb = min_val(Na.y, Nb.y);
        }
        if (FORM == EDGE) {
            va = inA ? va : big;
            vb = inB ? vb : big;
        }
        T vl, vr;
        sides(mk2(va, vb), vl, vr);
        const T ma = min_val(min_val(vl, va), vb), mb = min_val(min_val(va, vb), vr);
        const bool ba = outA && ma < T(0), bb = outB && mb < T(0);
        if (__any_sync(0xffffffffu, ba || bb)) {
            // full quadrature: neighbours of three rows of psi and t - t_i
            T pl[3], pr[3], dl[3], dr[3];
            sides(Na, pl[0], pr[0]);
            sides(Nb, pl[1], pr[1]);
            sides(Nc, pl[2], pr[2]);
            sides(Da, dl[0], dr[0]);
            sides(Db, dl[1], dr[1]);
            sides(Dc, dl[2], dr[2]);
            const V Nr[3] = {Na, Nb, Nc}, Dr[3] = {Da, Db, Dc};
            if constexpr (sizeof(T) == 4) {
                // away from the domain boundary: both cells of the lane in
                // one packed evaluation; F = 1 stays where no node of a
                // cell's neighbourhood burns
                if (FORM != EDGE || (rD > 0 && rD < ny - 1 && xa > 0 && xa + 1 < nx - 1)) {
                    if (ba || bb) {
                        float2 qp[3][3], ep[3][3];
#pragma unroll
                        for (int b = 0; b < 3; ++b) {
                            qp[b][0] = mk2(pl[b], Nr[b].x);
                            qp[b][1] = Nr[b];
                            qp[b][2] = mk2(Nr[b].y, pr[b]);
                            ep[b][0] = mk2(dl[b], Dr[b].x);
                            ep[b][1] = Dr[b];
                            ep[b][2] = mk2(Dr[b].y, dr[b]);
                        }
                        const int g = rD * nx + xa;
                        const int ca = ba ? a.fuel[WF_CHK(g, nx * ny, st)] : 0;
                        const int cb = bb ? a.fuel[WF_CHK(g + 1, nx * ny, st)] : 0;
                        const float2 tf = mk2(sm.lut[(ca > ncm1 ? ncm1 : ca) * 8 + 6],
                                              sm.lut[(cb > ncm1 ? ncm1 : cb) * 8 + 6]);
                        const float2 f = cell_fraction_pair(qp, ep, tf);
                        F1.x = ba ? f.x : 1.0f;
                        F1.y = bb ? f.y : 1.0f;
                    }
                    return;
                }
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                if (!(j == 0 ? ba : bb)) continue;
                T q[3][3], e[3][3];
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    if (j == 0) {
                        q[b][0] = pl[b];
                        q[b][1] = Nr[b].x;
                        q[b][2] = Nr[b].y;
                        e[b][0] = dl[b];
                        e[b][1] = Dr[b].x;
                        e[b][2] = Dr[b].y;
                    } else {
                        q[b][0] = Nr[b].x;
                        q[b][1] = Nr[b].y;
                        q[b][2] = pr[b];
                        e[b][0] = Dr[b].x;
                        e[b][1] = Dr[b].y;
                        e[b][2] = dr[b];
                    }
                }
                const int x = xa + j;
                if (FORM == EDGE && (x == 0 || x == nx - 1 || rD == 0 || rD == ny - 1)) {
                    // ghost ring of psi^{n+1} (x first, then y) and of t - t_i
#pragma unroll
                    for (int b = 0; b < 3; ++b) {
                        const int yy = rD + b - 1;
                        if (yy < 0 || yy >= ny) continue;
                        if (x == 0) {
                            q[b][0] = ghost_value<T>(q[b][1], q[b][2]);
                            e[b][0] = q[b][0] >= T(0) ? T(0) : e[b][1];
                        }
                        if (x == nx - 1) {
                            q[b][2] = ghost_value<T>(q[b][1], q[b][0]);
                            e[b][2] = q[b][2] >= T(0) ? T(0) : e[b][1];
                        }
                    }
#pragma unroll
                    for (int h = 0; h < 3; ++h) {
                        if (rD == 0) {
                            q[0][h] = ghost_value<T>(q[1][h], q[2][h]);
                            e[0][h] = q[0][h] >= T(0) ? T(0) : e[1][h];
                        }
                        if (rD == ny - 1) {
                            q[2][h] = ghost_value<T>(q[1][h], q[0][h]);
                            e[2][h] = q[2][h] >= T(0) ? T(0) : e[1][h];
                        }
                    }
                }
                const int cls0 = a.fuel[WF_CHK(rD * nx + x, nx * ny, st)];
                const int cls = cls0 > ncm1 ? ncm1 : cls0;
                const T f = cell_fraction_vals<T>(q[0][0], q[0][1], q[0][2], q[1][0], q[1][1],
                                                  q[1][2], q[2][0], q[2][1], q[2][2], e[0][0],
                                                  e[0][1], e[0][2], e[1][0], e[1][1], e[1][2],
                                                  e[2][0], e[2][1], e[2][2], sm.lut[cls * 8 + 6]);
                if (j == 0) F1.x = f;
                else F1.y = f;
            }
        }
    }
};

template <typename T, int MODE, int WIDTH, bool FULL>
__global__ void __launch_bounds__(32 * kRowWarps, (row_ctas<T, MODE>())) k_fire_warp(const StepArgs a) {
    extern __shared__ __align__(16) unsigned char row_smem[];
    constexpr int NW = kRowWarps;
    RowSmem<T, NW> sm;
    sm.carve(row_smem, a.ky, a.sry, a.ncls);
    const double tstart = *a.t_in;
    const int band = blockIdx.z * gridDim.y + blockIdx.y;  // (z: beyond 65535 rows of strips)
    const int y0 = band * a.ky * a.sry;
    if (y0 >= a.ny) return;
    if (threadIdx.x == 0 && blockIdx.x == 0 && band == 0) *a.t_out = tstart + a.dt;
    RowStrip<T, MODE, NW, WIDTH, FULL> s(a, sm, row_smem);
    s.run(blockIdx.x * a.kx * a.srx, y0, tstart);
    const int stw = __reduce_or_sync(0xffffffffu, s.st);
    if ((threadIdx.x & 31) == 0 && stw) atomicOr(a.status, stw);
}

// the kernel of a mode, a parity of the mesh width, and the full step or psi
// alone
using RowKernel = void (*)(const StepArgs);
template <typename T, bool FULL>
RowKernel row_kernel_of(int mode, bool even) {
    switch (mode) {
        case ROW_NC: return even ? k_fire_warp<T, ROW_NC, WIDTH_EVEN, FULL> : k_fire_warp<T, ROW_NC, WIDTH_ODD, FULL>;
        case ROW_MULT:
            return even ? k_fire_warp<T, ROW_MULT, WIDTH_EVEN, FULL> : k_fire_warp<T, ROW_MULT, WIDTH_ODD, FULL>;
        default:
            return even ? k_fire_warp<T, ROW_PLAIN, WIDTH_EVEN, FULL> : k_fire_warp<T, ROW_PLAIN, WIDTH_ODD, FULL>;
    }
}
template <typename T>
RowKernel row_kernel(int mode, bool even, bool full) {
    return full ? row_kernel_of<T, true>(mode, even) : row_kernel_of<T, false>(mode, even);
}

template <typename T>
size_t warp_smem_bytes(int ky, int sry, int ncls) {
    return RowSmem<T, kRowWarps>::bytes(ky, sry, ncls);
}

// raised monotonically, kernel by kernel as each is first launched (setting
// it loads the kernel, a third of a millisecond): the limit is shared by every
// context in the process
template <typename T>
cudaError_t prepare_row_kernel(int mode, bool even, bool full, size_t smem_bytes) {
    static std::mutex mu;
    static size_t current[kMaxDevices][12] = {};  // per device (the attribute is)
    std::lock_guard<std::mutex> lock(mu);
    const int dev = attr_device(), k = mode * 4 + (even ? 2 : 0) + (full ? 1 : 0);
    if (dev >= 0 && smem_bytes <= current[dev][k]) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(row_kernel<T>(mode, even, full),
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes);
    if (e == cudaSuccess && dev >= 0) current[dev][k] = smem_bytes;
    return e;
}

template <typename T>
cudaError_t launch_warp(const StepArgs &args, cudaStream_t s) {
    StepArgs a = args;
    const int W = a.kx * a.srx;
    if (W > kWarpMaxColumns || (W & 1) || W < 2 || a.ky * a.sry > kWarpMaxRows ||
        (long long)a.nx * a.ny > kWarpMaxNodes)
        return cudaErrorInvalidValue;
    a.ky = row_strip_bands(sizeof(T) == 8, a.ky, a.sry);
    const int L = a.ky * a.sry;
    const unsigned bands = (a.ny + L - 1) / L, rows = bands < 65535u ? bands : 65535u;
    const dim3 grid((a.nx + W - 1) / W, rows, (bands + rows - 1) / rows);
    const size_t smem = warp_smem_bytes<T>(a.ky, a.sry, a.ncls);
    const int mode = a.nco[0] ? ROW_NC : a.mult ? ROW_MULT : ROW_PLAIN;
    const bool even = (a.nx & 1) == 0, full = a.F_out != nullptr;
    const cudaError_t e = prepare_row_kernel<T>(mode, even, full, smem);
    if (e != cudaSuccess) return e;
    row_kernel<T>(mode, even, full)<<<grid, 32 * kRowWarps, smem, s>>>(a);
    return cudaGetLastError();
}

#define WF_INSTANTIATE_WARP(T)                                          \
    template size_t warp_smem_bytes<T>(int, int, int);                  \
    template cudaError_t launch_warp<T>(const StepArgs &, cudaStream_t);

}  // namespace wf
