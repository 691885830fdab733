// The coefficient chain of Table 2, shared by the kernels of coeffs.cu and the
// allocation-free step.
//
// The chain's powers and exponentials (some 16 calls of a hundred FP64
// instructions each) are its whole cost, and in one thread a serial one: 41 us
// for a class table.  What depends on the class alone is formed by a group of
// eight lanes, one call of pow and one of exp each (class_terms); what depends
// on the moisture too by one thread per node (moisture_chain: five calls) or by
// the same eight lanes (class_chain: two).
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include "fire_internal.h"

namespace wf {
namespace coefs {

constexpr double kFt = 0.3048;          // m per ft
constexpr double kLb = 0.45359237;      // kg per lb
constexpr double kBtu = 1055.05585262;  // J per BTU
constexpr double kLatent = 2.5e6;       // L (J/kg)
constexpr double kWindMax = 30.0;       // m/s

// Scalars of the chain: double, or a forward-mode dual number (value and
// derivative with respect to the fuel moisture M_f) for the adjoint.
struct Dual {
    double v, d;
};
__device__ __forceinline__ Dual mk(double v, double d) { return Dual{v, d}; }
__device__ __forceinline__ Dual operator+(Dual a, Dual b) { return mk(a.v + b.v, a.d + b.d); }
__device__ __forceinline__ Dual operator-(Dual a, Dual b) { return mk(a.v - b.v, a.d - b.d); }
// (the derivatives' products are contracted one way only: per class and per
// node, the chain gives the same bits)
__device__ __forceinline__ Dual operator*(Dual a, Dual b) {
    return mk(a.v * b.v, fma(a.d, b.v, a.v * b.d));
}
__device__ __forceinline__ Dual operator/(Dual a, Dual b) {
    return mk(a.v / b.v, fma(a.d, b.v, -(a.v * b.d)) / (b.v * b.v));
}
__device__ __forceinline__ Dual operator+(Dual a, double b) { return mk(a.v + b, a.d); }
__device__ __forceinline__ Dual operator+(double a, Dual b) { return mk(a + b.v, b.d); }
__device__ __forceinline__ Dual operator-(double a, Dual b) { return mk(a - b.v, -b.d); }
__device__ __forceinline__ Dual operator*(Dual a, double b) { return mk(a.v * b, a.d * b); }
__device__ __forceinline__ Dual operator*(double a, Dual b) { return mk(a * b.v, a * b.d); }
__device__ __forceinline__ Dual operator/(Dual a, double b) { return mk(a.v / b, a.d / b); }
__device__ __forceinline__ Dual operator/(double a, Dual b) {
    return mk(a / b.v, -a * b.d / (b.v * b.v));
}
__device__ __forceinline__ Dual pow_c(Dual a, double p) {  // a.v > 0
    const double v = pow(a.v, p);
    return mk(v, p * (v / a.v) * a.d);
}
__device__ __forceinline__ double pow_c(double a, double p) { return pow(a, p); }
__device__ __forceinline__ Dual exp_s(Dual a) {
    const double e = exp(a.v);
    return mk(e, e * a.d);
}
__device__ __forceinline__ double exp_s(double a) { return exp(a); }
__device__ __forceinline__ double val(Dual a) { return a.v; }
__device__ __forceinline__ double val(double a) { return a; }
template <typename S>
__device__ __forceinline__ S constant(double x);
template <>
__device__ __forceinline__ double constant<double>(double x) { return x; }
template <>
__device__ __forceinline__ Dual constant<Dual>(double x) { return mk(x, 0.0); }

__device__ __forceinline__ double from_lane(double x, int l) { return __shfl_sync(0xffffffffu, x, l); }

// what the chain takes from the class alone
struct ClassTerms {
    double load, dep, rhoP, heat, bop, gmax, A, wst, mce, etaS, xk, xd, epsh, B, C, cw, E;
    double fgi, cmb, Tf;
    int kind;  // 0 Rothermel, 1 chaparral, 2 no fuel
};

// called by all lanes of a warp, eight lanes per class (q: lane of the group)
__device__ __forceinline__ void class_terms(const fire_fuel_class &f, ClassTerms &o) {
    const int q = threadIdx.x & 7, g = threadIdx.x & 24;
    o.fgi = f.fgi;
    o.cmb = f.cmbcnst;
    o.Tf = f.weight_is_tf ? f.weight : f.weight / (-1000.0 * log(0.6) / 600.0);
    o.kind = f.chaparral ? 1 : (f.fgi > 0.0 ? 0 : 2);
    // English units
    const double sig = f.savr * kFt;               // 1/ft
    o.load = f.fgi * kFt * kFt / kLb;              // lb/ft^2
    o.dep = f.fueldepthm / kFt;                    // ft
    o.rhoP = f.fueldens * kFt * kFt * kFt / kLb;   // lb/ft^3
    o.heat = f.cmbcnst * kLb / kBtu;               // BTU/lb
    const double ex = q == 0 ? -0.8189 : q == 1 ? 1.5 : q == 2 ? 0.1 : q == 3 ? -0.19 : q == 4 ? 0.54 : 0.55;
    const double pw = pow(q == 3 ? f.se : sig, ex);
    auto from = [&](double x, int k) { return __shfl_sync(0xffffffffu, x, g + k); };
    o.bop = 3.348 * from(pw, 0);
    const double sig15 = from(pw, 1);
    o.gmax = sig15 / (495.0 + 0.0594 * sig15);
    o.A = 1.0 / (4.77 * from(pw, 2) - 7.27);
    o.etaS = 0.174 * from(pw, 3);
    o.B = 0.02526 * from(pw, 4);
    const double sig55 = from(pw, 5);
    const double e = exp(q == 0 ? -138.0 / sig : q == 1 ? -3.59e-4 * sig : -0.133 * sig55);
    o.epsh = from(e, 0);
    o.E = 0.715 * from(e, 1);
    o.C = 7.47 * from(e, 2);
    o.cw = pow(f.windrf * (60.0 / kFt), o.B);
    o.wst = 1.0 + f.st;
    o.mce = f.fuelmce;
    o.xk = 0.792 + 0.681 * sqrt(sig);
    o.xd = 192.0 + 0.2595 * sig;
}

// The chain at moisture Mf.  GROUP: by the eight lanes of class_terms (one
// call of pow and exp for them together), else by one thread; co receives the
// K_N slots.
template <bool GROUP, typename S>
__device__ __forceinline__ void moisture_chain(const ClassTerms &f, S Mf, S *co) {
    co[K_TF] = constant<S>(f.Tf);
    co[K_HS] = f.fgi * f.cmb / (1.0 + Mf);
    co[K_HQ] = (Mf + 0.56) / (1.0 + Mf) * kLatent * f.fgi;
    if (!GROUP && f.kind) {
        co[K_S0] = constant<S>(f.kind == 1 ? 0.03333 : 0.0);
        co[K_R0] = constant<S>(0.0);
        co[K_B] = constant<S>(1.0);
        co[K_C] = constant<S>(f.kind == 1 ? 1.2974 : 0.0);
        co[K_D] = constant<S>(0.0);
        co[K_E] = constant<S>(f.kind == 1 ? 6.0 / 1.2974 : kWindMax);
        return;
    }
    co[K_S0] = constant<S>(0.0);
    co[K_E] = constant<S>(kWindMax);
    // packing
    const S w0 = f.load / (1.0 + Mf);
    const S rhob = w0 / f.dep;
    const S beta = rhob / f.rhoP;
    const S rel = beta / f.bop;
    // reaction intensity
    S relA, relE, beta3, eA, ex;
    if constexpr (GROUP) {
        const int q = threadIdx.x & 7, g = threadIdx.x & 24;
        const S p = pow_c(q == 2 ? beta : rel, q == 0 ? f.A : q == 1 ? -f.E : -0.3);
        const S e = exp_s(q == 0 ? f.A * (1.0 - rel) : f.xk * (beta + 0.1));
        relA = from_lane(p, g);
        relE = from_lane(p, g + 1);
        beta3 = from_lane(p, g + 2);
        eA = from_lane(e, g);
        ex = from_lane(e, g + 1);
    } else {
        relA = pow_c(rel, f.A);
        relE = pow_c(rel, -f.E);
        beta3 = pow_c(beta, -0.3);
        eA = exp_s(f.A * (1.0 - rel));
        ex = exp_s(f.xk * (beta + 0.1));
    }
    const S gam = f.gmax * relA * eA;
    const S wn = w0 / f.wst;
    const S x = Mf / f.mce;
    S etaM = 1.0 - 2.59 * x + 5.11 * x * x - 3.52 * x * x * x;
    if (val(x) >= 1.0 || val(etaM) < 0.0) etaM = constant<S>(0.0);
    if (val(etaM) > 1.0) etaM = constant<S>(1.0);
    const S IR = gam * wn * f.heat * etaM * f.etaS;
    // propagating flux, heat sink
    const S xi = ex / f.xd;
    const S Qig = 250.0 + 1116.0 * Mf;
    const S R0 = IR * xi / (rhob * f.epsh * Qig) * (kFt / 60.0);  // ft/min -> m/s
    // wind and slope factors
    co[K_R0] = R0;
    co[K_B] = constant<S>(f.B);
    co[K_C] = R0 * f.C * f.cw * relE;
    co[K_D] = R0 * 5.275 * beta3;
    if (GROUP && f.kind) {  // (the lanes of other classes of the warp took the calls above with these)
        co[K_S0] = constant<S>(f.kind == 1 ? 0.03333 : 0.0);
        co[K_R0] = constant<S>(0.0);
        co[K_B] = constant<S>(1.0);
        co[K_C] = constant<S>(f.kind == 1 ? 1.2974 : 0.0);
        co[K_D] = constant<S>(0.0);
        co[K_E] = constant<S>(f.kind == 1 ? 6.0 / 1.2974 : kWindMax);
    }
}

// the coefficients of class k of n (K_N slots), eight lanes per class, by a
// CTA of at least 8 n threads, whole warps; moist turns a class's moisture into
// an S.  Dual numbers take the chain as a node does (each lane all of it).
template <typename S, typename F>
__device__ __forceinline__ void class_chain(const fire_fuel_class *cls, int n, S (&co)[K_N], F moist) {
    const int k = threadIdx.x >> 3;
    const fire_fuel_class f = cls[k < n ? k : n - 1];
    ClassTerms t;
    class_terms(f, t);
    moisture_chain<sizeof(S) == sizeof(double), S>(t, moist(f.fuelmc_g), co);
}

}  // namespace coefs
}  // namespace wf
