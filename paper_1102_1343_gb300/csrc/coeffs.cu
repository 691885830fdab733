// Fuel-class properties (Table 1) -> the coefficients of eq.
// (spread-WRF-Fire), the burn time T_f and the heat factors of eqs.
// (sensible-heat-flux), (latent-heat-flux), per class or per node, FP64.
//
// The Rothermel chain of Table 2 runs in English units (the caption of
// Table 2 converts inputs from metric); the spread rate is
//   S = R0 (1 + phi_W + phi_S),  phi_W = C U_a^B (beta/beta_op)^(-E),
//   phi_S = 5.275 beta^(-0.3) tan^2(phi),  U_a = a U,
// with the CAWFE limits 0 <= U <= 30 m/s and tan(phi) >= 0, which gives the
// coefficient form S = max{S0, R0 + c min{e, max{0,U}}^b + d max{0,tan}^2}
// with b = B, c = R0 C (a * 196.85)^B (beta/beta_op)^(-E), d = 5.275 R0
// beta^(-0.3), e = 30 m/s, S0 = 0 (SI, U in m/s).  Chaparral (eq. chapparal):
// S0 = 0.03333, R0 = 0, b = 1, c = 1.2974, d = 0, e = 6/1.2974.
// Readings of the table's garbled entries: Gamma_max uses Rothermel's
// constant 0.0594; Q_ig = 250 + 1116 M_f; B = 0.02526 sigma^0.54 and
// beta_op = 3.348 sigma^(-0.8189).  eta_M is clamped to [0, 1]; a class
// without fuel load does not spread.
#include "coeffs.cuh"

namespace wf {

using namespace coefs;

namespace {

constexpr int kClassThreads = 8 * FIRE_MAX_CLASSES;

__global__ void __launch_bounds__(kClassThreads) k_coefficients(const fire_fuel_class *cls, int n, double *coef) {
    double co[K_N];
    class_chain<double>(cls, n, co, [](double m) { return m; });
    const int k = threadIdx.x >> 3;
    if ((threadIdx.x & 7) == 0 && k < n)
        for (int q = 0; q < K_N; ++q) coef[(size_t)k * K_N + q] = co[q];
}

// d(coefficients)/d(M_f) at the class moisture (clamped branches of eta_M
// and the chaparral rule have derivative 0)
__global__ void __launch_bounds__(kClassThreads) k_coefficients_dMf(const fire_fuel_class *cls, int n, double *dcoef) {
    Dual co[K_N];
    class_chain<Dual>(cls, n, co, [](double m) { return mk(m, 1.0); });
    const int k = threadIdx.x >> 3;
    if ((threadIdx.x & 7) == 0 && k < n)
        for (int q = 0; q < K_N; ++q) dcoef[(size_t)k * K_N + q] = co[q].d;
}

// Per-node coefficients for a per-node fuel moisture M_f (Table 1 M_f per
// grid point; eq. spread-WRF-Fire keeps its coefficients per node): the
// chain of the node's class at the node's moisture (the class moisture where
// moist is null).  R0, c, d and the two heat factors depend on M_f; S0, b, e
// and T_f do not and stay in the class table.  Planes in the path precision:
// values R0, c, d, H_s, H_q, or (deriv) the derivatives of R0, c, d.  Bound by
// the FP64 pipe: the terms of the classes are formed once per CTA, each node
// then takes 5 of the chain's 16 powers and exponentials (510x510 nodes: 586
// us for the values and 746 for the derivatives before, each node taking all).
template <typename T>
struct Planes5 {
    T *p[5];
};
constexpr int kNodeThreads = 256;

template <typename T, bool DERIV>
__global__ void __launch_bounds__(kNodeThreads) k_node_coefficients(const fire_fuel_class *cls, int ncls,
                                                                    const uint8_t *fuel, const T *moist, size_t n,
                                                                    const Planes5<T> pl) {
    __shared__ ClassTerms terms[FIRE_MAX_CLASSES];
    __shared__ double mc[FIRE_MAX_CLASSES];
    for (int k0 = 0; k0 < ncls; k0 += kNodeThreads / 8) {
        const int k = k0 + (threadIdx.x >> 3);
        const fire_fuel_class f = cls[k < ncls ? k : ncls - 1];
        ClassTerms t;
        class_terms(f, t);
        if ((threadIdx.x & 7) == 0 && k < ncls) {
            terms[k] = t;
            mc[k] = f.fuelmc_g;
        }
    }
    __syncthreads();
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x) {
        int c = fuel[k];
        c = c < ncls ? c : ncls - 1;
        const double M = moist ? (double)moist[k] : mc[c];
        if constexpr (DERIV) {
            Dual co[K_N];
            moisture_chain<false, Dual>(terms[c], mk(M, 1.0), co);
            pl.p[0][k] = T(co[K_R0].d);
            pl.p[1][k] = T(co[K_C].d);
            pl.p[2][k] = T(co[K_D].d);
        } else {
            double co[K_N];
            moisture_chain<false, double>(terms[c], M, co);
            pl.p[0][k] = T(co[K_R0]);
            pl.p[1][k] = T(co[K_C]);
            pl.p[2][k] = T(co[K_D]);
            pl.p[3][k] = T(co[K_HS]);
            pl.p[4][k] = T(co[K_HQ]);
        }
    }
}

// CTAs that stay (the terms of the classes are formed by each)
int node_grid(size_t n) {
    const size_t b = (n + kNodeThreads - 1) / kNodeThreads;
    return (int)(b < 152 * 4 ? b : 152 * 4);
}

}  // namespace

template <typename T>
cudaError_t launch_node_coefficients(const fire_fuel_class *classes_dev, int ncls, const uint8_t *fuel,
                                     const void *moist, size_t n, T *const *planes, bool deriv, cudaStream_t s) {
    Planes5<T> pl;
    for (int q = 0; q < 5; ++q) pl.p[q] = q < 3 || !deriv ? planes[q] : nullptr;
    if (deriv)
        k_node_coefficients<T, true><<<node_grid(n), kNodeThreads, 0, s>>>(classes_dev, ncls, fuel,
                                                                           static_cast<const T *>(moist), n, pl);
    else
        k_node_coefficients<T, false><<<node_grid(n), kNodeThreads, 0, s>>>(classes_dev, ncls, fuel,
                                                                            static_cast<const T *>(moist), n, pl);
    return cudaGetLastError();
}
template cudaError_t launch_node_coefficients<float>(const fire_fuel_class *, int, const uint8_t *, const void *,
                                                     size_t, float *const *, bool, cudaStream_t);
template cudaError_t launch_node_coefficients<double>(const fire_fuel_class *, int, const uint8_t *, const void *,
                                                      size_t, double *const *, bool, cudaStream_t);

cudaError_t launch_coefficients(const fire_fuel_class *classes_dev, int n, double *coef_dev,
                                cudaStream_t s) {
    k_coefficients<<<1, ((8 * n + 31) / 32) * 32, 0, s>>>(classes_dev, n, coef_dev);
    return cudaGetLastError();
}

cudaError_t launch_coefficients_dMf(const fire_fuel_class *classes_dev, int n, double *dcoef_dev,
                                    cudaStream_t s) {
    k_coefficients_dMf<<<1, ((8 * n + 31) / 32) * 32, 0, s>>>(classes_dev, n, dcoef_dev);
    return cudaGetLastError();
}

}  // namespace wf
