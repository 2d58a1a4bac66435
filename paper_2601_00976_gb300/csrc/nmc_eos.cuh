// Synthetic closed-form equation of state on the device (FP64).
//
// Stands in for the tabulated EoS the paper interpolates with weaklib
// (Sec. 3.5.2, paragraph after Eq. eulerianNumberLG): a massless e+e- gas
// (exact Fermi--Dirac moments), a non-degenerate nucleon gas and photons.
//   n_e   = (mu^3 + pi^2 T^2 mu) / (3 pi^2 (hbar c)^3) = rho Ye / m_B
//   u_e   = (7 pi^2 T^4/60 + T^2 mu^2/2 + mu^4/(4 pi^2)) / (hbar c)^3
//   u_N   = 1.5 T rho / m_B,   u_gamma = pi^2 T^4 / (15 (hbar c)^3)
//   eps   = (u_e + u_N + u_gamma) / rho        [erg/g after unit conversion]
//   mu_nue = mu_e - T ln((1-Ye)/Ye) - (m_n - m_p),  mu_anue = -mu_nue, mu_x = 0.
#pragma once

#include "nmc_internal.h"

namespace nmc {

// (float)x and (double)x in integers, the same values bit for bit: a conversion instruction runs on the FP64
// pipe (~64 cycles of an SMSP).  Values whose FP32 form is not a normal number take the instruction.
__device__ __forceinline__ float narrow(double x) {
    const unsigned hi = (unsigned)__double2hiint(x);
    if (((hi >> 20) & 0x7ffu) - 897u > 253u) return (float)x;
    const uint64_t u = word_of(x);
    const uint64_t t = u + 0x0fffffffull + ((u >> 29) & 1u);   // round to nearest, ties to even
    return __uint_as_float(((unsigned)(t >> 29) - (896u << 23)) | (hi & 0x80000000u));
}

__device__ __forceinline__ double widen(float x) {
    const unsigned u = __float_as_uint(x), e = (u >> 23) & 0xffu;
    if (e - 1u > 253u) return (double)x;
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
}

__device__ __forceinline__ double eos_mu_e(double rho, double T, double Ye) {
    const double pi2 = kPi * kPi;
    const double hc3 = kHbarC * kHbarC * kHbarC;
    const double ne = Ye * rho / kMB;
    const double p = pi2 * T * T;
    const double q = -3.0 * pi2 * hc3 * ne;
    // real root of x^3 + p x + q = 0 (p > 0): hyperbolic form of Cardano's solution
    return -2.0 * sqrt(p / 3.0) * sinh(asinh(1.5 * q / p * sqrt(3.0 / p)) / 3.0);
}

// eps(rho, T, Ye) in erg/g and d eps / dT at fixed rho, Ye, given the electron
// chemical potential mu at (rho, T, Ye).
__device__ __forceinline__ void eos_eps_at_mu(double rho, double T, double mu, double* eps, double* deps) {
    const double pi2 = kPi * kPi;
    const double hc3 = kHbarC * kHbarC * kHbarC;
    const double T2 = T * T, mu2 = mu * mu;
    const double ue = (7.0 * pi2 * T2 * T2 / 60.0 + 0.5 * T2 * mu2 + mu2 * mu2 / (4.0 * pi2)) / hc3;
    const double nb = rho / kMB;
    const double ug = pi2 / 15.0 * T2 * T2 / hc3;
    const double f = kMeVErg / rho;
    *eps = (ue + 1.5 * T * nb + ug) * f;
    // mu(T) at fixed n_e: dmu/dT = -(dn/dT)/(dn/dmu) = -2 pi^2 T mu / (3 mu^2 + pi^2 T^2)
    const double dmu = -2.0 * pi2 * T * mu / (3.0 * mu2 + pi2 * T2);
    const double due = (7.0 * pi2 * T2 * T / 15.0 + T * mu2 + (T2 * mu + mu2 * mu / pi2) * dmu) / hc3;
    *deps = (due + 1.5 * nb + 4.0 * pi2 / 15.0 * T2 * T / hc3) * f;
}

__device__ __forceinline__ void eos_eps(double rho, double T, double Ye, double* eps, double* deps) {
    eos_eps_at_mu(rho, T, eos_mu_e(rho, T, Ye), eps, deps);
}

// ---- the same by a whole warp ----
// Every lane passes the same arguments and gets the same results, those of the functions above bit for
// bit.  An FP64 instruction costs an SMSP's pipe ~64 cycles on one lane or on 32, and a division or a
// square root is ten of them; the independent ones of an evaluation go to different lanes and cost as
// one (an evaluation of eps and its derivative: 5 divisions and 1 square root deep instead of 15 and 2).
__device__ __forceinline__ double lane_value(double x, int lane) { return __shfl_sync(0xffffffffu, x, lane); }

// mu_e, and on request 1 / T (in one of the divisions' spare lanes)
__device__ __forceinline__ double eos_mu_e_warp(double ne, double T, double* rT = nullptr) {
    const int ln = threadIdx.x & 31;
    const double pi2 = kPi * kPi;
    const double hc3 = kHbarC * kHbarC * kHbarC;
    const double p = pi2 * T * T;
    const double q = -3.0 * pi2 * hc3 * ne;
    // lane 0: p / 3, 1: 3 / p, 2: 1.5 q / p, 3: 1 / T
    const double num = ln == 0 ? p : (ln == 1 ? 3.0 : (ln == 2 ? 1.5 * q : 1.0));
    const double den = ln == 0 ? 3.0 : (ln == 3 ? T : p);
    const double d = num / den;
    const double r = sqrt(ln < 2 ? d : 1.0);
    if (rT) *rT = lane_value(d, 3);
    return -2.0 * lane_value(r, 0) * sinh(asinh(lane_value(d, 2) * lane_value(r, 1)) / 3.0);
}

// eos_eps_at_mu with nb = rho / m_B and f = (MeV in erg) / rho.  The products and sums are written as the
// fused operations the compiler contracts them to in eos_eps_at_mu, so that both round alike; kShared: where
// pi^2 T^2 is shared with eos_deps_dye_at_mu, it is rounded before it is added.
// kLanes: numerators formed lane-parallel as well (not in the adjoint, where it overruns the narrow register class).
template <bool kShared = false, bool kLanes = true>
__device__ __forceinline__ void eos_eps_at_mu_warp(double nb, double f, double T, double mu, double* eps, double* deps) {
    const int ln = threadIdx.x & 31;
    const double pi2 = kPi * kPi;
    const double hc3 = kHbarC * kHbarC * kHbarC;
    const double T2 = T * T, mu2 = mu * mu;
    // numerators (k x) y, denominators
    double k = 7.0 * pi2, x = T2, y = T2, den = 60.0;
    if (ln == 1) { k = 1.0; x = mu2; y = mu2; den = 4.0 * pi2; }
    if (ln == 2) { k = pi2 / 15.0; den = hc3; }
    if (ln == 3) { k = -2.0 * pi2; x = T; y = mu; den = kShared ? __fma_rn(3.0, mu2, __dmul_rn(pi2, T2)) : __fma_rn(pi2, T2, __dmul_rn(3.0, mu2)); }
    if (ln == 4) { y = T; den = 15.0; }
    if (ln == 5) { k = 1.0; x = mu2; y = mu; den = pi2; }
    if (ln == 6) { k = 4.0 * pi2 / 15.0; y = T; den = hc3; }
    double num = __dmul_rn(__dmul_rn(k, x), y);
    if (!kLanes) {
        num = 7.0 * pi2 * T2 * T2;
        if (ln == 1) num = mu2 * mu2;
        if (ln == 2) num = pi2 / 15.0 * T2 * T2;
        if (ln == 3) num = -2.0 * pi2 * T * mu;
        if (ln == 4) num = 7.0 * pi2 * T2 * T;
        if (ln == 5) num = mu2 * mu;
        if (ln == 6) num = 4.0 * pi2 / 15.0 * T2 * T;
    }
    const double d = num / den;
    const double u1 = lane_value(d, 0), u2 = lane_value(d, 1), ug = lane_value(d, 2), dmu = lane_value(d, 3);
    const double v1 = lane_value(d, 4), v2 = lane_value(d, 5), dug = lane_value(d, 6);
    // lane 0: eps's numerator, the others its derivative's; one more division
    const double un = __dadd_rn(__fma_rn(__dmul_rn(0.5, T2), mu2, u1), u2);
    const double dn = __fma_rn(__fma_rn(T2, mu, v2), dmu, __fma_rn(T, mu2, v1));
    const double w = (ln == 0 ? un : dn) / hc3;
    *eps = __dmul_rn(__dadd_rn(__fma_rn(__dmul_rn(1.5, T), nb, lane_value(w, 0)), ug), f);
    *deps = __dmul_rn(__dadd_rn(__fma_rn(1.5, nb, lane_value(w, 1)), dug), f);
}

// T with eps(rho, T, Ye) = eps_t: safeguarded Newton in T within [kTMin, kTMax].
// The bracket starts as the whole range without evaluating its ends (a warm
// start from the previous T needs ~3 evaluations); every evaluation narrows it,
// and a Newton step that leaves it is replaced by a geometric bisection.
// eps is strictly increasing in T, so an eps_t outside [eps(kTMin), eps(kTMax)]
// drives the iterate to a range end: *ok = false and T clamped there.
__device__ inline double eos_temperature(double rho, double eps_t, double Ye, double T0, bool* ok) {
    *ok = true;
    if (!(Ye > 0.0 && Ye < 1.0) || !isfinite(eps_t)) {
        *ok = false;
        return isfinite(T0) ? T0 : 1.0;
    }
    double lo = kTMin, hi = kTMax, e, de, f = 0.0;
    double T = (T0 > lo && T0 < hi) ? T0 : sqrt(lo * hi);
    for (int it = 0; it < 300; ++it) {
        eos_eps(rho, T, Ye, &e, &de);
        f = e - eps_t;
        if (f > 0.0) hi = T; else lo = T;
        if (f == 0.0) break;
        double Tn = T - f / de;
        if (!(Tn > lo && Tn < hi)) Tn = hi > 2.0 * lo ? sqrt(lo * hi) : 0.5 * (lo + hi);
        const double d = fabs(Tn - T);
        T = Tn;
        if (d <= 2e-16 * T || hi - lo <= 4e-16 * hi) break;
    }
    if (f > 0.0 && T <= kTMin * (1.0 + 1e-12)) {   // eps_t below eps(kTMin)
        eos_eps(rho, kTMin, Ye, &e, &de);
        if (eps_t <= e) { *ok = false; return kTMin; }
    }
    if (f < 0.0 && T >= kTMax * (1.0 - 1e-12)) {   // eps_t above eps(kTMax)
        eos_eps(rho, kTMax, Ye, &e, &de);
        if (eps_t >= e) { *ok = false; return kTMax; }
    }
    return T;
}

// eos_temperature by a whole warp (nb = rho / m_B, f = (MeV in erg) / rho); the comparisons of the
// positive T and its bracket on the integer pipe.  mu_T: (T, Ye, mu_e) of the last evaluation.
__device__ inline double eos_temperature_warp(double rho, double nb, double f, double eps_t, double Ye, double T0, bool* ok,
                                              double* mu_T) {
    *ok = true;
    auto bits = [](double x) { return __double_as_longlong(x); };   // orders positive doubles; negatives and -NaN below them
    if (!(Ye > 0.0 && Ye < 1.0) || !isfinite(eps_t)) {
        *ok = false;
        return isfinite(T0) ? T0 : 1.0;
    }
    const double ne = Ye * rho / kMB;
    double lo = kTMin, hi = kTMax, e, de, r = 0.0, mu = 0.0;
    double T = (T0 > lo && T0 < hi) ? T0 : sqrt(lo * hi), Te = T;
    for (int it = 0; it < 300; ++it) {
        mu = eos_mu_e_warp(ne, T);
        Te = T;
        eos_eps_at_mu_warp(nb, f, T, mu, &e, &de);
        r = __dsub_rn(e, eps_t);
        const long long rb = bits(r);
        if (rb > 0 && rb <= 0x7ff0000000000000ll) hi = T; else lo = T;   // r > 0
        if ((rb << 1) == 0) break;                                      // r == 0
        double Tn = T - r / de;
        if (!(bits(Tn) > bits(lo) && bits(Tn) < bits(hi))) Tn = hi > 2.0 * lo ? sqrt(lo * hi) : 0.5 * (lo + hi);
        const double d = fabs(Tn - T);
        T = Tn;
        if (bits(d) <= bits(2e-16 * T) || bits(hi - lo) <= bits(4e-16 * hi)) break;
    }
    if (mu_T) { mu_T[0] = Te; mu_T[1] = Ye; mu_T[2] = mu; }
    if (r > 0.0 && T <= kTMin * (1.0 + 1e-12)) {   // eps_t below eps(kTMin)
        eos_eps(rho, kTMin, Ye, &e, &de);
        if (eps_t <= e) { *ok = false; return kTMin; }
    }
    if (r < 0.0 && T >= kTMax * (1.0 - 1e-12)) {   // eps_t above eps(kTMax)
        eos_eps(rho, kTMax, Ye, &e, &de);
        if (eps_t >= e) { *ok = false; return kTMax; }
    }
    return T;
}

// d eps / dYe at fixed rho, T (kShared: see eos_eps_at_mu_warp)
template <bool kShared = false>
__device__ __forceinline__ double eos_deps_dye_at_mu(double T, double mu) {
    const double pi2 = kPi * kPi;
    const double mu2 = mu * mu, T2 = T * T;
    const double t = __dmul_rn(pi2, T2);
    const double num = kShared ? __dadd_rn(mu2, t) : __fma_rn(pi2, T2, mu2);
    const double den = kShared ? __fma_rn(3.0, mu2, t) : __fma_rn(pi2, T2, __dmul_rn(3.0, mu2));
    return kMeVErg / kMB * 3.0 * mu * num / den;
}

// ---- FP32 variants for the mixed-precision path ----
// Densities are carried times (hbar c)^3 (MeV^3) and energy densities times
// (hbar c)^3 (MeV^4), so every intermediate stays inside FP32 range:
// u (hbar c)^3 = 7 pi^2 T^4/60 + T^2 mu^2/2 + mu^4/(4 pi^2) + 1.5 T nb + pi^2 T^4/15.

struct EosScaleF {
    float nb;      // (rho / m_B) (hbar c)^3
    float ne;      // Ye nb
};

__device__ __forceinline__ float eos_mu_e_f(float ne, float T) {
    const float pi2 = (float)(kPi * kPi);
    const float p = pi2 * T * T;
    const float q = -3.0f * pi2 * ne;
    return -2.0f * sqrtf(p / 3.0f) * sinhf(asinhf(1.5f * q / p * sqrtf(3.0f / p)) / 3.0f);
}

// mu_e in FP64 for the mixed path: the FP32 root of the electron cubic
// x^3 + pi^2 T^2 x - 3 pi^2 n_e (hbar c)^3 = 0 and one FP64 Newton step on it,
// which squares its relative error (~1e-7 to ~1e-14) for a handful of FP64
// operations instead of the closed form's FP64 asinh and sinh.  ne_f: FP32
// n_e (hbar c)^3; nel: Ye rho / m_B.
__device__ __forceinline__ double eos_mu_e_refine(float ne_f, double nel, double T, float Tf) {
    const double m0 = widen(eos_mu_e_f(ne_f, Tf));
    const double pi2T2 = kPi * kPi * T * T;
    const double ned = nel * (kHbarC * kHbarC * kHbarC);   // FP64 target
    const double cub = __fma_rn(m0, __fma_rn(kPi * kPi * T, T, __dmul_rn(m0, m0)), -__dmul_rn(3.0 * kPi * kPi, ned));
    return m0 - cub / __fma_rn(__dmul_rn(3.0, m0), m0, pi2T2);
}

// by a whole warp, with 1 / T
__device__ __forceinline__ double eos_mu_e_refined_warp(double rho, double T, double Ye, double* rT) {
    const int ln = threadIdx.x & 31;
    const double d = (ln == 0 ? rho : (ln == 1 ? Ye * rho : 1.0)) / (ln < 2 ? kMB : T);
    *rT = lane_value(d, 2);
    const double nb = lane_value(d, 0) * (kHbarC * kHbarC * kHbarC);
    return eos_mu_e_refine(narrow(Ye * nb), lane_value(d, 1), T, narrow(T));
}

__device__ __forceinline__ void eos_u_f(const EosScaleF& sc, float T, float* u, float* du) {
    const float pi2 = (float)(kPi * kPi);
    const float mu = eos_mu_e_f(sc.ne, T);
    const float T2 = T * T, mu2 = mu * mu;
    *u = 7.0f * pi2 * T2 * T2 / 60.0f + 0.5f * T2 * mu2 + mu2 * mu2 / (4.0f * pi2) + 1.5f * T * sc.nb +
         pi2 / 15.0f * T2 * T2;
    const float dmu = -2.0f * pi2 * T * mu / (3.0f * mu2 + pi2 * T2);
    *du = 7.0f * pi2 * T2 * T / 15.0f + T * mu2 + (T2 * mu + mu2 * mu / pi2) * dmu + 1.5f * sc.nb +
          4.0f * pi2 / 15.0f * T2 * T;
}

// Temperature for the mixed path, by a whole warp (every lane the same arguments and results):
// bracketed Newton in FP32 to ~1e-7, then one FP64 Newton step on eps(rho, T, Ye) (with mu_e refined
// from its FP32 root), which squares the relative error.  The range's ends and the first iterate are
// evaluated side by side on different lanes.  nb = rho / m_B, f = (MeV in erg) / rho, ku = MeV/erg /
// ((hbar c)^3 rho).
__device__ inline double eos_temperature_mixed_warp(double rho, double nb, double f, double ku, double eps_t, double Ye,
                                                    double T0, bool* ok) {
    *ok = true;
    if (!(Ye > 0.0 && Ye < 1.0) || !isfinite(eps_t)) {
        *ok = false;
        return isfinite(T0) ? T0 : 1.0;
    }
    const int ln = threadIdx.x & 31;
    const double q = (ln == 0 ? eps_t : Ye * rho) / (ln == 0 ? ku : kMB);
    const double nel = lane_value(q, 1), nbh = nb * (kHbarC * kHbarC * kHbarC);
    const float ut = narrow(lane_value(q, 0));
    EosScaleF sc;
    sc.nb = narrow(nbh);
    sc.ne = narrow(Ye * nbh);
    float lo = (float)kTMin, hi = (float)kTMax, u, du;
    float T = (T0 > kTMin && T0 < kTMax) ? narrow(T0) : sqrtf(lo * hi);
    for (int it = 0; it < 100; ++it) {
        eos_u_f(sc, it > 0 || ln > 1 ? T : (ln == 0 ? lo : hi), &u, &du);
        if (it == 0) {
            if (ut <= __shfl_sync(0xffffffffu, u, 0)) { *ok = false; return kTMin; }
            if (ut >= __shfl_sync(0xffffffffu, u, 1)) { *ok = false; return kTMax; }
            u = __shfl_sync(0xffffffffu, u, 2);
            du = __shfl_sync(0xffffffffu, du, 2);
        }
        const float r = u - ut;
        if (r > 0.0f) hi = T; else lo = T;
        if (r == 0.0f) break;
        float Tn = T - r / du;
        if (!(Tn > lo && Tn < hi)) Tn = 0.5f * (lo + hi);
        const float d = fabsf(Tn - T);
        T = Tn;
        if (d <= 2e-7f * T || hi - lo <= 4e-7f * hi) break;
    }
    const double Td = widen(T);
    double e, de;
    eos_eps_at_mu_warp(nb, f, Td, eos_mu_e_refine(sc.ne, nel, Td, T), &e, &de);
    const double Tn = Td - __dsub_rn(e, eps_t) / de;
    return (Tn > kTMin && Tn < kTMax) ? Tn : Td;
}

}  // namespace nmc
