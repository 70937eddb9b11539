// Pointwise energy densities and potentials (Sec. 2 and Sec. 3.3.1), device side.
#pragma once

#include <cuda_runtime.h>

namespace of {

// C_F = (3/10)(3 pi^2)^{2/3}  (Eq. LR:KineticEnergy)
constexpr double OF_CF = 2.8712340001881915;
// (3/pi)^{1/3}, the exchange prefactor of V_x (Sec. 3.3.1); eps_x carries 3/4 of it
constexpr double OF_CX = 0.98474502184269654;
// (3/(4 pi))^{1/3}: r_s = OF_RS0 * rho^{-1/3}
constexpr double OF_RS0 = 0.62035049089940009;
constexpr double OF_RHO_FLOOR = 1e-24;   // xc terms use max(rho, floor)
constexpr double OF_U_FLOOR = 1e-12;     // negative powers of u use max(u, floor)

// Perdew-Zunger constants as printed in Sec. 2
constexpr double PZ_G1 = -0.1423, PZ_B1 = 1.0529, PZ_B2 = 0.3334;
constexpr double PZ_A1 = 0.0311, PZ_BB1 = -0.048, PZ_C1 = 0.002, PZ_D1 = -0.0116;

// rho^{-1/3} by Newton's method for f(t) = t^{-3} - rho, t <- t (4 - rho t^3) / 3, from a
// single-precision seed; the error squares each step (1e-7 -> 1e-14 -> rounding), so two
// FP64 steps reach full double accuracy at a fraction of the cost of a double cube root.
__device__ __forceinline__ double inv_cbrt(double rho) {
    double t = (double)rcbrtf((float)rho);
#pragma unroll
    for (int k = 0; k < 2; ++k) t = t * (4.0 - rho * t * t * t) * (1.0 / 3.0);
    return t;
}

// sqrt(x) = x / sqrt(x) with 1/sqrt(x) from Newton's method y <- y (3 - x y^2) / 2 on a
// single-precision seed (two FP64 steps)
__device__ __forceinline__ double sqrt_newton(double x) {
    double y = (double)rsqrtf((float)x);
#pragma unroll
    for (int k = 0; k < 2; ++k) y = y * (1.5 - 0.5 * x * y * y);
    return x * y;
}

// e = eps_xc(rho) * rho and v = V_xc(rho) for the exchange (Slater) and PZ correlation.
__device__ __forceinline__ void lda_xc(double rho, double& e, double& v) {
    const double r = fmax(rho, OF_RHO_FLOOR);
    const double t = inv_cbrt(r);                   // rho^{-1/3}
    const double c = r * t * t;                     // rho^{1/3} = u^{2/3}
    const double ex = -0.75 * OF_CX * c;            // eps_x
    const double vx = -OF_CX * c;                   // V_x
    const double rs = OF_RS0 * t;
    double ec, vc;
    if (rs >= 1.0) {
        const double sq = sqrt_newton(rs);
        const double den = 1.0 + PZ_B1 * sq + PZ_B2 * rs;
        ec = PZ_G1 / den;
        vc = (PZ_G1 + (7.0 / 6.0) * PZ_G1 * PZ_B1 * sq + (4.0 / 3.0) * PZ_G1 * PZ_B2 * rs) / (den * den);
    } else {
        const double lr = log(rs);
        ec = PZ_A1 * lr + PZ_BB1 + PZ_C1 * rs * lr + PZ_D1 * rs;
        vc = (PZ_A1 + (2.0 / 3.0) * PZ_C1 * rs) * lr + (PZ_BB1 - PZ_A1 / 3.0) +
             (1.0 / 3.0) * (2.0 * PZ_D1 - PZ_C1) * rs;
    }
    e = (ex + ec) * r;
    v = vx + vc;
}

// Thomas-Fermi: energy density C_F rho^{5/3} and V_TF = (5/3) C_F rho^{2/3}
__device__ __forceinline__ void thomas_fermi(double rho, double& e, double& v) {
    if (!(rho > 1e-30)) { e = 0.0; v = 0.0; return; }   // below 1e-50 Ha per point
    const double t = inv_cbrt(rho);
    const double c = rho * t * t;                   // rho^{1/3}
    const double c2 = c * c;
    e = OF_CF * rho * c2;
    v = (5.0 / 3.0) * OF_CF * c2;
}

// ---- TF and xc at a density given by its amplitude, rho = c2 x^2
// The forms that the minimisation evaluates at every point, hundreds of times per ground state.
// GB300 runs FP64 at 2 operations per clock and SM, so these are bound by their count: with t =
// x^{-1/3} every power needed is a product (rho^{1/3} = c2^{1/3} x t, sqrt(r_s) = ks t), one root
// stands for the cube root and the square root of lda_xc, each Newton step is of third order (one
// step from a single-precision seed: 1e-7 -> 1e-21), and seeds are converted by integer shifts
// (an FP64 conversion costs as much as a multiply-add).  29 FP64 operations per point of the
// line's energy and slope where two roots, a reciprocal and three conversions took 65: 112 -> 65
// us on 96^3; the Hamiltonian's sweep, which also divided, 132 -> 72 us.
struct XcScale {
    double c2, k3, ks, lo;   // c2^{1/3}, sqrt(OF_RS0) c2^{-1/6}, the least x taken here
};
inline XcScale xc_scale(double c2) {
    const double k3 = cbrt(c2);
    // rho >= 100 OF_RHO_FLOOR, and x far from the ends of single precision
    return {c2, k3, sqrt(OF_RS0 / k3), fmax(1e-11, 1e-11 / sqrt(c2))};
}
// positive values inside the normal range of single precision
__device__ __forceinline__ float narrow_positive(double v) {   // truncated
    return __uint_as_float((((unsigned)__double2hiint(v) - (896u << 20)) << 3) | ((unsigned)__double2loint(v) >> 29));
}
__device__ __forceinline__ double widen_positive(float v) {
    const unsigned b = __float_as_uint(v);
    return __hiloint2double((int)((b >> 3) + (896u << 20)), (int)(b << 29));
}
// rho^{1/3}, eps_c and V_c at rho = c2 x^2; false (nothing computed) outside lo <= x <= 1e15
__device__ __forceinline__ bool xc_of_amplitude(double x, const XcScale& S, double& c, double& ec, double& vc) {
    if (!(x >= S.lo && x <= 1e15)) return false;
    double t = widen_positive(rcbrtf(narrow_positive(x)));
    const double e = fma(-x, t * t * t, 1.0);       // x^{-1/3} = t (1 - e)^{-1/3}
    t = fma(t, e * fma(e, 2.0 / 9.0, 1.0 / 3.0), t);
    c = S.k3 * (x * t);
    const double sq = S.ks * t;                     // sqrt(r_s)
    if (sq >= 1.0) {
        const double den = fma(sq, fma(PZ_B2, sq, PZ_B1), 1.0);
        double inv = widen_positive(__frcp_rn(narrow_positive(den)));
        const double f = fma(-den, inv, 1.0);       // 1 / den = inv / (1 - f)
        inv = fma(inv, fma(f, f, f), inv);
        ec = PZ_G1 * inv;
        vc = ec * inv * fma(sq, fma((4.0 / 3.0) * PZ_B2, sq, (7.0 / 6.0) * PZ_B1), 1.0);
    } else {
        const double rs = sq * sq;
        const double lr = log(rs);
        ec = PZ_A1 * lr + PZ_BB1 + PZ_C1 * rs * lr + PZ_D1 * rs;
        vc = (PZ_A1 + (2.0 / 3.0) * PZ_C1 * rs) * lr + (PZ_BB1 - PZ_A1 / 3.0) +
             (1.0 / 3.0) * (2.0 * PZ_D1 - PZ_C1) * rs;
    }
    return true;
}
// v = V_TF + V_xc and the energy densities per rho: eps = C_F rho^{2/3} + eps_xc
__device__ __forceinline__ void tf_xc_of_amplitude(double w, const XcScale& S, double& eps, double& v) {
    double c, ec, vc;
    if (xc_of_amplitude(fabs(w), S, c, ec, vc)) {
        eps = fma(c, fma(OF_CF, c, -0.75 * OF_CX), ec);
        v = fma(c, fma((5.0 / 3.0) * OF_CF, c, -OF_CX), vc);
    } else {   // a vanishing density: the floors of the separate forms
        const double rho = S.c2 * w * w, r = fmax(rho, OF_RHO_FLOOR);
        double etf, vtf, exc, vxc;
        thomas_fermi(rho, etf, vtf);
        lda_xc(rho, exc, vxc);
        eps = rho > 0.0 ? etf / rho + exc / r * (r / rho) : 0.0;
        v = vtf + vxc;
    }
}

}  // namespace of
