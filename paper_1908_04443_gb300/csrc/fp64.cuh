// FP64 arithmetic of the step, written for few FP64 instructions.
//
// GB300's FP64 pipe issues about 1.7 lane operations per clock and SM (lbm_probe_fp64_rate), 1/76 of the
// FP32 rate: the FP64 kernels are bound by the count of FP64 instructions and by nothing else, integer
// and memory work beside them being free.  The functions here are the ones of the FP32 path and of the
// adjoint (psi_arg, collide_d2q9) with the same mathematics in fewer operations:
//   * psi = sqrt(num / den) = |num| rsqrt(num den): one reciprocal square root in place of a division
//     (two with Peng-Robinson) and a square root, 2/G folded into the equation of state's constants;
//   * |F_m|^2 / psi^2 = |G sum w psi(x + e) e|^2 (F_m carries the factor psi): no division;
//   * rho u = j + F/2 is used as it stands wherever rho u appears, and rho u_i u_j = (rho u_i) u_j;
//   * relaxation rates folded with the row norms of M, sums and differences of opposite populations
//     shared between density, momentum and moments.
// One bulk D2Q9 node takes 26 FP64 instructions for density and psi and 110 for the rest, against about
// 230 for the general functions (from the FP64 pipe's utilisation): the 24-grid 600 x 400 sweep's step
// 2509 -> 1522 us, the pipe at 84 % of its nominal 2 operations per clock, the rate of the probe, in both.
// Every operation is written as an explicitly rounded intrinsic, so that the kernels that share these
// functions agree bit for bit.
// In FP64 the stored deviation is the distribution itself (rho_ref = 0).
#pragma once

#include "kernels.h"
#include "lattice.cuh"
#include "tile_common.cuh"

namespace lbmwet {

__device__ __forceinline__ double dadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double dsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double dmul(double a, double b) { return __dmul_rn(a, b); }

// psi of a density (Eq. 6 with Eq. 18 or Carnahan-Starling); a non-positive square-root argument
// flags ERR_PSI and gives 0.
__device__ __forceinline__ double psi64(double x, const Phys<double>& e, unsigned* err) {
    double num, den;
    if (e.eos_kind == 1) {
        // arg = x (k RT poly / om^3 - (k a x + k / 3)), k = 2 / G
        const double om = __fma_rn(-e.b4, x, 1.0), eta = dmul(e.b4, x);
        const double poly = __fma_rn(eta, __fma_rn(eta, om, 1.0), 1.0);   // 1 + eta + eta^2 - eta^3
        den = dmul(dmul(om, om), om);
        const double w = __fma_rn(-e.fold.ka, x, -e.fold.k3);
        num = dmul(x, __fma_rn(w, den, dmul(e.fold.kRT, poly)));
    } else {
        // arg = x (k RT / d1 - k a phi x / d2 - k / 3)
        const double br = dmul(e.b, x), d1 = dsub(1.0, br);
        const double d2 = __fma_rn(br, dsub(2.0, br), 1.0);               // 1 + 2 b x - b^2 x^2
        den = dmul(d1, d2);
        const double s = __fma_rn(e.fold.kRT, d2, -dmul(dmul(e.fold.kaphi, x), d1));
        num = dmul(x, __fma_rn(-e.fold.k3, den, s));
    }
    const double nd = dmul(num, den);   // the sign of the argument
    if (!(nd > 0.0)) {
        atomicOr(err, ERR_PSI);
        return 0.0;
    }
    return dmul(fabs(num), rsqrt(nd));
}

// Density of the nine pulled populations, opposite pairs first (the sums collide2d64 needs again).
__device__ __forceinline__ double density64(const double (&f)[9]) {
    const double s14 = dadd(dadd(f[1], f[3]), dadd(f[2], f[4]));
    const double s58 = dadd(dadd(f[5], f[7]), dadd(f[6], f[8]));
    return dadd(f[0], dadd(s14, s58));
}

// Force, velocity and, with COLLIDE, the MRT collision (Eqs. 2, 4, 5, 7, 8) of one node.  d1, d2, d5, d6:
// psi(x + e_a) - psi(x - e_a) of the directions 1, 2, 5, 6; (ax, ay): sum_a w_a s(x + e_a) e_a of the
// solid-fluid interaction scheme (sf).
template <bool COLLIDE>
__device__ __forceinline__ void node2d64(double (&f)[9], double rho, double d1, double d2, double d5, double d6,
                                         double psi, bool sf, double ax, double ay, const Phys<double>& ph, double& ux,
                                         double& uy) {
    const Fold64& k = ph.fold;
    const double q13 = dsub(f[1], f[3]), q24 = dsub(f[2], f[4]), q57 = dsub(f[5], f[7]), q86 = dsub(f[8], f[6]);
    const double t = dadd(q57, q86), s = dsub(q57, q86);
    const double jx = dadd(q13, t), jy = dadd(q24, s);
    // F_m = psi (gx, gy)
    const double gx = __fma_rn(k.g1, d1, dmul(k.g2, dsub(d5, d6)));
    const double gy = __fma_rn(k.g1, d2, dmul(k.g2, dadd(d5, d6)));
    double Fx = dmul(psi, gx), Fy = dmul(psi, gy);
    if (sf) {
        const double gr = dmul(-ph.wall_param, rho);
        Fx = __fma_rn(gr, ax, Fx);
        Fy = __fma_rn(gr, ay, Fy);
    }
    if (k.body) {
        Fx = dadd(Fx, ph.fx);
        Fy = dadd(Fy, ph.fy);
    }
    // Eq. 4: h = rho u = sum e f + F / 2
    const double hx = __fma_rn(0.5, Fx, jx), hy = __fma_rn(0.5, Fy, jy);
    const double inv = __drcp_rn(rho);
    ux = dmul(hx, inv);
    uy = dmul(hy, inv);
    if constexpr (COLLIDE) {
        const double X = __fma_rn(gx, gx, dmul(gy, gy));
        const double p13 = dadd(f[1], f[3]), p24 = dadd(f[2], f[4]), p57 = dadd(f[5], f[7]), p68 = dadd(f[6], f[8]);
        const double s14 = dadd(p13, p24), s58 = dadd(p57, p68);
        const double m1 = __fma_rn(2.0, s58, __fma_rn(-4.0, f[0], -s14));
        const double m2 = __fma_rn(4.0, f[0], __fma_rn(-2.0, s14, s58));
        const double m4 = __fma_rn(-2.0, q13, t), m6 = __fma_rn(-2.0, q24, s);
        const double rxx = dmul(hx, ux), ryy = dmul(hy, uy);
        const double R = dadd(rxx, ryy), D = dsub(rxx, ryy);              // rho u^2, rho (ux^2 - uy^2)
        const double uFx = dmul(ux, Fx), uFy = dmul(uy, Fy);
        const double uF = dadd(uFx, uFy), dF = dsub(uFx, uFy);
        const double cF = __fma_rn(ux, Fy, dmul(uy, Fx));
        // a_k = (m*_k - m_k) / |row_k|^2; e_eq = -2 rho + 3 rho u^2, eps_eq = rho - 3 rho u^2
        const double E1 = __fma_rn(-3.0, R, __fma_rn(2.0, rho, m1));
        const double E2 = __fma_rn(3.0, R, dsub(m2, rho));
        const double a1 = __fma_rn(k.ke3, X, __fma_rn(k.ke2, uF, dmul(k.ke1, E1)));
        const double a2 = __fma_rn(k.kp3, X, __fma_rn(k.kp2, uF, dmul(k.kp1, E2)));
        const double a4 = __fma_rn(k.kq2, Fx, dmul(k.kq1, dadd(m4, hx)));
        const double a6 = __fma_rn(k.kq2, Fy, dmul(k.kq1, dadd(m6, hy)));
        const double a7 = __fma_rn(k.kn2, dF, dmul(k.kn1, dsub(dsub(p13, p24), D)));
        const double a8 = __fma_rn(k.kh8, cF, dmul(k.kn1, __fma_rn(-hx, uy, dsub(p57, p68))));
        const double a3 = dmul(1.0 / 6.0, Fx), a5 = dmul(1.0 / 6.0, Fy);
        // f += M^T diag(1/|row|^2) (m* - m)
        const double b = __fma_rn(-2.0, a2, -a1), c = __fma_rn(2.0, a1, a2);
        f[0] = __fma_rn(4.0, dsub(a2, a1), f[0]);
        const double r3 = __fma_rn(-2.0, a4, a3), r5 = __fma_rn(-2.0, a6, a5);
        const double bp = dadd(b, a7), bm = dsub(b, a7);
        f[1] = dadd(f[1], dadd(bp, r3));
        f[3] = dadd(f[3], dsub(bp, r3));
        f[2] = dadd(f[2], dadd(bm, r5));
        f[4] = dadd(f[4], dsub(bm, r5));
        const double t1 = dadd(a3, a4), t2 = dadd(a5, a6);
        const double pp = dadd(t1, t2), qq = dsub(t2, t1);
        const double cu = dadd(c, a8), cv = dsub(c, a8);
        f[5] = dadd(f[5], dadd(cu, pp));
        f[7] = dadd(f[7], dsub(cu, pp));
        f[6] = dadd(f[6], dadd(cv, qq));
        f[8] = dadd(f[8], dsub(cv, qq));
    }
}

}  // namespace lbmwet
