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

// cell k of the one-cell ring of an ax x ay box
__device__ __forceinline__ void ring_cell(int k, int ax, int ay, int& x, int& y) {
    if (k < 2 * ax) {
        y = k < ax ? 0 : ay - 1;
        x = k < ax ? k : k - ax;
    } else {
        const int j = k - 2 * ax;
        y = 1 + (j >> 1);
        x = (j & 1) ? ax - 1 : 0;
    }
}

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
        const double m4 = __fma_rn(-2.0, q13, t), m6 = __fma_rn(-2.0, q24, s);
        const double rxx = dmul(hx, ux), ryy = dmul(hy, uy);
        const double R = dadd(rxx, ryy), D = dsub(rxx, ryy);              // rho u^2, rho (ux^2 - uy^2)
        const double uFx = dmul(ux, Fx), uFy = dmul(uy, Fy);
        const double uF = dadd(uFx, uFy), dF = dsub(uFx, uFy);
        const double cF = __fma_rn(ux, Fy, dmul(uy, Fx));
        // a_k = (m*_k - m_k) / |row_k|^2; with rho = f0 + s14 + s58
        //   e - e_eq = e + 2 rho - 3 rho u^2 = -2 f0 + s14 + 4 s58 - 3 R,
        //   eps - eps_eq = eps - rho + 3 rho u^2 = 3 (f0 - s14 + R)
        const double E1 = __fma_rn(-3.0, R, __fma_rn(4.0, s58, __fma_rn(-2.0, f[0], s14)));
        const double E2 = dadd(dsub(f[0], s14), R);
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

// The same of a D3Q19 node: density (18 FP64 instructions) and force, velocity and collision (247).  d: the psi
// differences of the directions 1, 3, 5, 7, 9, 11, 13, 15, 17.
__device__ __forceinline__ double density64(const double (&f)[19]) {
    const double s16 = dadd(dadd(f[1], f[2]), dadd(dadd(f[3], f[4]), dadd(f[5], f[6])));
    const double exy = dadd(dadd(f[7], f[8]), dadd(f[9], f[10])), exz = dadd(dadd(f[11], f[12]), dadd(f[13], f[14]));
    const double eyz = dadd(dadd(f[15], f[16]), dadd(f[17], f[18]));
    return dadd(f[0], dadd(s16, dadd(dadd(exy, exz), eyz)));
}

template <bool COLLIDE>
__device__ __forceinline__ void node3d64(double (&f)[19], double rho, const double (&d)[9], double psi, bool sf, double ax,
                                         double ay, double az, const Phys<double>& ph, double& ux, double& uy, double& uz) {
    const Fold64& k = ph.fold;
    const double q1 = dsub(f[1], f[2]), q3 = dsub(f[3], f[4]), q5 = dsub(f[5], f[6]);
    const double q7 = dsub(f[7], f[8]), q9 = dsub(f[9], f[10]), q11 = dsub(f[11], f[12]), q13 = dsub(f[13], f[14]);
    const double q15 = dsub(f[15], f[16]), q17 = dsub(f[17], f[18]);
    const double s1 = dadd(q7, q9), s2 = dadd(q11, q13), t1 = dsub(q7, q9), t2 = dadd(q15, q17);
    const double v1 = dsub(q11, q13), v2 = dsub(q15, q17);
    const double Tx = dadd(s1, s2), Ty = dadd(t1, t2), Tz = dadd(v1, v2);
    // F_m = psi (gx, gy, gz), Eq. 5 weights 1/6 and 1/12
    const double gx = __fma_rn(k.g3, d[0], dmul(k.g2, dadd(dadd(d[3], d[4]), dadd(d[5], d[6]))));
    const double gy = __fma_rn(k.g3, d[1], dmul(k.g2, dadd(dsub(d[3], d[4]), dadd(d[7], d[8]))));
    const double gz = __fma_rn(k.g3, d[2], dmul(k.g2, dadd(dsub(d[5], d[6]), dsub(d[7], d[8]))));
    double Fx = dmul(psi, gx), Fy = dmul(psi, gy), Fz = dmul(psi, gz);
    if (sf) {
        const double gr = dmul(-ph.wall_param, rho);
        Fx = __fma_rn(gr, ax, Fx);
        Fy = __fma_rn(gr, ay, Fy);
        Fz = __fma_rn(gr, az, Fz);
    }
    if (k.body) {
        Fx = dadd(Fx, ph.fx);
        Fy = dadd(Fy, ph.fy);
        Fz = dadd(Fz, ph.fz);
    }
    // Eq. 4: h = rho u = sum e f + F / 2
    const double hx = __fma_rn(0.5, Fx, dadd(q1, Tx)), hy = __fma_rn(0.5, Fy, dadd(q3, Ty));
    const double hz = __fma_rn(0.5, Fz, dadd(q5, Tz));
    const double inv = __drcp_rn(rho);
    ux = dmul(hx, inv);
    uy = dmul(hy, inv);
    uz = dmul(hz, inv);
    if constexpr (COLLIDE) {
        const double X = __fma_rn(gx, gx, __fma_rn(gy, gy, dmul(gz, gz)));
        const double p1 = dadd(f[1], f[2]), p3 = dadd(f[3], f[4]), p5 = dadd(f[5], f[6]);
        const double p7 = dadd(f[7], f[8]), p9 = dadd(f[9], f[10]), p11 = dadd(f[11], f[12]), p13 = dadd(f[13], f[14]);
        const double p15 = dadd(f[15], f[16]), p17 = dadd(f[17], f[18]);
        const double ayz = dadd(p3, p5), s16 = dadd(p1, ayz);
        const double exy = dadd(p7, p9), exz = dadd(p11, p13), eyz = dadd(p15, p17);
        const double exyz = dadd(exy, exz), s718 = dadd(exyz, eyz);
        const double rxx = dmul(hx, ux), ryy = dmul(hy, uy), rzz = dmul(hz, uz);
        const double R = dadd(dadd(rxx, ryy), rzz);                                   // rho u^2
        // with rho = f0 + s16 + s718:
        //   e - e_eq = e + 11 rho - 19 rho u^2 = 19 (s718 - f0 - R),
        //   eps - eps_eq = eps - 3 rho + 11/2 rho u^2 = 9 f0 - 7 s16 - 2 s718 + 11/2 R
        const double E1 = dsub(dsub(s718, f[0]), R);
        const double E2 = __fma_rn(9.0, f[0], __fma_rn(-7.0, s16, __fma_rn(-2.0, s718, dmul(5.5, R))));
        const double W = __fma_rn(-2.0, eyz, exyz), V = __fma_rn(2.0, p1, -ayz);
        const double m9 = dadd(W, V), m10 = __fma_rn(-2.0, V, W);
        const double da = dsub(p3, p5), de = dsub(exy, exz);
        const double m11 = dadd(da, de), m12 = __fma_rn(-2.0, da, de);
        const double p3xx = __fma_rn(3.0, rxx, -R), pww = dsub(ryy, rzz);
        const double uFx = dmul(ux, Fx), uFy = dmul(uy, Fy), uFz = dmul(uz, Fz);
        const double yz = dadd(uFy, uFz), uF = dadd(uFx, yz);
        const double Sx = __fma_rn(2.0, uFx, -yz), Sw = dsub(uFy, uFz);               // half of S_3pxx and S_pww
        // a_k = (m*_k - m_k) / |row_k|^2
        const double a1 = __fma_rn(k.t3e, X, __fma_rn(k.t2e, uF, dmul(k.t1e, E1)));
        const double a2 = __fma_rn(k.t3p, X, __fma_rn(k.t2p, uF, dmul(k.t1p, E2)));
        const double a4 = __fma_rn(k.tq2, Fx, dmul(k.tq1, __fma_rn(2.0 / 3.0, hx, __fma_rn(-4.0, q1, Tx))));
        const double a6 = __fma_rn(k.tq2, Fy, dmul(k.tq1, __fma_rn(2.0 / 3.0, hy, __fma_rn(-4.0, q3, Ty))));
        const double a8 = __fma_rn(k.tq2, Fz, dmul(k.tq1, __fma_rn(2.0 / 3.0, hz, __fma_rn(-4.0, q5, Tz))));
        const double a9 = __fma_rn(k.th9, Sx, dmul(k.tn9, dsub(m9, p3xx)));
        const double a10 = __fma_rn(k.th10, Sx, dmul(k.tp10, __fma_rn(0.5, p3xx, m10)));
        const double a11 = __fma_rn(k.th11, Sw, dmul(k.tn11, dsub(m11, pww)));
        const double a12 = __fma_rn(k.th12, Sw, dmul(k.tp12, __fma_rn(0.5, pww, m12)));
        const double a13 = __fma_rn(k.th13, __fma_rn(ux, Fy, dmul(uy, Fx)), dmul(k.tn13, __fma_rn(-hx, uy, dsub(p7, p9))));
        const double a14 = __fma_rn(k.th13, __fma_rn(uy, Fz, dmul(uz, Fy)), dmul(k.tn13, __fma_rn(-hy, uz, dsub(p15, p17))));
        const double a15 = __fma_rn(k.th13, __fma_rn(ux, Fz, dmul(uz, Fx)), dmul(k.tn13, __fma_rn(-hx, uz, dsub(p11, p13))));
        const double a16 = dmul(k.tm, dsub(s1, s2)), a17 = dmul(k.tm, dsub(t2, t1)), a18 = dmul(k.tm, dsub(v1, v2));
        const double a3 = dmul(0.1, Fx), a5 = dmul(0.1, Fy), a7 = dmul(0.1, Fz);
        // f += M^T diag(1/|row|^2) (m* - m), columns of M per velocity
        f[0] = __fma_rn(-30.0, a1, __fma_rn(12.0, a2, f[0]));
        const double axis = __fma_rn(-11.0, a1, dmul(-4.0, a2));
        const double a910 = __fma_rn(-2.0, a10, a9), a1112 = __fma_rn(-2.0, a12, a11);
        const double axx = __fma_rn(2.0, a910, axis), am = dsub(axis, a910), ayy = dadd(am, a1112), azz = dsub(am, a1112);
        const double r3 = __fma_rn(-4.0, a4, a3), r5 = __fma_rn(-4.0, a6, a5), r7 = __fma_rn(-4.0, a8, a7);
        f[1] = dadd(f[1], dadd(axx, r3));
        f[2] = dadd(f[2], dsub(axx, r3));
        f[3] = dadd(f[3], dadd(ayy, r5));
        f[4] = dadd(f[4], dsub(ayy, r5));
        f[5] = dadd(f[5], dadd(azz, r7));
        f[6] = dadd(f[6], dsub(azz, r7));
        const double edge = __fma_rn(8.0, a1, a2), b910 = dadd(a9, a10), b1112 = dadd(a11, a12);
        const double eb = dadd(edge, b910), exy0 = dadd(eb, b1112), exz0 = dsub(eb, b1112), eyz0 = __fma_rn(-2.0, b910, edge);
        const double t34 = dadd(a3, a4), t56 = dadd(a5, a6), t78 = dadd(a7, a8);
        auto edges = [&](int a, double base, double cross, double g, double h, double g2, double h2) {
            const double up = dadd(base, cross), dn = dsub(base, cross), o1 = dadd(g, h), o2 = dadd(g2, h2);
            f[a] = dadd(f[a], dadd(up, o1));
            f[a + 1] = dadd(f[a + 1], dsub(up, o1));
            f[a + 2] = dadd(f[a + 2], dadd(dn, o2));
            f[a + 3] = dadd(f[a + 3], dsub(dn, o2));
        };
        edges(7, exy0, a13, dadd(t34, t56), dsub(a16, a17), dsub(t34, t56), dadd(a16, a17));
        edges(11, exz0, a15, dadd(t34, t78), dsub(a18, a16), dsub(t34, t78), -dadd(a16, a18));
        edges(15, eyz0, a14, dadd(t56, t78), dsub(a17, a18), dsub(t56, t78), dadd(a17, a18));
    }
}

}  // namespace lbmwet
