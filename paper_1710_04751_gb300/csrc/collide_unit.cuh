// collide_unit.cuh -- the collisions of arXiv:1710.04751 at the paper's own choice of the
// higher-order rates, computed directly from the few moments that choice leaves alive.
//
// The paper sets every relaxation rate it does not tie to a transport coefficient to
// unity: for the scalar (Sec. 2.2, App. C) all but omega_1..3, which give the
// diffusivity (Eq. 23); for the flow (App. A) all but the viscous ones (read here as the
// five shear moments; the bulk moment and the third and fourth orders relax at 1).  A
// central moment relaxed at rate 1 takes its equilibrium (plus, for the flow, its source
// share (1 - omega) Gamma = 0) whatever its pre-collision value.  So the post-collision
// state depends on the pulled populations only through
//   flow:   rho, the momentum and the six second-order moments (ten raw moments);
//   scalar: phi (Eq. 25) and the three first-order moments.
// collide.cuh computes every moment and relaxes each with its own rate; for these rates
// the result is the same up to rounding (the tests hold both to the FP64 oracle, which
// runs the paper's closed-form cascades).  Here the post-collision central moments are
//   flow   c0 = rho, c_i = F_i/2, c_xy.. = (1 - omega) k_xy.., traceless second-order
//          combinations (1 - omega) k, trace rho (= 3 c_s^2 rho), third order 0,
//          c_xxyy = E (reading R1: c_xx c_yy / rho, or rho c_s^4);
//   scalar c0 = phi + R/2, c_i = (1 - omega_i)(m_i - u_i m0), c_ii = c_sphi^2 phi,
//          mixed and third order 0, c_xxyy = c_sphi^4 phi (Eq. 15);
// shifted to raw moments by the binomial theorem about u (Eqs. 14, 17) and inverted to
// populations.  Everything is written for moments taken RELATIVE TO THE REST STATE
// (f - w_a for the flow, g - w^phi_a phi for the scalar): the quantities stay small, which
// keeps the rounding of the single-precision forms far below their storage resolution.
//
// Templated on the arithmetic type: float, double, or Pair (two nodes in packed FP32
// pair instructions, pair.cuh).
#pragma once

#include "collide.cuh"

namespace lbm {

// Fused multiply-add and constants for the arithmetic types.
__device__ __forceinline__ float fmad(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fmad(double a, double b, double c) { return fma(a, b, c); }
template <typename T>
__device__ __forceinline__ T cst(double v) { return T(v); }

// The ten raw moments up to second order of a D3Q15 vector (the sign transform of raw15
// without its third- and fourth-order outputs).
template <typename T>
struct Low10 {
    T m0, x, y, z, xy, xz, yz, xx, yy, zz;
};

template <typename T>
__device__ __forceinline__ Low10<T> raw_low15(const T (&p)[15]) {
    const T a0 = p[7] + p[8], b0 = p[7] - p[8];
    const T a1 = p[9] + p[10], b1 = p[9] - p[10];
    const T a2 = p[11] + p[12], b2 = p[11] - p[12];
    const T a3 = p[13] + p[14], b3 = p[13] - p[14];
    const T c0 = a0 + a1, c1 = a0 - a1, c2 = a2 + a3, c3 = a2 - a3;
    const T e0 = b0 + b1, e1 = b0 - b1, e2 = b2 + b3, e3 = b2 - b3;
    const T H0 = c0 + c2, Hz = c0 - c2, Hy = c1 + c3, Hyz = c1 - c3;
    const T Hx = e0 + e2, Hxz = e0 - e2, Hxy = e1 + e3;
    const T px = p[1] + p[2], qx = p[1] - p[2];
    const T py = p[3] + p[4], qy = p[3] - p[4];
    const T pz = p[5] + p[6], qz = p[5] - p[6];
    Low10<T> m;
    m.m0 = p[0] + px + py + pz + H0;
    m.x = qx + Hx;
    m.y = qy + Hy;
    m.z = qz + Hz;
    m.xy = Hxy;
    m.xz = Hxz;
    m.yz = Hyz;
    m.xx = px + H0;
    m.yy = py + H0;
    m.zz = pz + H0;
    return m;
}

// Zeroth and first raw moments of a D3Q15 or D3Q7 vector.
template <typename T, int Q>
__device__ __forceinline__ void raw_first(const T (&p)[Q], T& m0, T& mx, T& my, T& mz) {
    const T px = p[1] + p[2], qx = p[1] - p[2];
    const T py = p[3] + p[4], qy = p[3] - p[4];
    const T pz = p[5] + p[6], qz = p[5] - p[6];
    if constexpr (Q == 15) {
        const T a0 = p[7] + p[8], b0 = p[7] - p[8];
        const T a1 = p[9] + p[10], b1 = p[9] - p[10];
        const T a2 = p[11] + p[12], b2 = p[11] - p[12];
        const T a3 = p[13] + p[14], b3 = p[13] - p[14];
        const T c0 = a0 + a1, c1 = a0 - a1, c2 = a2 + a3, c3 = a2 - a3;
        const T e0 = b0 + b1, e2 = b2 + b3;
        m0 = p[0] + px + py + pz + (c0 + c2);
        mx = qx + (e0 + e2);
        my = qy + (c1 + c3);
        mz = qz + (c0 - c2);
    } else {
        m0 = p[0] + px + py + pz;
        mx = qx;
        my = qy;
        mz = qz;
    }
}

// The populations whose raw moments are r (the inverse of raw15): p = K^-1 applied in the
// monomial basis, diagonal links by the inverse three-level sign transform.
template <typename T>
__device__ __forceinline__ void populations15(const Raw15<T>& r, T (&p)[15]) {
    const T G0 = r.xxyy, Gx = r.xyy, Gy = r.xxy, Gz = r.xxz;
    const T P0 = G0 + Gz, P0m = G0 - Gz, Px = Gx + r.xz, Pxm = Gx - r.xz;
    const T Py = Gy + r.yz, Pym = Gy - r.yz, Pxy = r.xy + r.xyz, Pxym = r.xy - r.xyz;
    const T Q0 = P0 + Py, Q1 = P0 - Py, X0 = Px + Pxy, X1 = Px - Pxy;
    const T Q2 = P0m + Pym, Q3 = P0m - Pym, X2 = Pxm + Pxym, X3 = Pxm - Pxym;
    const T e = cst<T>(0.125), h = cst<T>(0.5);
    p[7] = e * (Q0 + X0);
    p[8] = e * (Q0 - X0);
    p[9] = e * (Q1 + X1);
    p[10] = e * (Q1 - X1);
    p[11] = e * (Q2 + X2);
    p[12] = e * (Q2 - X2);
    p[13] = e * (Q3 + X3);
    p[14] = e * (Q3 - X3);
    const T px = r.xx - G0, qx = r.x - Gx;
    const T py = r.yy - G0, qy = r.y - Gy;
    const T pz = r.zz - G0, qz = r.z - Gz;
    p[1] = h * (px + qx);
    p[2] = h * (px - qx);
    p[3] = h * (py + qy);
    p[4] = h * (py - qy);
    p[5] = h * (pz + qz);
    p[6] = h * (pz - qz);
    p[0] = r.m0 - px - py - pz - G0;
}

// The relaxation rates and constants the unit-rate collisions use.
template <typename T>
struct UnitRates {
    T om1[3];      // 1 - omega_4, 5, 6 (flow xy, xz, yz) ...
    T omA, omB;    // 1 - omega_7, 1 - omega_8 (flow xx - yy, xx + yy - 2 zz)
    T omg[3];      // 1 - omega_1, 2, 3 (scalar first order)
    T cs2, cs4;    // c_sphi^2, c_sphi^4
    T R, halfR;    // scalar source R and R/2
    int e4_mode;
};

template <typename T, typename real>
__device__ __forceinline__ UnitRates<T> unit_rates(const DevParams<real>& p) {
    UnitRates<T> r;
    for (int i = 0; i < 3; ++i) {
        r.om1[i] = cst<T>(1.0 - (double)p.om_f[4 + i]);
        r.omg[i] = cst<T>(1.0 - (double)p.om_g[1 + i]);
    }
    r.omA = cst<T>(1.0 - (double)p.om_f[7]);
    r.omB = cst<T>(1.0 - (double)p.om_f[8]);
    r.cs2 = cst<T>((double)p.cs2_phi);
    r.cs4 = cst<T>((double)p.cs2_phi * (double)p.cs2_phi);
    r.R = cst<T>((double)p.heat_source);
    r.halfR = cst<T>(0.5 * (double)p.heat_source);
    r.e4_mode = p.e4_mode;
    return r;
}

// Powers of u shared by the binomial shifts.
template <typename T>
struct UPow {
    T x, y, z, xx, yy, zz, xy, xz, yz;
};
template <typename T>
__device__ __forceinline__ UPow<T> upow(T ux, T uy, T uz) {
    return UPow<T>{ux, uy, uz, ux * ux, uy * uy, uz * uz, ux * uy, ux * uz, uy * uz};
}

// The flow's post-collision central moments (App. A at unit bulk / third / fourth-order
// rates): first order h = F / 2, shear c_ab and the trace-free parts t_aa = c_aa - rho / 3.
template <typename T>
struct FlowRelaxed {
    T delta, rho;  // rho - 1, rho
    T hx, hy, hz, cxy, cxz, cyz, txx, tyy, tzz;
};

// dm: moments of f - w_a up to second order; F: the body force.  Returns u (Eq. 3).
template <typename T>
__device__ __forceinline__ FlowRelaxed<T> flow_relax(const Low10<T>& dm, T Fx, T Fy, T Fz, const UnitRates<T>& r,
                                                     T inv_rho, UPow<T>& u) {
    FlowRelaxed<T> k;
    const T h = cst<T>(0.5);
    k.delta = dm.m0;
    k.rho = cst<T>(1.0) + k.delta;
    k.hx = h * Fx, k.hy = h * Fy, k.hz = h * Fz;
    u = upow<T>((dm.x + k.hx) * inv_rho, (dm.y + k.hy) * inv_rho, (dm.z + k.hz) * inv_rho);
    // pre-collision second-order central moments about u (the 1/3 of the rest state
    // cancels in every combination that relaxes): k_ab = m_ab - rho u_a u_b
    // + (u_a F_b + u_b F_a)/2, k_aa = m_aa - rho u_a^2 + u_a F_a
    const T kxy = fmad(u.x, k.hy, fmad(u.y, k.hx, dm.xy - k.rho * u.xy));
    const T kxz = fmad(u.x, k.hz, fmad(u.z, k.hx, dm.xz - k.rho * u.xz));
    const T kyz = fmad(u.y, k.hz, fmad(u.z, k.hy, dm.yz - k.rho * u.yz));
    const T sxx = fmad(u.x, Fx, dm.xx - k.rho * u.xx);  // k_xx - 1/3
    const T syy = fmad(u.y, Fy, dm.yy - k.rho * u.yy);
    const T szz = fmad(u.z, Fz, dm.zz - k.rho * u.zz);
    // relaxation: shear at its rates, trace to rho (its equilibrium 3 c_s^2 rho)
    k.cxy = r.om1[0] * kxy, k.cxz = r.om1[1] * kxz, k.cyz = r.om1[2] * kyz;
    const T A = r.omA * (sxx - syy);
    const T B = r.omB * (sxx + syy - cst<T>(2.0) * szz);
    const T B6 = B * cst<T>(1.0 / 6.0);
    k.txx = fmad(h, A, B6), k.tyy = B6 - h * A, k.tzz = cst<T>(-2.0) * B6;  // c_aa - rho/3
    return k;
}

// Flow (App. A) at unit bulk / third / fourth-order rates.  dm: moments of f - w_a up to
// second order; F: the body force.  Returns u (Eq. 3) and D, the raw moments of the
// post-collision f~ - w_a.
template <typename T>
__device__ __forceinline__ void flow_unit(const Low10<T>& dm, T Fx, T Fy, T Fz, const UnitRates<T>& r,
                                          T inv_rho, UPow<T>& u, Raw15<T>& D) {
    const FlowRelaxed<T> k = flow_relax<T>(dm, Fx, Fy, Fz, r, inv_rho, u);
    const T delta = k.delta, rho = k.rho, hx = k.hx, hy = k.hy, hz = k.hz;
    const T cxy = k.cxy, cxz = k.cxz, cyz = k.cyz, txx = k.txx, tyy = k.tyy, tzz = k.tzz;
    const T d3 = delta * cst<T>(1.0 / 3.0);
    const T cxx = cst<T>(1.0 / 3.0) * rho + txx, cyy = cst<T>(1.0 / 3.0) * rho + tyy;
    // fourth-order equilibrium E (reading R1), less the rest value 1/9
    T E9 = delta * cst<T>(1.0 / 9.0);
    if (r.e4_mode == 0) E9 = fmad(txx * tyy, inv_rho, fmad(cst<T>(1.0 / 3.0), txx + tyy, E9));
    // raw moments of the post-collision state about the origin (binomial theorem with
    // third-order central moments 0), less the rest state's
    D.m0 = delta;
    D.x = fmad(rho, u.x, hx);
    D.y = fmad(rho, u.y, hy);
    D.z = fmad(rho, u.z, hz);
    D.xy = fmad(rho, u.xy, fmad(u.x, hy, fmad(u.y, hx, cxy)));
    D.xz = fmad(rho, u.xz, fmad(u.x, hz, fmad(u.z, hx, cxz)));
    D.yz = fmad(rho, u.yz, fmad(u.y, hz, fmad(u.z, hy, cyz)));
    D.xx = fmad(rho, u.xx, fmad(u.x, Fx, d3 + txx));
    D.yy = fmad(rho, u.yy, fmad(u.y, Fy, d3 + tyy));
    D.zz = fmad(rho, u.zz, fmad(u.z, Fz, d3 + tzz));
    const T ruxy = rho * u.xy;
    // xyy = u_x c_yy + 2 u_y c_xy + u_y^2 c_x + 2 u_x u_y c_y + rho u_x u_y^2
    D.xyy = fmad(ruxy, u.y, fmad(u.xy, Fy, fmad(u.yy, hx, fmad(cst<T>(2.0) * u.y, cxy, u.x * cyy))));
    D.xxy = fmad(ruxy, u.x, fmad(u.xy, Fx, fmad(u.xx, hy, fmad(cst<T>(2.0) * u.x, cxy, u.y * cxx))));
    D.xxz = fmad(rho * u.xz, u.x, fmad(u.xz, Fx, fmad(u.xx, hz, fmad(cst<T>(2.0) * u.x, cxz, u.z * cxx))));
    // xyz = u_x c_yz + u_y c_xz + u_z c_xy + u_x u_y c_z + u_x u_z c_y + u_y u_z c_x + rho u_x u_y u_z
    D.xyz = fmad(ruxy, u.z, fmad(u.xy, hz, fmad(u.xz, hy, fmad(u.yz, hx,
                 fmad(u.x, cyz, fmad(u.y, cxz, u.z * cxy))))));
    // xxyy = E + u_x^2 c_yy + u_y^2 c_xx + 4 u_x u_y c_xy + 2 u_x u_y^2 c_x + 2 u_x^2 u_y c_y
    //        + rho u_x^2 u_y^2, less 1/9
    D.xxyy = fmad(ruxy, u.xy, fmad(u.xy, fmad(u.y, Fx, u.x * Fy), fmad(cst<T>(4.0) * u.xy, cxy,
                  fmad(u.yy, cxx, fmad(u.xx, cyy, E9)))));
}

// Scalar D3Q15 (Sec. 2.2) at unit higher-order rates.  phi = sum g + R/2 (Eq. 25), m0 =
// sum g, m_i the first raw moments of the pulled g.  D: raw moments of g~ - w^phi_a phi.
template <typename T>
__device__ __forceinline__ void thermal15_unit(T phi, T m0, T mx, T my, T mz, const UPow<T>& u,
                                               const UnitRates<T>& r, Raw15<T>& D) {
    const T c0 = phi + r.halfR;  // m0 + R: the zeroth moment gains the source
    const T cx = r.omg[0] * (mx - u.x * m0);
    const T cy = r.omg[1] * (my - u.y * m0);
    const T cz = r.omg[2] * (mz - u.z * m0);
    const T C2 = r.cs2 * phi;
    const T two = cst<T>(2.0);
    D.m0 = r.halfR;
    D.x = fmad(u.x, c0, cx);
    D.y = fmad(u.y, c0, cy);
    D.z = fmad(u.z, c0, cz);
    D.xy = fmad(u.xy, c0, fmad(u.x, cy, u.y * cx));
    D.xz = fmad(u.xz, c0, fmad(u.x, cz, u.z * cx));
    D.yz = fmad(u.yz, c0, fmad(u.y, cz, u.z * cy));
    D.xx = fmad(u.xx, c0, two * u.x * cx);   // c_xx = c_sphi^2 phi cancels the rest value
    D.yy = fmad(u.yy, c0, two * u.y * cy);
    D.zz = fmad(u.zz, c0, two * u.z * cz);
    D.xyy = fmad(u.xy * u.y, c0, fmad(two * u.xy, cy, fmad(u.yy, cx, u.x * C2)));
    D.xxy = fmad(u.xy * u.x, c0, fmad(two * u.xy, cx, fmad(u.xx, cy, u.y * C2)));
    D.xxz = fmad(u.xz * u.x, c0, fmad(two * u.xz, cx, fmad(u.xx, cz, u.z * C2)));
    D.xyz = fmad(u.xy * u.z, c0, fmad(u.xy, cz, fmad(u.xz, cy, u.yz * cx)));
    D.xxyy = fmad(u.xx * u.yy, c0, fmad(two * u.xy, fmad(u.y, cx, u.x * cy), (u.xx + u.yy) * C2));
}

// Scalar D3Q7 (App. C) at unit higher-order rates: the post-collision g~ - w^phi_a phi.
template <typename T>
__device__ __forceinline__ void thermal7_unit(T phi, T m0, T mx, T my, T mz, const UPow<T>& u,
                                              const UnitRates<T>& r, T (&d)[7]) {
    const T c0 = phi + r.halfR;
    const T cx = r.omg[0] * (mx - u.x * m0);
    const T cy = r.omg[1] * (my - u.y * m0);
    const T cz = r.omg[2] * (mz - u.z * m0);
    const T two = cst<T>(2.0), h = cst<T>(0.5);
    const T Dx = fmad(u.x, c0, cx), Dy = fmad(u.y, c0, cy), Dz = fmad(u.z, c0, cz);
    const T Dxx = fmad(u.xx, c0, two * u.x * cx);
    const T Dyy = fmad(u.yy, c0, two * u.y * cy);
    const T Dzz = fmad(u.zz, c0, two * u.z * cz);
    d[1] = h * (Dxx + Dx);
    d[2] = h * (Dxx - Dx);
    d[3] = h * (Dyy + Dy);
    d[4] = h * (Dyy - Dy);
    d[5] = h * (Dzz + Dz);
    d[6] = h * (Dzz - Dz);
    d[0] = r.halfR - Dxx - Dyy - Dzz;
}

// ---- the same with nested products --------------------------------------------------------
// flow_unit and thermal15_unit write every raw moment as its binomial sum; nested, the lower
// moments serve the higher ones (D.xyy = u_x (D.yy + c_yy ...) and so on) and the pre-collision
// moments need no product with rho (rho u = dm.x + F/2): with populations15_on about 320 instead
// of 396 operations a node (D3Q15).  FP64, bound by its two lanes per clock and SM: 300 steps at
// 32^3 8.41 -> 7.45 ms; FP32: 100 steps at 64^3 1.20 -> 1.15 ms.  The 16-bit forms keep the sums:
// a different FP32 rounding there changes which stored values round up.

// The populations w + p of populations15(r): rest weights w0, w1 (axis), w7 (diagonal) added.
template <typename T>
__device__ __forceinline__ void populations15_on(const Raw15<T>& r, T w0, T w1, T w7, T (&p)[15]) {
    const T G0 = r.xxyy, Gx = r.xyy, Gy = r.xxy, Gz = r.xxz;
    const T P0 = G0 + Gz, P0m = G0 - Gz, Px = Gx + r.xz, Pxm = Gx - r.xz;
    const T Py = Gy + r.yz, Pym = Gy - r.yz, Pxy = r.xy + r.xyz, Pxym = r.xy - r.xyz;
    const T Q0 = P0 + Py, Q1 = P0 - Py, X0 = Px + Pxy, X1 = Px - Pxy;
    const T Q2 = P0m + Pym, Q3 = P0m - Pym, X2 = Pxm + Pxym, X3 = Pxm - Pxym;
    const T e = cst<T>(0.125), h = cst<T>(0.5);
    p[7] = fmad(e, Q0 + X0, w7);
    p[8] = fmad(e, Q0 - X0, w7);
    p[9] = fmad(e, Q1 + X1, w7);
    p[10] = fmad(e, Q1 - X1, w7);
    p[11] = fmad(e, Q2 + X2, w7);
    p[12] = fmad(e, Q2 - X2, w7);
    p[13] = fmad(e, Q3 + X3, w7);
    p[14] = fmad(e, Q3 - X3, w7);
    const T px = r.xx - G0, qx = r.x - Gx;
    const T py = r.yy - G0, qy = r.y - Gy;
    const T pz = r.zz - G0, qz = r.z - Gz;
    p[1] = fmad(h, px + qx, w1);
    p[2] = fmad(h, px - qx, w1);
    p[3] = fmad(h, py + qy, w1);
    p[4] = fmad(h, py - qy, w1);
    p[5] = fmad(h, pz + qz, w1);
    p[6] = fmad(h, pz - qz, w1);
    p[0] = r.m0 - px - py - pz - G0 + w0;
}

template <typename T>
__device__ __forceinline__ void flow_unit_nested(const Low10<T>& dm, T Fx, T Fy, T Fz, const UnitRates<T>& r,
                                                 T inv_rho, T& ux, T& uy, T& uz, Raw15<T>& D) {
    const T h = cst<T>(0.5), third = cst<T>(1.0 / 3.0);
    const T delta = dm.m0;  // rho - 1
    const T hx = h * Fx, hy = h * Fy, hz = h * Fz;
    const T jx = dm.x + hx, jy = dm.y + hy, jz = dm.z + hz;  // rho u
    ux = jx * inv_rho, uy = jy * inv_rho, uz = jz * inv_rho;
    // pre-collision central moments: k_ab = m_ab - u_b m_a + u_a F_b/2 (m_a = rho u_a - F_a/2),
    // k_aa - 1/3 = dm_aa - u_a (m_a - F_a/2)
    const T kxy = fmad(ux, hy, fmad(-uy, dm.x, dm.xy));
    const T kxz = fmad(ux, hz, fmad(-uz, dm.x, dm.xz));
    const T kyz = fmad(uy, hz, fmad(-uz, dm.y, dm.yz));
    const T sxx = fmad(-ux, dm.x - hx, dm.xx);
    const T syy = fmad(-uy, dm.y - hy, dm.yy);
    const T szz = fmad(-uz, dm.z - hz, dm.zz);
    const T cxy = r.om1[0] * kxy, cxz = r.om1[1] * kxz, cyz = r.om1[2] * kyz;
    const T A = r.omA * (sxx - syy);
    const T B6 = (cst<T>(1.0 / 6.0) * r.omB) * fmad(cst<T>(-2.0), szz, sxx + syy);
    const T txx = fmad(h, A, B6), tyy = fmad(-h, A, B6);  // c_aa - rho/3; tzz = -2 B6
    T E9 = delta * cst<T>(1.0 / 9.0);  // E - 1/9 (reading R1)
    if (r.e4_mode == 0) E9 = fmad(txx * tyy, inv_rho, fmad(third, txx + tyy, E9));
    const T d3 = delta * third;
    D.m0 = delta;
    D.x = jx + hx;
    D.y = jy + hy;
    D.z = jz + hz;
    D.xy = fmad(uy, D.x, fmad(ux, hy, cxy));
    D.xz = fmad(uz, D.x, fmad(ux, hz, cxz));
    D.yz = fmad(uz, D.y, fmad(uy, hz, cyz));
    D.xx = fmad(ux, D.x + hx, d3 + txx);
    D.yy = fmad(uy, D.y + hy, d3 + tyy);
    D.zz = fmad(uz, D.z + hz, fmad(cst<T>(-2.0), B6, d3));
    const T Mxx = third + D.xx, Myy = third + D.yy;  // raw xx, yy
    const T c2 = cxy + cxy, uxx = ux * ux, uxy = ux * uy;
    // xyy = u_x M_yy + u_y (2 c_xy + u_y F_x/2), likewise xxy and xxz
    D.xyy = fmad(ux, Myy, uy * fmad(uy, hx, c2));
    D.xxy = fmad(uy, Mxx, ux * fmad(ux, hy, c2));
    D.xxz = fmad(uz, Mxx, ux * fmad(ux, hz, cxz + cxz));
    // xyz = u_z xy + u_x c_yz + u_y c_xz + u_x u_y F_z/2
    D.xyz = fmad(uz, D.xy, fmad(ux, cyz, fmad(uy, cxz, uxy * hz)));
    // xxyy = u_x^2 M_yy + u_y^2 (c_xx + u_x F_x) + 4 u_x u_y c_xy + E, less 1/9
    D.xxyy = fmad(uxx, Myy, fmad(uy * uy, fmad(ux, Fx, third + d3 + txx), fmad(uxy, c2 + c2, E9)));
}

template <typename T>
__device__ __forceinline__ void thermal15_unit_nested(T phi, T m0, T mx, T my, T mz, T ux, T uy, T uz,
                                                      const UnitRates<T>& r, Raw15<T>& D) {
    const T c0 = phi + r.halfR;
    const T cx = r.omg[0] * fmad(-ux, m0, mx);
    const T cy = r.omg[1] * fmad(-uy, m0, my);
    const T cz = r.omg[2] * fmad(-uz, m0, mz);
    const T C2 = r.cs2 * phi;
    D.m0 = r.halfR;
    D.x = fmad(ux, c0, cx);
    D.y = fmad(uy, c0, cy);
    D.z = fmad(uz, c0, cz);
    D.xy = fmad(uy, D.x, ux * cy);
    D.xz = fmad(uz, D.x, ux * cz);
    D.yz = fmad(uz, D.y, uy * cz);
    D.xx = ux * (D.x + cx);
    D.yy = uy * (D.y + cy);
    D.zz = uz * (D.z + cz);
    const T Nxx = D.xx + C2, Nyy = D.yy + C2;  // raw xx, yy
    const T ucx = ux * cx, ucz = ux * cz;
    D.xyy = fmad(ux, Nyy, uy * (uy * cx));
    D.xxy = fmad(uy, Nxx, ux * (ux * cy));
    D.xxz = fmad(uz, Nxx, ux * ucz);
    D.xyz = fmad(uz, D.xy, uy * ucz);
    D.xxyy = fmad(ux * ux, Nyy, (uy * uy) * fmad(cst<T>(2.0), ucx, C2));
}

template <typename T>
__device__ __forceinline__ void thermal7_unit_nested(T phi, T m0, T mx, T my, T mz, T ux, T uy, T uz,
                                                     const UnitRates<T>& r, T (&d)[7]) {
    const T c0 = phi + r.halfR, h = cst<T>(0.5);
    const T cx = r.omg[0] * fmad(-ux, m0, mx);
    const T cy = r.omg[1] * fmad(-uy, m0, my);
    const T cz = r.omg[2] * fmad(-uz, m0, mz);
    const T Dx = fmad(ux, c0, cx), Dy = fmad(uy, c0, cy), Dz = fmad(uz, c0, cz);
    const T Dxx = ux * (Dx + cx), Dyy = uy * (Dy + cy), Dzz = uz * (Dz + cz);
    d[1] = h * (Dxx + Dx);
    d[2] = h * (Dxx - Dx);
    d[3] = h * (Dyy + Dy);
    d[4] = h * (Dyy - Dy);
    d[5] = h * (Dzz + Dz);
    d[6] = h * (Dzz - Dz);
    d[0] = r.halfR - Dxx - Dyy - Dzz;
}

// ---- u and T imposed after the collision (lbm_init_fields) --------------------------------
// p <- p~ - p_eq(u, T) + p_eq(v, S): the node keeps its departure from equilibrium and its rho
// and takes the imposed v and S.  The post-collision state of the collisions above has the u
// and T they were computed from (the force enters both at the same time level), so p~ -
// p_eq(u, T) is what is left of D without its equilibrium part, and no population is needed.

// Raw moments of f - w_a: those of f~ - f_eq(rho, u) plus those of f_eq(rho, v) - w_a.
template <typename T>
__device__ __forceinline__ void flow_unit_imposed(const Low10<T>& dm, T Fx, T Fy, T Fz, const UnitRates<T>& r,
                                                  T inv_rho, UPow<T>& u, const UPow<T>& v, Raw15<T>& D) {
    const FlowRelaxed<T> k = flow_relax<T>(dm, Fx, Fy, Fz, r, inv_rho, u);
    // fourth-order equilibrium E (reading R1), less f_eq's rho / 9
    T E9 = cst<T>(0.0);
    if (r.e4_mode == 0) E9 = fmad(k.txx * k.tyy, inv_rho, cst<T>(1.0 / 3.0) * (k.txx + k.tyy));
    const T two = cst<T>(2.0), r3 = cst<T>(1.0 / 3.0) * k.rho, d3 = cst<T>(1.0 / 3.0) * k.delta;
    D.m0 = k.delta;
    D.x = fmad(k.rho, v.x, k.hx);
    D.y = fmad(k.rho, v.y, k.hy);
    D.z = fmad(k.rho, v.z, k.hz);
    D.xy = fmad(k.rho, v.xy, fmad(u.x, k.hy, fmad(u.y, k.hx, k.cxy)));
    D.xz = fmad(k.rho, v.xz, fmad(u.x, k.hz, fmad(u.z, k.hx, k.cxz)));
    D.yz = fmad(k.rho, v.yz, fmad(u.y, k.hz, fmad(u.z, k.hy, k.cyz)));
    D.xx = fmad(k.rho, v.xx, fmad(u.x, Fx, d3 + k.txx));
    D.yy = fmad(k.rho, v.yy, fmad(u.y, Fy, d3 + k.tyy));
    D.zz = fmad(k.rho, v.zz, fmad(u.z, Fz, d3 + k.tzz));
    const T nxyy = fmad(u.xy, Fy, fmad(u.yy, k.hx, fmad(two * u.y, k.cxy, u.x * k.tyy)));
    const T nxxy = fmad(u.xy, Fx, fmad(u.xx, k.hy, fmad(two * u.x, k.cxy, u.y * k.txx)));
    const T nxxz = fmad(u.xz, Fx, fmad(u.xx, k.hz, fmad(two * u.x, k.cxz, u.z * k.txx)));
    const T nxyz = fmad(u.xy, k.hz, fmad(u.xz, k.hy, fmad(u.yz, k.hx, fmad(u.x, k.cyz, fmad(u.y, k.cxz, u.z * k.cxy)))));
    const T nxxyy = fmad(u.xy, fmad(u.y, Fx, u.x * Fy), fmad(cst<T>(4.0) * u.xy, k.cxy,
                         fmad(u.yy, k.txx, fmad(u.xx, k.tyy, E9))));
    const T rvxy = k.rho * v.xy;
    D.xyy = fmad(rvxy, v.y, fmad(r3, v.x, nxyy));
    D.xxy = fmad(rvxy, v.x, fmad(r3, v.y, nxxy));
    D.xxz = fmad(k.rho * v.xz, v.x, fmad(r3, v.z, nxxz));
    D.xyz = fmad(rvxy, v.z, nxyz);
    D.xxyy = fmad(rvxy, v.xy, fmad(r3, v.xx + v.yy, fmad(cst<T>(1.0 / 9.0), k.delta, nxxyy)));
}

// Raw moments of g - w^phi_a S: thermal15_unit at phi = 0 is g~ - g_eq(phi, u).
template <typename T>
__device__ __forceinline__ void thermal15_unit_imposed(T m0, T mx, T my, T mz, const UPow<T>& u,
                                                       const UnitRates<T>& r, T S, const UPow<T>& v, Raw15<T>& D) {
    thermal15_unit<T>(cst<T>(0.0), m0, mx, my, mz, u, r, D);
    const T C2 = r.cs2 * S;
    D.x = fmad(v.x, S, D.x);
    D.y = fmad(v.y, S, D.y);
    D.z = fmad(v.z, S, D.z);
    D.xy = fmad(v.xy, S, D.xy);
    D.xz = fmad(v.xz, S, D.xz);
    D.yz = fmad(v.yz, S, D.yz);
    D.xx = fmad(v.xx, S, D.xx);
    D.yy = fmad(v.yy, S, D.yy);
    D.zz = fmad(v.zz, S, D.zz);
    D.xyy = fmad(v.xy * v.y, S, fmad(v.x, C2, D.xyy));
    D.xxy = fmad(v.xy * v.x, S, fmad(v.y, C2, D.xxy));
    D.xxz = fmad(v.xz * v.x, S, fmad(v.z, C2, D.xxz));
    D.xyz = fmad(v.xy * v.z, S, D.xyz);
    D.xxyy = fmad(v.xx * v.yy, S, fmad(v.xx + v.yy, C2, D.xxyy));
}

template <typename T>
__device__ __forceinline__ void thermal7_unit_imposed(T m0, T mx, T my, T mz, const UPow<T>& u,
                                                      const UnitRates<T>& r, T S, const UPow<T>& v, T (&d)[7]) {
    thermal7_unit<T>(cst<T>(0.0), m0, mx, my, mz, u, r, d);
    const T h = cst<T>(0.5);
    const T Dx = v.x * S, Dy = v.y * S, Dz = v.z * S, Dxx = v.xx * S, Dyy = v.yy * S, Dzz = v.zz * S;
    d[1] += h * (Dxx + Dx);
    d[2] += h * (Dxx - Dx);
    d[3] += h * (Dyy + Dy);
    d[4] += h * (Dyy - Dy);
    d[5] += h * (Dzz + Dz);
    d[6] += h * (Dzz - Dz);
    d[0] -= Dxx + Dyy + Dzz;
}

// Whether a context's rates are the paper's unit higher-order rates (host side).
template <typename real>
inline bool has_unit_rates(const DevParams<real>& p, int Q) {
    for (int b = 9; b < 15; ++b)
        if (p.om_f[b] != real(1)) return false;
    for (int b = 4; b < Q; ++b)
        if (p.om_g[b] != real(1)) return false;
    return true;
}

}  // namespace lbm
