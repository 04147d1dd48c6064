// igks_gks.cuh -- the gas-kinetic interface flux of one face (Eq. 4-14, 33-34) as device
// functions.
//
// What bounds it: the FP64 pipe of GB300, which issues one warp instruction per 19 cycles
// and SM whatever it is (a comparison or a conversion costs as much as a fused
// multiply-add). The algebra is arranged to issue few of them:
//
//  - Slopes. The slope polynomials a . psi of a Maxwellian (Eq. 101, 11, 12) are the
//    logarithmic derivatives of the Maxwellian, so they are carried as derivatives of the
//    primitive variables (density ratio, U, V, h = 1/(2 lambda)) and no 4x4 system is
//    solved: ten operations take a conserved slope to a primitive one.
//  - Time slopes. <(a_n u + a_t v + A) psi> = 0 (Eq. 11) says that A is the time derivative
//    of the Euler equations for those slopes: thirteen operations.
//  - Hermite moments. With c = u - U the sum a_n u + a_t v + A is the Chapman-Enskog
//    polynomial of the gradients; everything that multiplies a Maxwellian in Eq. 13,
//    q3 + q4 (a_n u + a_t v) + q5 A, is collected first and written, after integration over
//    v and xi, in Hermite polynomials He_k(c) of the variance h. He_k f is a k-th derivative
//    of the Gaussian f, so that by parts, over u >= 0 or u < 0,
//        <u^j He_k> = h^k j! / (j - k)! <u^(j-k)>       (j >= k),
//    and for j < k boundary terms at u = 0 in f(0): moments up to <u^3> (<u^4> once) are
//    enough, and every flux component is a few fused multiply-adds.
//  - One table look-up per Maxwellian gives both half-space integrals, the normal tail
//    Q(z) = erfc(z / sqrt 2) / 2 and its density, from a Taylor polynomial about the nearest
//    node (half_line below): 14 FP64 instructions against 55 for erfcx and exp.
//
// k_flux with it against the moment solves of igks_gks_moment.cuh: 2623 -> 1300 us on 16
// airfoils (1,018,076 faces), 106 -> 57 us on the 20,480-cell plate (35,056 faces).
#pragma once
#include "igks_dev.h"

namespace igks {
namespace gks {

constexpr double HK = 2.0 / (KDOF + 2);               // gamma - 1; h = HK e_int / rho
static_assert(KDOF == 3, "the moments over v and xi below are written for K = 3");

// ---- normal tail and density ----
// Node k at z = k / 512: Taylor coefficients of Q(z) = P(N(0,1) > z), degree 6 (|t| <= 2^-10:
// the remainder is below 1e-16 of Q, and of the density -Q', up to z = 6). 64 bytes a node,
// 192 KiB, computed by the host in extended precision (upload_flux_table).
constexpr int TAIL_PER_UNIT = 512, TAIL_MAX = 6, TAIL_NODES = TAIL_PER_UNIT * TAIL_MAX + 1;
static __device__ __align__(64) double g_tail[TAIL_NODES * 8];

// q = Q(|z|), p = density at z (both accurate to a few ulp, also in the tail)
__device__ __forceinline__ void normal_tail(double z, double& q, double& p) {
  const double a = fabs(z);
  if (a < (double)TAIL_MAX) {
    constexpr double M = 6755399441055744.0 / TAIL_PER_UNIT;   // 1.5 * 2^52 / 512: rounds to a multiple of 1/512
    const double zm = a + M;
    const double t = a - (zm - M);
    const double2* c = reinterpret_cast<const double2*>(g_tail) + 4 * __double2loint(zm);
    const double2 c01 = __ldg(c), c23 = __ldg(c + 1), c45 = __ldg(c + 2), c6 = __ldg(c + 3);
    double b = c6.x, d = b;                  // Horner for Q and, alongside, its derivative
    b = fma(b, t, c45.y); d = fma(d, t, b);
    b = fma(b, t, c45.x); d = fma(d, t, b);
    b = fma(b, t, c23.y); d = fma(d, t, b);
    b = fma(b, t, c23.x); d = fma(d, t, b);
    b = fma(b, t, c01.y); d = fma(d, t, b);
    q = fma(b, t, c01.x);
    p = -d;
  } else {                                   // more than six standard deviations, or not a number
    q = 0.5 * erfc(a * 0.70710678118654752440);
    p = 0.39894228040143267794 * exp(-0.5 * a * a);
  }
}

// A Maxwellian in the face frame: density and its reciprocal, velocity (U normal, V
// tangential), energy per mass, h (the variance of each velocity component), s = 1/sqrt(h)
struct Maxw {
  double r, ir, U, V, et, h, s;
};

__device__ __forceinline__ Maxw maxw_of(const double* W) {
  Maxw g;
  g.r = W[0];
  g.ir = __drcp_rn(W[0]);
  g.U = W[1] * g.ir;
  g.V = W[2] * g.ir;
  g.et = W[3] * g.ir;
  g.h = HK * (g.et - 0.5 * (g.U * g.U + g.V * g.V));
  g.s = rsqrt(g.h);
  return g;
}

// Half-line quantities, sgn = +1: u >= 0, -1: u < 0. m[j] = <u^j> (density one), f = sgn f(0)
// with f(0) the density of u at 0, y = U / h, y2 = y^2 - 1/h.
struct Half {
  double m0, m1, m2, m3, f, y, y2;
};
__device__ __forceinline__ Half half_line(const Maxw& g, double sgn) {
  Half a;
  const double z = g.U * g.s, ih = g.s * g.s;
  double q, p;
  normal_tail(z, q, p);
  const bool big = (__double2hiint(z) < 0) == (sgn < 0.0);     // the half line that holds the mean
  a.m0 = big ? 1.0 - q : q;
  a.f = sgn * (g.s * p);
  a.y = g.U * ih;
  a.y2 = a.y * a.y - ih;
  a.m1 = g.U * a.m0 + g.h * a.f;
  a.m2 = g.U * a.m1 + g.h * a.m0;
  a.m3 = g.U * a.m2 + 2.0 * (g.h * a.m1);
  return a;
}

// slope of the primitive variables from a conserved slope times c (1/rho, or 1/rho over a
// distance): density ratio, U, V, h
struct Slope {
  double a, U, V, h;
};
__device__ __forceinline__ Slope slope_of(const Maxw& g, const double* s, double c) {
  Slope o;
  o.a = s[0] * c;
  o.U = s[1] * c - g.U * o.a;
  o.V = s[2] * c - g.V * o.a;
  o.h = HK * (s[3] * c - g.et * o.a - g.U * o.U - g.V * o.V);
  return o;
}

// What the two slopes of a Maxwellian enter the flux with: minus its Euler time derivative
// (A, U, V, h) and the Chapman-Enskog combinations
struct Rates {
  double A, U, V, h;        // -(time slope) of density ratio, U, V, h
  double st, sh, qn, qt;    // U_n - (U_n + V_t)/5, V_n + U_t, h_n, h_t
};
__device__ __forceinline__ Rates rates_of(const Maxw& g, const Slope& n, const Slope& t) {
  Rates o;
  const double div = n.U + t.V;
  o.A = g.U * n.a + (g.V * t.a + div);
  o.U = g.U * n.U + (g.V * t.U + (g.h * n.a + n.h));
  o.V = g.U * n.V + (g.V * t.V + (g.h * t.a + t.h));
  o.h = g.U * n.h + (g.V * t.h + (HK * g.h) * div);
  o.st = n.U - 0.2 * div;
  o.sh = n.V + t.U;
  o.qn = n.h;
  o.qt = t.h;
  return o;
}

// the flux <u B psi> (four components) and the state integrals <B psi_k>, k = 0, 2, 3
struct Out {
  double F0, F1, F2, F3, S0, S2, S3;
};

// One side of the interface: B = w3 + w4 (a_n u + a_t v) + w5 A times the density one
// Maxwellian over a half line, added to o; with a_n u + a_t v = D - A (D: Chapman-Enskog) and
// n54 = w4 - w5, R = -A: B = w3 + w4 D + n54 R.
__device__ __forceinline__ void side_flux(const Maxw& g, const Half& a, const Rates& R, double w3, double w4,
                                          double n54, Out& o) {
  const double w4h = w4 * g.h, w4h2 = 0.5 * w4h;
  const double b0 = w3 + n54 * R.A;                  // He_0 .. He_3 coefficients times h^k
  const double b1 = n54 * R.U;
  const double k = w4h * R.st, th = n54 * R.h;
  const double b2 = 0.5 * th + k;
  const double b3 = w4h2 * R.qn;
  const double d0 = n54 * R.V, d1 = w4h * R.sh, d2 = w4h2 * R.qt;   // the same of <c_v B>
  const double x = 2.0 * th - k;                     // <(c_v^2 + xi^2) B> / 2 beyond 2 h <B>
  const double P0 = b0 * a.m0 + a.f * (b3 * a.y2 + (b1 - a.y * b2));
  const double P1 = b0 * a.m1 + (b1 * a.m0 + a.f * (b2 - a.y * b3));
  const double P2 = b0 * a.m2 + 2.0 * (b1 * a.m1 + (b2 * a.m0 + b3 * a.f));
  const double P3 = b0 * a.m3 + 3.0 * (b1 * a.m2 + 2.0 * (b2 * a.m1 + b3 * a.m0));
  const double Q0 = d0 * a.m0 + a.f * (d1 - a.y * d2);
  const double Q1 = d0 * a.m1 + (d1 * a.m0 + d2 * a.f);
  const double kk = 2.0 * g.h + (0.5 * g.V) * g.V, b34 = 4.0 * b3;
  o.F0 += P1;
  o.F1 += P2;
  o.F2 += g.V * P1 + Q1;
  o.F3 += 0.5 * P3 + (kk * P1 + (g.V * Q1 + (x * a.m1 + b34 * a.m0)));
  o.S0 += P0;
  o.S2 += g.V * P0 + Q0;
  o.S3 += 0.5 * P2 + (kk * P0 + (g.V * Q0 + (x * a.m0 + b34 * a.f)));
}

// The time-integrated flux of one face in the face frame (Eq. 13-14) with the Prandtl
// fix. WL, WR: reconstructed face states; SLn.. their normal and tangential slopes;
// WcL, WcR: the centre states of the two cells (rotated); idL, idR: reciprocal normal
// distances centre to face; visc(h0, s0) gives the laminar viscosity of the interface state
// from h0 and 1/sqrt(h0) (Sutherland's law); mut: face eddy viscosity.
template <class Visc>
__device__ __forceinline__ void face_flux(const double* WL, const double* WR, const double* SLn, const double* SLt,
                                          const double* SRn, const double* SRt, const double* WcL,
                                          const double* WcR, double idL, double idR, double mut, double dt,
                                          double c_num, double pr_fix, Visc visc, double* Fn) {
  // the two sides: Maxwellian, half-line moments, slopes and rates
  const Maxw gl = maxw_of(WL), gr = maxw_of(WR);
  const Rates Rl = rates_of(gl, slope_of(gl, SLn, gl.ir), slope_of(gl, SLt, gl.ir));
  const Rates Rr = rates_of(gr, slope_of(gr, SRn, gr.ir), slope_of(gr, SRt, gr.ir));
  const Half hl = half_line(gl, 1.0), hr = half_line(gr, -1.0);
  // interface equilibrium g0 (Eq. 5): W0 = <psi> over both half lines
  double W0[4];
  {
    const double l0 = gl.r * hl.m0, r0 = gr.r * hr.m0;
    W0[0] = l0 + r0;
    W0[1] = gl.r * hl.m1 + gr.r * hr.m1;
    W0[2] = gl.V * l0 + gr.V * r0;
    W0[3] = gl.r * (0.5 * hl.m2 + (2.0 * gl.h + (0.5 * gl.V) * gl.V) * hl.m0) +
            gr.r * (0.5 * hr.m2 + (2.0 * gr.h + (0.5 * gr.V) * gr.V) * hr.m0);
  }
  const Maxw g = maxw_of(W0);
  double s[4];
#pragma unroll
  for (int k = 0; k < 4; k++) s[k] = W0[k] - WcL[k];
  Slope L = slope_of(g, s, g.ir * idL);
#pragma unroll
  for (int k = 0; k < 4; k++) s[k] = WcR[k] - W0[k];
  const Slope N = slope_of(g, s, g.ir * idR);
#pragma unroll
  for (int k = 0; k < 4; k++) s[k] = SLt[k] + SRt[k];
  const Rates R = rates_of(g, N, slope_of(g, s, 0.5 * g.ir));
  // a_l u H + a_r u (1 - H) = a_r u + (a_l - a_r) u H: the right slope over the whole line and
  // the difference (a, U, V, h below) over u >= 0, v1 = <u . psi>, v2 = <u^2 . psi> of it
  const Half a = half_line(g, 1.0);
  L.a -= N.a; L.U -= N.U; L.V -= N.V; L.h -= N.h;
  const double m4 = g.U * a.m3 + 3.0 * (g.h * a.m2), kk = 2.0 * g.h + (0.5 * g.V) * g.V;
  const double P1 = L.a * a.m1 + (L.U * a.m0 + (0.5 * L.h) * a.f);
  const double P2 = L.a * a.m2 + (2.0 * (L.U * a.m1) + L.h * a.m0);
  const double P3 = L.a * a.m3 + 3.0 * (L.U * a.m2 + L.h * a.m1);
  const double P4 = L.a * m4 + 2.0 * (2.0 * (L.U * a.m3) + 3.0 * (L.h * a.m2));
  const double Q1 = L.V * a.m1, Q2 = L.V * a.m2;
  const double E1 = 0.5 * P3 + (kk * P1 + (g.V * Q1 + 2.0 * (L.h * a.m1)));
  const double E2 = 0.5 * P4 + (kk * P2 + (g.V * Q2 + 2.0 * (L.h * a.m2)));
  // Eq. 12: minus the time slope is R (right and tangential slopes) plus that of v1
  const double DU = P2 - g.U * P1;
  const double Dh = HK * (E1 - g.et * P1 - g.U * DU - g.V * Q1);

  // collision time (Eq. 33-34 with the pressure-jump term) and the time weights of Eq. 13
  double tau = (visc(g.h, g.s) + mut) * ((g.s * g.s) * g.ir);
  if (c_num != 0.0) {
    const double pL = gl.r * gl.h, pR = gr.r * gr.h;
    tau += c_num * fabs(pL - pR) * __drcp_rn(pL + pR) * dt;
  }
  const double ome = -expm1(-(dt * __drcp_rn(tau)));   // 1 - e^{-dt/tau}
  const double e = 1.0 - ome, to = tau * ome, td = tau * dt;
  const double q0 = dt - to;
  const double q1 = 2.0 * (tau * to) - td * (1.0 + e);
  const double q2 = 0.5 * dt * dt - td + tau * to;
  const double q4 = td * e - 2.0 * (tau * to);
  const double n54 = q4 + tau * to;                    // q4 - q5, q5 = -tau^2 (1 - e^{-dt/tau}); q3 = to

  // Eq. 14 and the state integrals for the heat flux: the equilibrium part over the whole
  // line, q0 + q1 (D - A) + q2 (A + A of the difference), R = -A
  Out o;
  {
    const double v0 = g.r * q0, v1 = g.r * q1, e2 = -(g.r * q2), e1 = v1 + e2;
    const double v1h = v1 * g.h;
    const double b0 = v0 + (e1 * R.A + e2 * P1);
    const double b1 = e1 * R.U + e2 * DU;
    const double d0 = e1 * R.V + e2 * Q1;
    const double th = e1 * R.h + e2 * Dh;
    const double k = v1h * R.st;
    const double b2 = 0.5 * th + k, b3 = (0.5 * v1h) * R.qn, d1 = v1h * R.sh, x = 2.0 * th - k;
    const double M2 = g.U * g.U + g.h, M3 = g.U * (M2 + 2.0 * g.h);
    const double F0 = b0 * g.U + b1;
    const double F1 = b0 * M2 + 2.0 * (b1 * g.U + b2);
    const double F3 = b0 * M3 + 3.0 * (b1 * M2 + 2.0 * (b2 * g.U + b3));
    const double T1 = d0 * g.U + d1;
    o.F0 = F0 + v1 * P2;
    o.F1 = F1 + v1 * P3;
    o.F2 = g.V * F0 + (T1 + v1 * (g.V * P2 + Q2));
    o.F3 = 0.5 * F3 + (kk * F0 + (g.V * T1 + (x * g.U + (4.0 * b3 + v1 * E2))));
    o.S0 = b0 + v1 * P1;
    o.S2 = g.V * b0 + (d0 + v1 * (g.V * P1 + Q1));
    o.S3 = 0.5 * F1 + (kk * b0 + (g.V * d0 + (x + v1 * E1)));
  }
  side_flux(gl, hl, Rl, gl.r * to, gl.r * q4, gl.r * n54, o);
  side_flux(gr, hr, Rr, gr.r * to, gr.r * q4, gr.r * n54, o);
  // heat flux about (U0, V0) and the Prandtl-number fix
  const double he = 0.5 * (g.U * g.U + g.V * g.V);
  const double heat = o.F3 - g.U * o.F1 - g.V * o.F2 + he * o.F0 -
                      g.U * (o.S3 - g.U * o.F0 - g.V * o.S2 + he * o.S0);
  Fn[0] = o.F0;
  Fn[1] = o.F1;
  Fn[2] = o.F2;
  Fn[3] = o.F3 + pr_fix * heat;
}

}  // namespace gks
}  // namespace igks
