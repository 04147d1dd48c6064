// igks_flux.cu -- BGK-NS gas-kinetic interface flux (Eq. 1-14, 33-34) and the
// Spalart-Allmaras face terms (Eq. 28-30) on sm_103a, one thread per face.
//
// Per face: reconstruct both sides at the face midpoint from the limited least-squares
// gradients (Eq. 10), rotate into the face frame, take the time-integrated flux of Eq. 4-14
// with the Prandtl-number fix, rotate back and scale by the face length.
//
// The kernel is bound by FP64 arithmetic, not by HBM: it reads ~250 B and writes ~80 B per
// face. What does not need the FP64 pipe stays off it: limited gradients come from the
// gradient kernel, signs are taken from the sign bit (an FP64 maximum costs as much as a
// multiply-add).
//
// Two kernels: k_flux (igks_gks.cuh) for FP64 and double-float sweeps, k_flux_moment
// (igks_gks_moment.cuh) for mixed precision, whose iterates keep their bits.
#include <cmath>
#include <vector>

#include "igks_dev.h"
#include "igks_gks.cuh"
#include "igks_gks_moment.cuh"
#include "igks_phys.cuh"

namespace igks {

// momentum of a conserved 4-vector (or of its slope) into the face frame (n, t)
__device__ __forceinline__ void rot(const double* g, double nx, double ny, double* o) {
  o[0] = g[0];
  o[1] = g[1] * nx + g[2] * ny;
  o[2] = -g[1] * ny + g[2] * nx;
  o[3] = g[3];
}

// x where it is positive / negative, else zero (by the sign bit)
__device__ __forceinline__ double pos_part(double x) { return __double2hiint(x) < 0 ? 0.0 : x; }
__device__ __forceinline__ double neg_part(double x) { return __double2hiint(x) < 0 ? x : 0.0; }

// state and slopes of a cell's side of the face: reconstruction (Eq. 10), rotation
__device__ __forceinline__ void side_of(const Dev& d, const double* gr, int c, double mx, double my, double nx,
                                        double ny, double* Wc, double* W, double* Sn, double* St) {
  const int n = d.nc_pad;
  double g[4], sn[4], st[4];
  const double ox = mx - d.cx[c], oy = my - d.cy[c];
#pragma unroll
  for (int v = 0; v < 5; v++) Wc[v] = d.W[v * n + c];
#pragma unroll
  for (int v = 0; v < 4; v++) {
    const double gx = gr[(2 * v) * n + c], gy = gr[(2 * v + 1) * n + c];
    g[v] = Wc[v] + (gx * ox + gy * oy);
    sn[v] = gx * nx + gy * ny;
    st[v] = gy * nx - gx * ny;
  }
  rot(g, nx, ny, W);
  rot(sn, nx, ny, Sn);
  rot(st, nx, ny, St);
}

__global__ void __launch_bounds__(128, 1) k_flux(Dev d) {
  chain_wait();
  const int f = d.g_face0 + blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= d.g_face0 + d.g_nface) return;
  const int s = d.fsolve[f];
  if (d.st[s].state != 0) return;
  const DevFlow& fl = d.flow[s];
  const int nf = d.nf;
  const int L = d.fL[f], R = d.fR[f], bc = d.fbc[f];
  const double nx = d.fnx[f], ny = d.fny[f];
  const double S = d.fS[f], mxf = d.fmx[f], myf = d.fmy[f];
  const double idL = d.fidL[f], idR = d.fidR[f];
  const double dt = __longlong_as_double((long long)d.dt_bits[s]);
  const double* gr = fl.limiter ? d.lgrad : d.grad;   // limited gradients

  double WcLg[5], WcL[4], WL[4], SLn[4], SLt[4];
  side_of(d, gr, L, mxf, myf, nx, ny, WcLg, WL, SLn, SLt);
  rot(WcLg, nx, ny, WcL);
  // right side: interior cell, mirrored ghost (wall, symmetry, moving wall) or the
  // free-stream / outflow ghost state without slopes
  double WcRg[5], WcR[4], WR[4], SRn[4], SRt[4];
  double nuR, mtR, vnR;            // kinematic viscosity, eddy viscosity, centre normal velocity
  if (R >= 0) {
    side_of(d, gr, R, mxf, myf, nx, ny, WcRg, WR, SRn, SRt);
    nuR = d.nul[R];
    mtR = d.mu_t[R];
    vnR = d.pu[R] * nx + d.pv[R] * ny;
  } else {
#pragma unroll
    for (int v = 0; v < 5; v++) WcRg[v] = d.G[v * nf + f];
    const double ir = __drcp_rn(WcRg[0]);
    nuR = d.Gmu[f] * ir;
    mtR = d.Gmu[nf + f];
    vnR = (WcRg[1] * nx + WcRg[2] * ny) * ir;
    if (bc == 2 || bc == 3 || bc == 5) {
      const double st2 = (bc == 2) ? 1.0 : -1.0;
      WR[0] = WL[0]; WR[1] = -WL[1]; WR[2] = st2 * WL[2]; WR[3] = WL[3];
      if (bc == 5) {   // moving wall: tangential velocity mirrored about the wall velocity
        const double uw = (fl.Winf[2] * nx - fl.Winf[1] * ny) / fl.Winf[0];
        const double ut = WL[2] / WL[0], utg = 2.0 * uw - ut;
        WR[2] = WL[0] * utg;
        WR[3] = WL[3] - 0.5 * WL[0] * ut * ut + 0.5 * WL[0] * utg * utg;
      }
      SRn[0] = -SLn[0]; SRn[1] = SLn[1]; SRn[2] = -st2 * SLn[2]; SRn[3] = -SLn[3];
      SRt[0] = SLt[0]; SRt[1] = -SLt[1]; SRt[2] = st2 * SLt[2]; SRt[3] = SLt[3];
    } else {
      rot(WcRg, nx, ny, WR);
#pragma unroll
      for (int v = 0; v < 4; v++) { SRn[v] = 0.0; SRt[v] = 0.0; }
    }
  }
  rot(WcRg, nx, ny, WcR);

  // ---- Eq. 4-14: the time-integrated flux in the face frame ----
  double Fn[4];
  gks::face_flux(WL, WR, SLn, SLt, SRn, SRt, WcL, WcR, idL, idR, 0.5 * (d.mu_t[L] + mtR), dt, fl.c_num, fl.pr_fix,
                 [&](double h, double is) { return fl.visc_c * (h * h) * is * __drcp_rn(fl.tr_h * h + fl.s_star); },
                 Fn);

  // ---- back to the global frame, times the face length ----
  d.F[f] = Fn[0] * S;
  d.F[nf + f] = (Fn[1] * nx - Fn[2] * ny) * S;
  d.F[2 * nf + f] = (Fn[1] * ny + Fn[2] * nx) * S;
  d.F[3 * nf + f] = Fn[3] * S;

  // ---- SA face terms (Eq. 28-30) and the coefficients of its implicit system ----
  double o4 = 0.0, o5 = 0.0, aLR = 0.0, aRL = 0.0, dgl = 0.0, dgr = 0.0;
  if (fl.sa_on) {
    const double idn = __drcp_rn(d.fdn[f]);
    const double vni = d.pu[L] * nx + d.pv[L] * ny, vnj = vnR;
    const double gradn = (WcRg[4] - WcLg[4]) * idn;
    const double vip = pos_part(vni), vjn = neg_part(vnj);
    const double finv = vip * WcLg[4] + vjn * WcRg[4];
    const double kap = 1.0 / (2.0 * SA_SIGMA) * ((d.nul[L] + nuR) + (1.0 + SA_CB2) * (WcLg[4] + WcRg[4]));
    const double net = S * (kap * gradn - finv), cg = (SA_CB2 / SA_SIGMA * S) * gradn;
    o4 = net - cg * WcLg[4];
    o5 = cg * WcRg[4] - net;
    const double kd = kap * idn;
    aLR = S * (vjn - kd);
    aRL = S * (neg_part(-vni) - kd);
    dgl = S * (vip + kd);
    dgr = S * (pos_part(-vnj) + kd);
  }
  d.F[4 * nf + f] = o4;
  d.F[5 * nf + f] = o5;
  d.sa_a[f] = aLR;
  d.sa_a[nf + f] = aRL;
  d.sa_a[2 * nf + f] = dgl;
  d.sa_a[3 * nf + f] = dgr;
}

__global__ void __launch_bounds__(128, 1) k_flux_moment(Dev d) {
  chain_wait();
  const int f = d.g_face0 + blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= d.g_face0 + d.g_nface) return;
  const int s = d.fsolve[f];
  if (d.st[s].state != 0) return;
  const DevFlow& fl = d.flow[s];
  const int n = d.nc_pad, nf = d.nf;
  const int L = d.fL[f], R = d.fR[f], bc = d.fbc[f];
  const double nx = d.fnx[f], ny = d.fny[f], tx = -ny, ty = nx;
  const double S = d.fS[f], mxf = d.fmx[f], myf = d.fmy[f];
  const double idL = d.fidL[f], idR = d.fidR[f];
  const double dt = __longlong_as_double((long long)d.dt_bits[s]);
  const double* gr = fl.limiter ? d.lgrad : d.grad;   // limited gradients

  // ---- left side: centre state, reconstruction (Eq. 10), slopes, rotation ----
  double WcLg[5], WcL[4], WL[4], SLn[4], SLt[4];
  {
    double g[4], sn[4], stt[4];
    const double ox = mxf - d.cx[L], oy = myf - d.cy[L];
#pragma unroll
    for (int v = 0; v < 5; v++) WcLg[v] = d.W[v * n + L];
#pragma unroll
    for (int v = 0; v < 4; v++) {
      double gx = gr[(2 * v) * n + L], gy = gr[(2 * v + 1) * n + L];
      g[v] = WcLg[v] + gx * ox + gy * oy;
      sn[v] = gx * nx + gy * ny;
      stt[v] = gx * tx + gy * ty;
    }
    rot(g, nx, ny, WL);
    rot(sn, nx, ny, SLn);
    rot(stt, nx, ny, SLt);
    rot(WcLg, nx, ny, WcL);
  }
  // ---- right side: interior cell, mirrored ghost (wall, symmetry, moving wall) or the
  //      free-stream / outflow ghost state without slopes ----
  double WcRg[5], WcR[4], WR[4], SRn[4], SRt[4];
  double muR, mtR;
  if (R >= 0) {
    double g[4], sn[4], stt[4];
    const double ox = mxf - d.cx[R], oy = myf - d.cy[R];
#pragma unroll
    for (int v = 0; v < 5; v++) WcRg[v] = d.W[v * n + R];
#pragma unroll
    for (int v = 0; v < 4; v++) {
      double gx = gr[(2 * v) * n + R], gy = gr[(2 * v + 1) * n + R];
      g[v] = WcRg[v] + gx * ox + gy * oy;
      sn[v] = gx * nx + gy * ny;
      stt[v] = gx * tx + gy * ty;
    }
    rot(g, nx, ny, WR);
    rot(sn, nx, ny, SRn);
    rot(stt, nx, ny, SRt);
    muR = d.mu_l[R];
    mtR = d.mu_t[R];
  } else {
#pragma unroll
    for (int v = 0; v < 5; v++) WcRg[v] = d.G[v * nf + f];
    muR = d.Gmu[f];
    mtR = d.Gmu[nf + f];
    if (bc == 2 || bc == 3 || bc == 5) {
      const double st2 = (bc == 2) ? 1.0 : -1.0;
      WR[0] = WL[0]; WR[1] = -WL[1]; WR[2] = st2 * WL[2]; WR[3] = WL[3];
      if (bc == 5) {   // moving wall: tangential velocity mirrored about the wall velocity
        const double uw = (fl.Winf[1] * tx + fl.Winf[2] * ty) / fl.Winf[0];
        const double ut = WL[2] / WL[0], utg = 2.0 * uw - ut;
        WR[2] = WL[0] * utg;
        WR[3] = WL[3] - 0.5 * WL[0] * ut * ut + 0.5 * WL[0] * utg * utg;
      }
      SRn[0] = -SLn[0]; SRn[1] = SLn[1]; SRn[2] = -st2 * SLn[2]; SRn[3] = -SLn[3];
      SRt[0] = SLt[0]; SRt[1] = -SLt[1]; SRt[2] = st2 * SLt[2]; SRt[3] = SLt[3];
    } else {
      rot(WcRg, nx, ny, WR);
#pragma unroll
      for (int v = 0; v < 4; v++) { SRn[v] = 0.0; SRt[v] = 0.0; }
    }
  }
  rot(WcRg, nx, ny, WcR);
  const double mut_face = gks_moment::hlf(d.mu_t[L] + mtR);

  // ---- Eq. 4-14: the time-integrated flux in the face frame ----
  double Fn[4];
  gks_moment::face_flux(WL, WR, SLn, SLt, SRn, SRt, WcL, WcR, idL, idR, mut_face, dt, fl.c_num, fl.pr_fix,
                        [&](double h2) { return viscosity_h2(fl, h2); }, Fn);

  // ---- back to the global frame, times the face length ----
  d.F[f] = Fn[0] * S;
  d.F[nf + f] = (Fn[1] * nx - Fn[2] * ny) * S;
  d.F[2 * nf + f] = (Fn[1] * ny + Fn[2] * nx) * S;
  d.F[3 * nf + f] = Fn[3] * S;

  // ---- SA face terms (Eq. 28-30) and the coefficients of its implicit system ----
  double o4 = 0.0, o5 = 0.0, aLR = 0.0, aRL = 0.0, dgl = 0.0, dgr = 0.0;
  if (fl.sa_on) {
    const double idn = __drcp_rn(d.fdn[f]);
    const double irl = __drcp_rn(WcLg[0]), irr = __drcp_rn(WcRg[0]);
    const double vni = (WcLg[1] * nx + WcLg[2] * ny) * irl;
    const double vnj = (WcRg[1] * nx + WcRg[2] * ny) * irr;
    const double nui = d.mu_l[L] * irl, nuj = muR * irr;
    const double gradn = (WcRg[4] - WcLg[4]) * idn;
    const double finv = pos_part(vni) * WcLg[4] + neg_part(vnj) * WcRg[4];
    const double kap = 1.0 / (2.0 * SA_SIGMA) * ((nui + nuj) + (1.0 + SA_CB2) * (WcLg[4] + WcRg[4]));
    const double fvis = kap * gradn;
    const double fadl = SA_CB2 / SA_SIGMA * WcLg[4] * gradn;
    const double fadr = SA_CB2 / SA_SIGMA * WcRg[4] * (-gradn);
    o4 = (-finv + fvis - fadl) * S;
    o5 = (finv - fvis - fadr) * S;
    const double kd = kap * idn;
    aLR = S * (neg_part(vnj) - kd);
    aRL = S * (neg_part(-vni) - kd);
    dgl = S * (pos_part(vni) + kd);
    dgr = S * (pos_part(-vnj) + kd);
  }
  d.F[4 * nf + f] = o4;
  d.F[5 * nf + f] = o5;
  d.sa_a[f] = aLR;
  d.sa_a[nf + f] = aRL;
  d.sa_a[2 * nf + f] = dgl;
  d.sa_a[3 * nf + f] = dgr;
}

// The nodes of gks::normal_tail in extended precision: c_0 = Q(z), c_(n+1) =
// (-1)^(n+1) He_n(z) phi(z) / (n + 1)!, He_(n+1) = z He_n - n He_(n-1).
static std::vector<double> tail_table() {
  std::vector<double> t(8 * (size_t)gks::TAIL_NODES, 0.0);
  for (int k = 0; k < gks::TAIL_NODES; k++) {
    const long double z = (long double)k / gks::TAIL_PER_UNIT;
    const long double phi = std::exp(-0.5L * z * z) * 0.39894228040143267793994605993438187L;
    double* c = t.data() + 8 * (size_t)k;
    c[0] = (double)(0.5L * std::erfc(z * 0.70710678118654752440084436210484904L));
    long double h0 = 0.0L, h1 = 1.0L, w = -phi;
    for (int n = 0; n < 6; n++) {
      w /= n + 1;
      c[n + 1] = (double)(w * h1);
      w = -w;
      const long double h2 = z * h1 - n * h0;
      h0 = h1;
      h1 = h2;
    }
  }
  return t;
}

// Every context uploads the table on its own stream, ahead of its kernels (192 KiB, always
// the same bytes): nothing is assumed about what other contexts, streams or a device reset
// before have left in it. Only the host's copy is kept.
cudaError_t upload_flux_table(cudaStream_t s) {
  static const std::vector<double> t = tail_table();
  return cudaMemcpyToSymbolAsync(gks::g_tail, t.data(), t.size() * sizeof(double), 0, cudaMemcpyHostToDevice, s);
}

void launch_flux(const Dev& d, int precision, cudaStream_t s) {
  // one-warp blocks by default: the FP64 pipe is shared by an SM, and whole warps spread a small
  // mesh over the SMs most evenly (20,200 faces: 55 us with blocks of 128, 43 with 32; the same from
  // 35,000 faces on)
  const int b = d.flux_block > 0 ? d.flux_block : 32;
  if (!d.g_nface) return;
  if (precision == 1) launch_chained(d.chained, k_flux_moment, (d.g_nface + b - 1) / b, b, 0, s, d);
  else launch_chained(d.chained, k_flux, (d.g_nface + b - 1) / b, b, 0, s, d);
}

}  // namespace igks
