// igks_sweep.cu -- matrix-free LU-SGS forward and backward sweeps (Eq. 19-22 for the
// mean flow, Eq. 31-32 for the SA variable) with the FP64 state update, in FP64, FP32 or
// double-float.
//
// Each sweep visits the cells in the dependency order of the sequential sweep of Eq. 20
// (cell i needs its lower neighbours j < i forward, its upper neighbours j > i backward),
// grouped into levels of mutually independent cells. Everything that does not depend on
// the unknowns is formed first by a parallel pre-pass (1/D, velocities, enthalpy, the
// signed face coefficients of every cell's stencil), so the dependency chain carries only
// the neighbour contributions, one multiply by 1/D and the incremental flux of the new
// increment. On GB300 each warp-wide FP64 instruction costs the same whatever the number
// of active lanes, so the chain's FP64 instruction count sets the time of a level.
//
// Two schedules:
//  - narrow: one block per solve (or a thread-block cluster) walks its levels with a
//    barrier between them (for orderings with hundreds of thin levels). Two threads work on
//    a cell; the increments of the last cells it produced stay in a shared-memory ring, so
//    a cell usually reads its neighbours' increments from shared memory; its record (stencil
//    neighbours, ring slots, coefficients and per-cell constants) is stored in
//    sweep-position order, and records are brought into shared memory by bulk copies on
//    mbarriers several levels ahead, and into registers one level ahead;
//  - wide: one launch per level covering that level's cells of every solve (for low-depth
//    orderings, e.g. multicolour, whose few levels hold thousands of cells each).
#include <cooperative_groups.h>
#include <float.h>

#include <algorithm>
#include <cstddef>
#include <type_traits>

#include "igks_df64.cuh"
#include "igks_dev.h"
#include "igks_phys.cuh"

namespace cg = cooperative_groups;

namespace igks {

// The sweeps' arithmetic is written with explicitly rounded operations (fma_x, mul_x,
// add_x: __fma_rn / __dmul_rn / __dadd_rn in FP64, the __f*_rn intrinsics in FP32, the
// double-float operators): the compiler may not fuse or split them, so every schedule (one
// block or a cluster of blocks per solve, one launch per level) and every inlining
// context gives the same bits for the same cell.
__device__ __forceinline__ double fma_x(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double mul_x(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double add_x(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float fma_x(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float mul_x(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float add_x(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ df64 fma_x(df64 a, df64 b, df64 c) { return a * b + c; }
__device__ __forceinline__ df64 mul_x(df64 a, df64 b) { return a * b; }
__device__ __forceinline__ df64 add_x(df64 a, df64 b) { return a + b; }
// 1 / x, correctly rounded (the bits of the division in FP64 and FP32, fewer instructions)
__device__ __forceinline__ double rcp_x(double x) { return __drcp_rn(x); }
__device__ __forceinline__ float rcp_x(float x) { return __frcp_rn(x); }
__device__ __forceinline__ df64 rcp_x(df64 x) { return df64(1.0f, 0.0f) / x; }

// Increment of the x and y Euler fluxes for the increment (dr, dmx, dmy, dE) of a state
// with density r, momenta mx, my, velocity u, v and total enthalpy density H = E + p,
// written without differences of large numbers. o = {x mass, y mass, x x-mom, y x-mom,
// x y-mom, y y-mom, x energy, y energy}.
template <class T>
__device__ __forceinline__ void delta_flux(T r, T mx, T my, T u, T v, T H, T dr, T dmx, T dmy, T dE, T* o) {
  const T g1 = (T)(GAMMA - 1.0);
  const T inv1 = rcp_x(add_x(r, dr));
  const T du = mul_x(fma_x(-u, dr, dmx), inv1);          // (dmx - u dr) / (r + dr)
  const T dv = mul_x(fma_x(-v, dr, dmy), inv1);
  const T u1 = add_x(u, du), v1 = add_x(v, dv);
  const T dmxu = fma_x(dmx, u1, mul_x(mx, du));          // increment of mx u
  const T dmyv = fma_x(dmy, v1, mul_x(my, dv));          // increment of my v
  const T dp = mul_x(g1, fma_x((T)(-0.5), add_x(dmxu, dmyv), dE));
  const T dH = add_x(dE, dp);
  o[0] = dmx;
  o[1] = dmy;
  o[2] = add_x(dmxu, dp);
  o[3] = fma_x(dmx, v1, mul_x(mx, dv));
  o[4] = fma_x(dmy, u1, mul_x(my, du));
  o[5] = add_x(dmyv, dp);
  o[6] = fma_x(dH, u1, mul_x(H, du));
  o[7] = fma_x(dH, v1, mul_x(H, dv));
}

// Contribution of one stencil entry to a cell's sweep sum: (1/2) S (dF . n - lambda dW)
// for the mean flow (sx, sy = signed S n / 2, sl = S lambda / 2) and a_ij dnu for SA,
// subtracted from (forward) or added to (backward) the cell's accumulator. Every schedule
// applies the entries of a cell with these helpers in the same order, so a solve gives
// the same bits whichever schedule runs it (alone or in a batch).
// One component v of an entry: f0, f1 = the x and y flux increments of component v, w its
// increment (fwd subtracts, bwd adds); the SA row has its scalar coefficient. The
// schedules that split a cell's components over threads call these per component, so
// every schedule does the same arithmetic.
template <class T>
__device__ __forceinline__ T entry_sum(T sx, T sy, T sl, T f0, T f1, T w) {   // sx f0 + sy f1 - sl w
  return fma_x(sx, f0, fma_x(sy, f1, -mul_x(sl, w)));
}
template <class T>
__device__ __forceinline__ void fwd_comp(T& a, T sx, T sy, T sl, T f0, T f1, T w) {
  a = add_x(a, -entry_sum(sx, sy, sl, f0, f1, w));
}
template <class T>
__device__ __forceinline__ void bwd_comp(T& a, T sx, T sy, T sl, T f0, T f1, T w) {
  a = add_x(a, entry_sum(sx, sy, sl, f0, f1, w));
}
// FP64: three fused multiply-adds onto the accumulator (a warp-wide FP64 instruction costs
// an SM 19 cycles whatever its active lanes: three instead of four per entry and component)
template <>
__device__ __forceinline__ void fwd_comp<double>(double& a, double sx, double sy, double sl, double f0, double f1,
                                                 double w) {
  a = fma_x(-sx, f0, fma_x(-sy, f1, fma_x(sl, w, a)));
}
template <>
__device__ __forceinline__ void bwd_comp<double>(double& a, double sx, double sy, double sl, double f0, double f1,
                                                 double w) {
  a = fma_x(sx, f0, fma_x(sy, f1, fma_x(-sl, w, a)));
}
template <class T>
__device__ __forceinline__ void fwd_sa(T& a, T sa, T w) { a = fma_x(-sa, w, a); }
template <class T>
__device__ __forceinline__ void bwd_sa(T& a, T sa, T w) { a = fma_x(sa, w, a); }

// A cell's increments from its accumulators: one rounded product (forward), one fused
// multiply-add (backward). Written with explicitly rounded operations so that the compiler
// cannot fuse the product into the arithmetic that consumes the increment (the flux
// increment of the same thread): a schedule that takes the increments from other threads
// by shuffles must get the same bits.
template <class T>
__device__ __forceinline__ T inc_fwd(T acc, T c);
template <>
__device__ __forceinline__ double inc_fwd<double>(double acc, double c) { return __dmul_rn(acc, c); }
template <>
__device__ __forceinline__ float inc_fwd<float>(float acc, float c) { return __fmul_rn(acc, c); }
template <>
__device__ __forceinline__ df64 inc_fwd<df64>(df64 acc, df64 c) { return acc * c; }
template <class T>
__device__ __forceinline__ T inc_bwd(T ws, T acc, T c);   // ws - acc c
template <>
__device__ __forceinline__ double inc_bwd<double>(double ws, double acc, double c) { return __fma_rn(-acc, c, ws); }
template <>
__device__ __forceinline__ float inc_bwd<float>(float ws, float acc, float c) { return __fmaf_rn(-acc, c, ws); }
template <>
__device__ __forceinline__ df64 inc_bwd<df64>(df64 ws, df64 acc, df64 c) { return ws - acc * c; }

template <class T>
__device__ __forceinline__ void fwd_acc(T* acc, T sx, T sy, T sl, T sa, const T* f, const T* w, bool sa_on) {
#pragma unroll
  for (int v = 0; v < 4; v++) fwd_comp<T>(acc[v], sx, sy, sl, f[2 * v], f[2 * v + 1], w[v]);
  if (sa_on) fwd_sa<T>(acc[4], sa, w[4]);
}

template <class T>
__device__ __forceinline__ void bwd_acc(T* acc, T sx, T sy, T sl, T sa, const T* f, const T* w, bool sa_on) {
#pragma unroll
  for (int v = 0; v < 4; v++) bwd_comp<T>(acc[v], sx, sy, sl, f[2 * v], f[2 * v + 1], w[v]);
  if (sa_on) bwd_sa<T>(acc[4], sa, w[4]);
}

// The same two for double-float: every product is accumulated exactly into the running
// high part (two-sum), its rounding errors and the product's low part into the running low
// part, without renormalising after each term (the multiply that uses the sum does).
__device__ __forceinline__ void df_mac(df64& acc, df64 a, df64 b) {   // acc += a b
  const float p = __fmul_rn(a.hi, b.hi);
  float pe = __fmaf_rn(a.hi, b.hi, -p);
  pe = __fmaf_rn(a.hi, b.lo, pe);
  pe = __fmaf_rn(a.lo, b.hi, pe);
  const float s = __fadd_rn(acc.hi, p);
  const float bb = __fsub_rn(s, acc.hi);
  const float e = __fadd_rn(__fsub_rn(acc.hi, __fsub_rn(s, bb)), __fsub_rn(p, bb));
  acc.hi = s;
  acc.lo = __fadd_rn(acc.lo, __fadd_rn(e, pe));
}

template <>
__device__ __forceinline__ void fwd_comp<df64>(df64& a, df64 sx, df64 sy, df64 sl, df64 f0, df64 f1, df64 w) {
  df_mac(a, -sx, f0);
  df_mac(a, -sy, f1);
  df_mac(a, sl, w);
}
template <>
__device__ __forceinline__ void bwd_comp<df64>(df64& a, df64 sx, df64 sy, df64 sl, df64 f0, df64 f1, df64 w) {
  df_mac(a, sx, f0);
  df_mac(a, sy, f1);
  df_mac(a, -sl, w);
}
template <>
__device__ __forceinline__ void fwd_sa<df64>(df64& a, df64 sa, df64 w) { df_mac(a, -sa, w); }
template <>
__device__ __forceinline__ void bwd_sa<df64>(df64& a, df64 sa, df64 w) { df_mac(a, sa, w); }

// The four mean-flow terms of a wall or symmetry ghost are formed ahead of the backward
// sweep's dependency chain (they need the cell's own forward increment only) and added at
// the entry's place in the order.
template <class T>
__device__ __forceinline__ void ghost_add(T& a, T term) { a = add_x(a, term); }
template <>
__device__ __forceinline__ void ghost_add<df64>(df64& a, df64 term) { df_mac(a, df64(1.0f, 0.0f), term); }

// the first BYTES bytes of src to dst (both 16-byte aligned) as 16-byte stores
template <size_t BYTES>
__device__ __forceinline__ void store_chunks(void* dst, const void* src) {
  static_assert(BYTES % 16 == 0, "whole chunks");
#pragma unroll
  for (int k = 0; k < (int)(BYTES / 16); k++)
    reinterpret_cast<uint4*>(dst)[k] = reinterpret_cast<const uint4*>(src)[k];
}

// A cell's increments in dWs and dW: in FP32 together (INC_STRIDE floats a cell, one 16-byte and
// one 4-byte access; five rows cost the narrow sweeps' store warps five stores each: the 60,160-cell
// O-mesh backward 516 -> 453 us), the 8-byte types in rows [5][nc_pad].
template <class T>
__device__ __forceinline__ int inc_at(int n, int v, int i) {
  return sizeof(T) == 4 ? INC_STRIDE * i + v : v * n + i;
}
template <class T>
__device__ __forceinline__ void load_incs(T* w, const T* a, int n, int i) {
  if constexpr (sizeof(T) == 4) {
    const float4 q = *reinterpret_cast<const float4*>(a + inc_at<T>(n, 0, i));
    w[0] = q.x; w[1] = q.y; w[2] = q.z; w[3] = q.w;
    w[4] = a[inc_at<T>(n, 4, i)];
  } else {
#pragma unroll
    for (int v = 0; v < 5; v++) w[v] = a[inc_at<T>(n, v, i)];
  }
}
template <class T>
__device__ __forceinline__ void store_incs(T* a, int n, int i, const T* w, T w4) {
  if constexpr (sizeof(T) == 4) {
    *reinterpret_cast<float4*>(a + inc_at<T>(n, 0, i)) = make_float4(w[0], w[1], w[2], w[3]);
  } else {
#pragma unroll
    for (int v = 0; v < 4; v++) a[inc_at<T>(n, v, i)] = w[v];
  }
  a[inc_at<T>(n, 4, i)] = w4;
}

// ---- pre-pass: per-cell constants and the signed stencil of every cell ----
template <class T>
__global__ void __launch_bounds__(CELL_BLOCK) k_sweep_prep(Dev d) {
  chain_wait();
  const int i = (d.g_blk0 + blockIdx.x) * CELL_BLOCK + threadIdx.x;
  if (i >= d.nc_pad) return;
  const int s = d.cell_solve[i];
  if (s < 0 || d.st[s].state != 0 || d.flow[s].scheme == 1) return;   // explicit solves: no sweeps
  const DevFlow& fl = d.flow[s];
  const int n = d.nc_pad, nf = d.nf;
  const double Lam = d.Lam[i];
  const double r = d.W[i], mx = d.W[n + i], my = d.W[2 * n + i], E = d.W[3 * n + i];
  const double u = d.pu[i], v = d.pv[i];          // mx / r, my / r (k_prep)
  const double p = (GAMMA - 1.0) * (E - 0.5 * (mx * u + my * v));
  T cc[5];
  const double lc = Lam * d.st[s].icfl;                                 // Omega / dt_imp (Eq. 24)
  cc[0] = (T)__drcp_rn(lc + Lam);                                        // 1/D (Eq. 20)
  cc[1] = fl.sa_on ? (T)__drcp_rn(lc + d.sa_diag[i]) : (T)0;             // 1/a_ii (Eq. 32)
  cc[2] = (T)u;
  cc[3] = (T)v;
  cc[4] = (T)(E + p);
  const bool wide = d.wide != 0;
  if (wide) {   // the one-launch-per-level sweeps read the cell constants in cell order
    T* c = (T*)d.sw_cell;
#pragma unroll
    for (int q = 0; q < 5; q++) c[q * n + i] = cc[q];
  }
  // position-ordered records of the narrow schedule: the heads as whole 16-byte chunks
  // (the backward head's dW* is written by the forward sweep afterwards)
  const int pf = d.pos_f[i], pb = d.pos_b[i];
  SweepRec<T>* rf = (SweepRec<T>*)d.frec + pf;
  SweepRec<T>* rb = (SweepRec<T>*)d.brec + pb;
  if (!wide) {
    constexpr size_t HEAD = offsetof(SweepRec<T>, co) - offsetof(SweepRec<T>, m);
    SweepRec<T> h;
    h.w[0] = (T)r; h.w[1] = (T)mx; h.w[2] = (T)my;
#pragma unroll
    for (int q = 0; q < 5; q++) { h.c[q] = cc[q]; h.m[q] = (T)0; }
    for (int q = 0; q < (int)(sizeof(h.pad0) / sizeof(T)); q++) h.pad0[q] = (T)0;
    store_chunks<HEAD>(rb->m, h.m);
#pragma unroll
    for (int q = 0; q < 5; q++) h.m[q] = (T)d.M[q * n + i];
    store_chunks<HEAD>(rf->m, h.m);
  }
  T* sc = (T*)d.sw_st;
  const int nnz = d.nnz;
  for (int k = d.cf_ptr[i]; k < d.cf_ptr[i + 1]; k++) {
    const int f = d.cf_face[k];
    const bool own = (d.fL[f] == i);
    const int j = own ? d.fR[f] : d.fL[f];
    const double hS = 0.5 * d.fS[f];
    const double sg = own ? hS : -hS;
    const T e0 = (T)(sg * d.fnx[f]), e1 = (T)(sg * d.fny[f]), e2 = (T)(hS * d.lam_f[f]);
    const T e3 = (T)d.sa_a[(own ? 0 : 1) * nf + f];
    if (wide) {   // the cell-ordered stencil of the one-launch-per-level sweeps
      d.sw_j[k] = j;                                  // -1 on a boundary face
      sc[k] = e0; sc[nnz + k] = e1; sc[2 * nnz + k] = e2; sc[3 * nnz + k] = e3;
    } else {
      // the narrow schedule: up to PF_E entries per position in its record; a larger stencil
      // and the ghosts in the position-ordered CSR lists
      const int ef = d.cf_to_fs[k], eb = d.cf_to_bs[k];
      const int xf = d.cf_to_ef[k], xb = d.cf_to_eb[k];   // record entry: position * PF_E + e
      if (ef >= 0 && xf < 0) {
        T* o = (T*)d.sc_f;
        o[ef] = e0; o[d.nfs + ef] = e1; o[2 * d.nfs + ef] = e2; o[3 * d.nfs + ef] = e3;
      }
      if (eb >= 0 && (xb < 0 || j < 0)) {
        T* o = (T*)d.sc_b;
        o[eb] = e0; o[d.nbs + eb] = e1; o[2 * d.nbs + eb] = e2; o[3 * d.nbs + eb] = e3;
      }
      alignas(16) const T ent[4] = {e0, e1, e2, e3};      // one entry: whole 16-byte chunks
      if (xf >= 0) store_chunks<sizeof(ent)>(((SweepRec<T>*)d.frec)[xf / PF_E].co[xf % PF_E], ent);
      if (xb >= 0) store_chunks<sizeof(ent)>(((SweepRec<T>*)d.brec)[xb / PF_E].co[xb % PF_E], ent);
    }
    // the ghost state of a wall or symmetry face in the form the backward sweep's flux
    // increment takes it (its only ghost entries), so the sweep itself does no FP64 work
    const int bc = d.fbc[f];
    if (j < 0 && (bc == 2 || bc == 3 || bc == 5)) {
      const double gr = d.G[f], gmx = d.G[nf + f], gmy = d.G[2 * nf + f], gE = d.G[3 * nf + f];
      const double gu = gmx / gr, gv = gmy / gr;
      const double gp = (GAMMA - 1.0) * (gE - 0.5 * (gmx * gu + gmy * gv));
      T* g = (T*)d.gprim;
      g[f] = (T)gr; g[nf + f] = (T)gmx; g[2 * nf + f] = (T)gmy;
      g[3 * nf + f] = (T)gu; g[4 * nf + f] = (T)gv; g[5 * nf + f] = (T)(gE + gp);
    }
  }
}

// ---- one cell of the wide schedule (stencil in cell-face order) ----
// A level is one launch of a few thousand cells at most, so its time is the latency of the
// loads one cell waits for: the entries are taken WIDE_E at a time, their neighbours and
// coefficients first, then all their increments together (an entry that does not apply reads
// the cell's own). On 1470 polygons (10 levels, double-float) the forward sweep takes 66 us,
// and took 133 us with one entry after the other.
constexpr int WIDE_E = 4;

template <class T>
struct WideBatch {
  int j[WIDE_E];
  T co[WIDE_E][4], f[WIDE_E][8], w[WIDE_E][5];
};
// entries [k0, k0 + WIDE_E) of cell i, those below end; use(j): the entry needs increments
template <class T, class Use>
__device__ __forceinline__ void wide_load(WideBatch<T>& b, const Dev& d, const T* dF, const T* dWv, int i, int k0,
                                          int end, Use use) {
  const int n = d.nc_pad, nnz = d.nnz;
  const T* sc = (const T*)d.sw_st;
#pragma unroll
  for (int e = 0; e < WIDE_E; e++) {
    const int k = min(k0 + e, end - 1);
    b.j[e] = d.sw_j[k];
#pragma unroll
    for (int q = 0; q < 4; q++) b.co[e][q] = sc[q * nnz + k];
  }
#pragma unroll
  for (int e = 0; e < WIDE_E; e++) {
    const int j = use(b.j[e]) ? b.j[e] : i;
#pragma unroll
    for (int q = 0; q < 8; q++) b.f[e][q] = dF[q * n + j];
    load_incs<T>(b.w[e], dWv, n, j);
  }
}

// the cell's increments and flux increments to global memory
template <class T>
__device__ __forceinline__ void wide_finish(const Dev& d, int i, const T* dw, T* dWv) {
  const int n = d.nc_pad;
  const T* c = (const T*)d.sw_cell;
  T* dF = (T*)d.dF;
  T o[8];
  delta_flux<T>((T)d.W[i], (T)d.W[n + i], (T)d.W[2 * n + i], c[2 * n + i], c[3 * n + i], c[4 * n + i],
                dw[0], dw[1], dw[2], dw[3], o);
  store_incs<T>(dWv, n, i, dw, dw[4]);
#pragma unroll
  for (int q = 0; q < 8; q++) dF[q * n + i] = o[q];
}

template <class T>
__device__ __forceinline__ void fwd_cell(const Dev& d, int i, bool sa_on) {
  const int n = d.nc_pad;
  T* dWs = (T*)d.dWs;
  const T* dF = (const T*)d.dF;
  const T* c = (const T*)d.sw_cell;
  T acc[5];
#pragma unroll
  for (int v = 0; v < 5; v++) acc[v] = (T)d.M[v * n + i];
  const int end = d.cf_ptr[i + 1];
  for (int k0 = d.cf_ptr[i]; k0 < end; k0 += WIDE_E) {
    auto use = [&](int j) { return j >= 0 && j < i; };   // ghost increments are zero forward
    WideBatch<T> b;
    wide_load<T>(b, d, dF, dWs, i, k0, end, use);
#pragma unroll
    for (int e = 0; e < WIDE_E; e++)
      if (k0 + e < end && use(b.j[e]))
        fwd_acc<T>(acc, b.co[e][0], b.co[e][1], b.co[e][2], b.co[e][3], b.f[e], b.w[e], sa_on);
  }
  T dw[5];
#pragma unroll
  for (int v = 0; v < 4; v++) dw[v] = inc_fwd<T>(acc[v], c[i]);
  dw[4] = sa_on ? inc_fwd<T>(acc[4], c[n + i]) : (T)0;
  wide_finish<T>(d, i, dw, dWs);
}

__device__ __forceinline__ void flush_eq40(const Dev& d, int s, double eq40, int bad);

template <class T>
__device__ __forceinline__ T mn_x(T a, T fx, T b, T fy) { return fma_x(a, fx, mul_x(b, fy)); }

// The terms of a wall / symmetry ghost (face fc) in a cell's backward sum: the boundary map
// of the cell's own forward increment ws and the flux increment about the ghost state give
// t[0..3] (entry_sum of the four mean-flow components); returns the ghost's SA increment.
template <class T>
__device__ __forceinline__ T ghost_terms(const Dev& d, int fc, const T* ws, T sx, T sy, T sl, T* t) {
  const int nf = d.nf;
  T f[8], w[5];
  w[0] = ws[0]; w[3] = ws[3];
  if (d.fbc[fc] == 3 || d.fbc[fc] == 5) { w[1] = -ws[1]; w[2] = -ws[2]; w[4] = -ws[4]; }
  else {
    const T fx = (T)d.fnx[fc], fy = (T)d.fny[fc];
    const T mn = mn_x(ws[1], fx, ws[2], fy);
    const T mn2 = add_x(mn, mn);                                      // 2 (dm . n), exact
    w[1] = fma_x(-mn2, fx, ws[1]); w[2] = fma_x(-mn2, fy, ws[2]); w[4] = ws[4];
  }
  const T* g = (const T*)d.gprim;   // ghost r, mx, my, u, v, H of this face (pre-pass)
  delta_flux<T>(g[fc], g[nf + fc], g[2 * nf + fc], g[3 * nf + fc], g[4 * nf + fc], g[5 * nf + fc],
                w[0], w[1], w[2], w[3], f);
#pragma unroll
  for (int v = 0; v < 4; v++) t[v] = entry_sum<T>(sx, sy, sl, f[2 * v], f[2 * v + 1], w[v]);
  return w[4];
}

template <class T>
__device__ __forceinline__ void bwd_cell(const Dev& d, int i, bool sa_on) {
  const int n = d.nc_pad;
  const T* dWs = (const T*)d.dWs;
  T* dWo = (T*)d.dW;
  const T* dF = (const T*)d.dF;
  const T* c = (const T*)d.sw_cell;
  T ws[5];
  load_incs<T>(ws, dWs, n, i);
  T acc[5] = {0, 0, 0, 0, 0};
  const int end = d.cf_ptr[i + 1];
  for (int k0 = d.cf_ptr[i]; k0 < end; k0 += WIDE_E) {
    auto use = [&](int j) { return j > i; };
    WideBatch<T> b;
    wide_load<T>(b, d, dF, dWo, i, k0, end, use);
#pragma unroll
    for (int e = 0; e < WIDE_E; e++) {
      if (k0 + e >= end) continue;
      if (use(b.j[e])) {
        bwd_acc<T>(acc, b.co[e][0], b.co[e][1], b.co[e][2], b.co[e][3], b.f[e], b.w[e], sa_on);
      } else if (b.j[e] < 0) {
        const int f = d.cf_face[k0 + e];
        if (d.fbc[f] == 1 || d.fbc[f] == 4) continue;  // free-stream and outflow increments are zero
        T t[4];
        const T w4 = ghost_terms<T>(d, f, ws, b.co[e][0], b.co[e][1], b.co[e][2], t);
#pragma unroll
        for (int v = 0; v < 4; v++) ghost_add<T>(acc[v], t[v]);
        if (sa_on) bwd_sa<T>(acc[4], b.co[e][3], w4);
      }
    }
  }
  T dw[5];
#pragma unroll
  for (int v = 0; v < 4; v++) dw[v] = inc_bwd<T>(ws[v], acc[v], c[i]);
  dw[4] = sa_on ? inc_bwd<T>(ws[4], acc[4], c[n + i]) : (T)0;
  wide_finish<T>(d, i, dw, dWo);
}

// ---- state update W += dW (FP64), nu_tilde floor, Eq. 40 ratio, divergence check ----
// Runs after the backward sweep over all cells at once: it is off the sweeps' dependency
// chain, and its FP64 square roots and division are spread over the whole GPU.
template <class T>
__global__ void __launch_bounds__(CELL_BLOCK) k_update(Dev d) {
  chain_wait();
  const int blk = d.g_blk0 + blockIdx.x;
  const int i = blk * CELL_BLOCK + threadIdx.x;
  const int s = d.cell_solve[blk * CELL_BLOCK];   // every block lies in one solve
  double eq40 = 0.0;                              // squared Eq. 40 ratio (the root once per solve)
  int bad = 0;
  // a solve whose sweep wait ran out keeps its state (the increments are incomplete)
  const bool live = (i < d.nc_pad) && d.cell_solve[i] >= 0 && d.st[d.cell_solve[i]].state == 0 &&
                    !d.tmo[d.cell_solve[i]];
  if (live) {
    const int n = d.nc_pad;
    const T* dWo = (const T*)d.dW;
    double Wi[5];
#pragma unroll
    for (int v = 0; v < 5; v++) Wi[v] = d.W[v * n + i];
    const int si = d.cell_solve[i];
    const bool expl = d.flow[si].scheme == 1;
    // explicit scheme (Eq. 15 as Eq. 16): dW = dt M / Omega, in FP64
    const double xf = expl ? __longlong_as_double((long long)d.dt_bits[si]) / d.area[i] : 0.0;
    double num = 0.0, den = 0.0;
    T dw[5] = {};
    if (!expl) load_incs<T>(dw, dWo, n, i);
#pragma unroll
    for (int v = 0; v < 4; v++) {
      const double dv = expl ? xf * d.M[v * n + i] : to_double(dw[v]);
      num += dv * dv;
      den += Wi[v] * Wi[v];
      Wi[v] += dv;
    }
    Wi[4] += expl ? (d.flow[si].sa_on ? xf * d.M[4 * n + i] : 0.0) : to_double(dw[4]);
    if (Wi[4] < 0.0) Wi[4] = 0.0;
    eq40 = num * __drcp_rn(den);
    const double p = Wi[3] - 0.5 * (Wi[1] * Wi[1] + Wi[2] * Wi[2]) * __drcp_rn(Wi[0]);   // for its sign
    if (!(Wi[0] > 0.0) || !(p > 0.0) || !isfinite(Wi[3]) || !isfinite(Wi[4])) bad = 1;
#pragma unroll
    for (int v = 0; v < 5; v++) d.W[v * n + i] = Wi[v];
  }
  flush_eq40(d, (s >= 0 && d.st[s].state == 0) ? s : -1, eq40, bad);
}

// warp maximum of the squared Eq. 40 ratio and OR of the divergence flag, one atomic each;
// positive doubles order like their bit patterns, so the per-solve maximum is exact
__device__ __forceinline__ void flush_eq40(const Dev& d, int s, double eq40, int bad) {
  // (a ratio that is not a number comes with bad; it must not pass for a large one)
  const unsigned long long x = eq40 > 0.0 ? (unsigned long long)__double_as_longlong(eq40) : 0ull;
  const unsigned hi = (unsigned)(x >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? (unsigned)x : 0u);
  bad = __any_sync(0xffffffffu, bad);
  if ((threadIdx.x & 31) == 0 && s >= 0) {
    const unsigned long long a = ((unsigned long long)mh << 32) | ml;
    if (a > *(volatile unsigned long long*)(d.eq40_bits + s)) atomicMax(d.eq40_bits + s, a);
    if (bad) atomicOr(d.bad + s, 1);
  }
}

// ---- narrow schedule: one block (or a cluster) per solve, shared-memory ring ----
//
// What bounds it: the latency of one cell's chain (neighbours' increments -> own increments
// -> own flux increments) times the number of levels. A level holds 20-200 cells and a warp
// with nobody beside it issues a dependent instruction every five cycles or so, so what
// counts is the number of instructions of the busiest warp between two level barriers:
//  - two threads per cell (lanes 2q, 2q + 1): lane 0 accumulates mass and x momentum and
//    forms the x flux increments, lane 1 y momentum, energy and the y flux increments (both
//    the SA row); they exchange the increments and one product by shuffles. Half the
//    instructions per thread and twice the schedulers in use (FP64 issues one warp
//    instruction per 64 cycles on a scheduler whatever its active lanes).
//  - the cell warps do nothing else: a warp of its own issues the bulk copies that bring the
//    records into shared memory (cp.async.bulk, chunks of 32 or 64 positions on an mbarrier each),
//    other warps take the finished increments from the ring to global memory one level
//    later, and one fetches the increments that left the ring ahead of their level.
//  - two sets of cell warps take the levels in turn: while one computes a level, the other
//    has the next level's records in registers and its ring addresses formed, and waits.
//    (One set that read its next records before the level barrier: FP32 195 + 209 us below,
//    double-float 360 + 385.) With six warps a set the registers suffice without spills.
//  - flux increments go to global memory only for the cells that a later cell reads there.
//  - the ring holds the 13 values of a cell as 12 + 1: x fluxes, y fluxes and increments of
//    the four mean-flow components (a lane reads its two of each with one vector load; 12
//    values are 48 or 96 bytes, which puts consecutive cells on distinct banks), SA apart.
// Forward + backward on the 20,480-cell hybrid plate (351 levels each way), against one
// thread per cell that read its record inside the level and stored its results itself:
// FP32 401 + 418 -> 169 + 149 us, double-float 592 + 719 -> 340 + 319, FP64 1192 + 1417 ->
// 740 + 685 (FP64: 37 warp instructions a level at 64-76 cycles are most of it). The
// 60,160-cell O-mesh (605 levels; every level has a seam cell whose neighbour left the ring
// 300 levels ago) FP32 946 + 895 -> 439 + 450 us; 5,040 cells of plate 160 + 188 -> 59 + 59.
// Every level counts by itself: where a deep solve has some levels wider than the record buffers
// (250,368-cell O-mesh, 32 of 1,265 above 352 cells), double-float 5.85 + 6.31 -> 5.03 + 5.37 ms,
// FP64 9.68 + 11.34 -> 8.44 + 8.74; staging none of such a solve's levels, 7.49 + 5.50 and 11.59 + 8.88.
// A level ends when the store warps have stored the level before: one 16-byte store instead of
// two of 8, and targets of two rounds read ahead instead of three, took FP32 forward from 184
// and 492 to 176 and 457 us; a cell's increments side by side in dW (INC_STRIDE) took backward
// from 155 and 516 to 151 and 450. Store warps that take two levels at a time, in the barrier of every other
// level, gained 2 us and lost 15; outside the level barrier, polling a counter, they were no
// faster (184 + 170, 65 + 65 us; the polls load the shared memory the cells wait for).

// With a cluster of C blocks per solve (C > 1), position q of the solve belongs to block
// q % C and its increments sit in that block's ring, read through distributed shared
// memory; the ring is a multiple of C, so the slot q % ring names the owner too.
template <class T, int C>
__device__ __forceinline__ const T* ring_of(const T* ring, int slot) {
  if constexpr (C == 1) {
    return ring;
  } else {
    cg::cluster_group cl = cg::this_cluster();
    const unsigned owner = (unsigned)(slot & (C - 1));
    return owner == cl.block_rank() ? ring : cl.map_shared_rank(ring, owner);
  }
}

static_assert(sizeof(SweepRec<df64>) == sizeof(SweepRec<double>), "double-float records");

// two or four consecutive values by vector loads / stores
template <class T>
struct alignas(2 * sizeof(T)) Pair { T a, b; };

// mbarrier and bulk copy
__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned bar, unsigned bytes) {   // the producer's arrival
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(unsigned bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// wait for a phase of the barrier, at most limit tries; false when it ran out
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, int limit) {
  for (int it = 0; it < limit; it++)
    if (mbar_try(bar, parity)) return true;
  return false;
}
__device__ __forceinline__ void bulk_g2s(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

// shared memory: ring, side slots and the zero slot [12] | their SA increments | NREC records
// | LVL_SMEM level offsets | an mbarrier per chunk | progress: levels finished | landed:
// records in shared memory. Records that find no place in a level wider than NREC - CHUNK
// positions, and all of a cluster's, are read from global memory. CHUNK: an FP32 level takes
// 0.5 us, so the copies come in fewer, larger pieces.
constexpr int LVL_SMEM = 2048;
// (three store warps in FP32: 1% slower, their shared-memory reads stand in the cells' way)
constexpr int STORE_WARPS = 2;
template <class T>
struct Smem {
  static constexpr int SLOTS = ring_slots((int)sizeof(T)), ZERO = zero_slot((int)sizeof(T)), ALL = ZERO + 1;
  static constexpr int CHUNK = sizeof(T) == 4 ? 64 : 32;
  static constexpr int NREC = sizeof(T) == 4 ? 640 : 384;
  static constexpr int NCHUNK = NREC / CHUNK;
  static constexpr size_t ring4 = (size_t)12 * ALL * sizeof(T);
  static constexpr size_t rec = (ring4 + (size_t)ALL * sizeof(T) + 15) / 16 * 16;
  static constexpr size_t lvl = rec + (size_t)NREC * sizeof(SweepRec<T>);
  static constexpr size_t bar = lvl + (size_t)LVL_SMEM * sizeof(int);
  static constexpr size_t flag = bar + 8 * (size_t)NCHUNK;
  static constexpr size_t total = flag + 16;
  static_assert(NCHUNK <= 32, "a phase bit per buffer");
  static_assert(total <= 232448, "shared memory of one block");
};

// what a thread holds of its cell's record: the sum's start (a0, a1, a4: forward the
// residual), backward the forward increments (m0, m1, m4), constants, two entries
template <class T>
struct LaneRec {
  int i, kind, pb, spill;
  int slot[PF_E];
  T a0, a1, a4, m0, m1, m4, r, mx, my, c0, c1, u, v, H;
  T co[2][4];       // quads and triangles mostly have no more
};

template <class T>
__device__ __forceinline__ void load_co(T* o, const T* co) {
#pragma unroll
  for (int k = 0; k < (int)(4 * sizeof(T) / 16); k++)
    reinterpret_cast<uint4*>(o)[k] = reinterpret_cast<const uint4*>(co)[k];
}

template <class T, bool FWD>
__device__ __forceinline__ void load_rec(LaneRec<T>& o, const SweepRec<T>* dy, int lane) {
  const int4 b = *reinterpret_cast<const int4*>(dy->st.slot), a = *reinterpret_cast<const int4*>(&dy->st);
  o.slot[0] = b.x; o.slot[1] = b.y; o.slot[2] = b.z;
  o.i = a.x; o.kind = a.y; o.pb = a.z; o.spill = a.w;
  const Pair<T> m = *reinterpret_cast<const Pair<T>*>(&dy->m[2 * lane]);
  constexpr int N = sizeof(T) == 4 ? 12 : 10;           // m[4], w[3], c[5], pad0[0]: whole chunks
  alignas(16) T q[N];
#pragma unroll
  for (int k = 0; k < (int)(N * sizeof(T) / 16); k++)
    reinterpret_cast<uint4*>(q)[k] = reinterpret_cast<const uint4*>(&dy->m[4])[k];
  if constexpr (FWD) {
    o.a0 = m.a; o.a1 = m.b; o.a4 = q[0];
  } else {
    const Pair<T> s = *reinterpret_cast<const Pair<T>*>(&dy->start[2 * lane]);
    o.a0 = s.a; o.a1 = s.b; o.a4 = q[9];
    o.m0 = m.a; o.m1 = m.b; o.m4 = q[0];
  }
  o.r = q[1]; o.mx = q[2]; o.my = q[3];
  o.c0 = q[4]; o.c1 = q[5]; o.u = q[6]; o.v = q[7]; o.H = q[8];
#pragma unroll
  for (int e = 0; e < 2; e++) load_co<T>(o.co[e], dy->co[e]);
}

// one stencil entry as a lane needs it: x and y flux increments and increments of its two
// components, and the SA increment
template <class T>
struct LaneNb { T x0, x1, y0, y1, w0, w1, w4; };

template <class T>
__device__ __forceinline__ void ring_read_at(LaneNb<T>& o, const T* b, const T* b4) {
  const Pair<T> x = *reinterpret_cast<const Pair<T>*>(b), y = *reinterpret_cast<const Pair<T>*>(b + 4),
                w = *reinterpret_cast<const Pair<T>*>(b + 8);
  o.x0 = x.a; o.x1 = x.b; o.y0 = y.a; o.y1 = y.b; o.w0 = w.a; o.w1 = w.b;
  o.w4 = *b4;
}
template <class T, int C>
__device__ __forceinline__ void ring_read(LaneNb<T>& o, const T* ring, const T* ring4, int slot, int lane) {
  ring_read_at<T>(o, ring_of<T, C>(ring, slot) + slot * 12 + 2 * lane, ring_of<T, C>(ring4, slot) + slot);
}

template <class T>
__device__ __forceinline__ void global_read(LaneNb<T>& o, const Dev& d, const T* dWv, int j, int lane) {
  const int n = d.nc_pad;
  const T* dF = (const T*)d.dF;
  o.x0 = dF[(4 * lane) * n + j]; o.y0 = dF[(4 * lane + 1) * n + j];
  o.x1 = dF[(4 * lane + 2) * n + j]; o.y1 = dF[(4 * lane + 3) * n + j];
  o.w0 = dWv[inc_at<T>(n, 2 * lane, j)]; o.w1 = dWv[inc_at<T>(n, 2 * lane + 1, j)]; o.w4 = dWv[inc_at<T>(n, 4, j)];
}

// a lane's results for one cell: its increments (w4: the SA row, both lanes) and the four
// mean-flow components of its flux direction
template <class T>
struct LaneOut { T w0, w1, w4, f[4]; };

template <class T>
__device__ __forceinline__ T shfl_pair(T x) { return __shfl_xor_sync(0xffffffffu, x, 1); }
template <>
__device__ __forceinline__ df64 shfl_pair<df64>(df64 x) {
  return df64(__shfl_xor_sync(0xffffffffu, x.hi, 1), __shfl_xor_sync(0xffffffffu, x.lo, 1));
}

// The increments and flux increments of one cell from its accumulators; the same operations
// as delta_flux, split over the two lanes. Called by whole warps.
template <class T, bool FWD>
__device__ __forceinline__ LaneOut<T> lane_finish(const LaneRec<T>& rc, T acc0, T acc1, T acc4, int lane, bool sa_on) {
  LaneOut<T> o;
  if constexpr (FWD) {
    o.w0 = inc_fwd<T>(acc0, rc.c0); o.w1 = inc_fwd<T>(acc1, rc.c0);
    o.w4 = sa_on ? inc_fwd<T>(acc4, rc.c1) : (T)0;
  } else {
    o.w0 = inc_bwd<T>(rc.m0, acc0, rc.c0); o.w1 = inc_bwd<T>(rc.m1, acc1, rc.c0);
    o.w4 = sa_on ? inc_bwd<T>(rc.m4, acc4, rc.c1) : (T)0;
  }
  const T p0 = shfl_pair(o.w0), p1 = shfl_pair(o.w1);
  const T dr = lane ? p0 : o.w0, dE = lane ? o.w1 : p1;
  const T dm = lane ? o.w0 : o.w1, dmo = lane ? p1 : p0;         // momentum along / across the lane's direction
  const T vel = lane ? rc.v : rc.u, mom = lane ? rc.my : rc.mx, mo = lane ? rc.mx : rc.my;
  const T inv1 = rcp_x(add_x(rc.r, dr));
  const T dv = mul_x(fma_x(-vel, dr, dm), inv1);
  const T v1 = add_x(vel, dv);
  const T q = fma_x(dm, v1, mul_x(mom, dv));
  const T dp = mul_x((T)(GAMMA - 1.0), fma_x((T)(-0.5), add_x(q, shfl_pair(q)), dE));
  const T dH = add_x(dE, dp);
  const T own = add_x(q, dp), cross = fma_x(dmo, v1, mul_x(mo, dv));
  o.f[0] = dm;
  o.f[1] = lane ? cross : own;
  o.f[2] = lane ? own : cross;
  o.f[3] = fma_x(dH, v1, mul_x(rc.H, dv));
  return o;
}

template <class T>
__device__ __forceinline__ void ring_put(T* b, T* b4, const LaneOut<T>& o, int lane) {
  Pair<T>* f = reinterpret_cast<Pair<T>*>(b + 4 * lane);
  f[0] = Pair<T>{o.f[0], o.f[1]};
  f[1] = Pair<T>{o.f[2], o.f[3]};
  *reinterpret_cast<Pair<T>*>(b + 8 + 2 * lane) = Pair<T>{o.w0, o.w1};
  if (lane) *b4 = o.w4;
}

// increments to global memory: the forward one into the cell's backward record (at = its
// position), the backward one into dW (at = the cell)
template <class T, bool FWD>
__device__ __forceinline__ void store_inc(const Dev& d, int at, const T* w, T w4) {
  if constexpr (FWD) {
    T* m = ((SweepRec<T>*)d.brec + at)->m;
    if constexpr (sizeof(T) == 4) {   // one store (double-float and FP64 were 1% slower with two wide ones)
      alignas(16) const T v[4] = {w[0], w[1], w[2], w[3]};
      store_chunks<sizeof(v)>(m, v);
    } else {
      reinterpret_cast<Pair<T>*>(m)[0] = Pair<T>{w[0], w[1]};
      reinterpret_cast<Pair<T>*>(m)[1] = Pair<T>{w[2], w[3]};
    }
    m[4] = w4;
  } else {
    store_incs<T>((T*)d.dW, d.nc_pad, at, w, w4);
  }
}

// the increments of a cell that a later one reads from global memory (before the barrier)
template <class T, bool FWD>
__device__ __noinline__ void store_spill(const Dev& d, int i, LaneOut<T> o, int lane) {
  const int n = d.nc_pad;
  T* dWv = (T*)(FWD ? d.dWs : d.dW);
  T* dF = (T*)d.dF;
  dWv[inc_at<T>(n, 2 * lane, i)] = o.w0;
  dWv[inc_at<T>(n, 2 * lane + 1, i)] = o.w1;
  if (lane) dWv[inc_at<T>(n, 4, i)] = o.w4;
  for (int v = 0; v < 4; v++) dF[(2 * v + lane) * n + i] = o.f[v];
}

// the increments of a cell in a level that the store warps do not take (SPILL_OWN; at as in store_inc)
template <class T, bool FWD>
__device__ __noinline__ void store_own(const Dev& d, int at, LaneOut<T> o, int lane) {
  const int n = d.nc_pad;
  T* m = FWD ? ((SweepRec<T>*)d.brec + at)->m : (T*)d.dW;
  m[FWD ? 2 * lane : inc_at<T>(n, 2 * lane, at)] = o.w0;
  m[FWD ? 2 * lane + 1 : inc_at<T>(n, 2 * lane + 1, at)] = o.w1;
  if (lane) m[FWD ? 4 : inc_at<T>(n, 4, at)] = o.w4;
}

// the accumulators of a cell with more entries than a record holds (p: its position)
template <class T, bool FWD, int C>
__device__ __noinline__ void csr_sum(const Dev& d, const T* ring, const T* ring4, int slots, int p, int lane, bool sa_on, T* acc) {
  const T* sc = (const T*)(FWD ? d.sc_f : d.sc_b);
  const int ne = FWD ? d.nfs : d.nbs;
  const int* ptr = FWD ? d.fs_ptr : d.bs_ptr;
  const int* sj = FWD ? d.fs_j : d.bs_j;
  const int* ss = FWD ? d.fs_slot : d.bs_slot;
  for (int k = ptr[p]; k < ptr[p + 1]; k++) {
    const T sx = sc[k], sy = sc[ne + k], sl = sc[2 * ne + k], sa = sc[3 * ne + k];
    if (!FWD && ss[k] == SLOT_GHOST) {
      const T* ws = ((const SweepRec<T>*)d.brec)[p].m;
      T t[4];
      const T w4 = ghost_terms<T>(d, -1 - sj[k], ws, sx, sy, sl, t);
      ghost_add<T>(acc[0], lane ? t[2] : t[0]);
      ghost_add<T>(acc[1], lane ? t[3] : t[1]);
      if (sa_on) bwd_sa<T>(acc[2], sa, w4);
      continue;
    }
    LaneNb<T> b;
    if ((unsigned)ss[k] < (unsigned)slots) ring_read<T, C>(b, ring, ring4, ss[k], lane);
    else global_read<T>(b, d, (const T*)(FWD ? d.dWs : d.dW), sj[k], lane);
    if constexpr (FWD) {
      fwd_comp<T>(acc[0], sx, sy, sl, b.x0, b.y0, b.w0);
      fwd_comp<T>(acc[1], sx, sy, sl, b.x1, b.y1, b.w1);
      if (sa_on) fwd_sa<T>(acc[2], sa, b.w4);
    } else {
      bwd_comp<T>(acc[0], sx, sy, sl, b.x0, b.y0, b.w0);
      bwd_comp<T>(acc[1], sx, sy, sl, b.x1, b.y1, b.w1);
      if (sa_on) bwd_sa<T>(acc[2], sa, b.w4);
    }
  }
}

// one interior entry applied to the accumulators
template <class T, bool FWD>
__device__ __forceinline__ void apply_entry(T& a0, T& a1, T& a4, const T* co, const LaneNb<T>& b, bool sa_on) {
  if constexpr (FWD) {
    fwd_comp<T>(a0, co[0], co[1], co[2], b.x0, b.y0, b.w0);
    fwd_comp<T>(a1, co[0], co[1], co[2], b.x1, b.y1, b.w1);
    if (sa_on) fwd_sa<T>(a4, co[3], b.w4);
  } else {
    bwd_comp<T>(a0, co[0], co[1], co[2], b.x0, b.y0, b.w0);
    bwd_comp<T>(a1, co[0], co[1], co[2], b.x1, b.y1, b.w1);
    if (sa_on) bwd_sa<T>(a4, co[3], b.w4);
  }
}

// a ghost entry behind an interior one (backward): ready terms in the entry's coefficients,
// the signed SA coefficient in the face's first ghost value
template <class T>
__device__ __forceinline__ void apply_ghost(const Dev& d, T& a0, T& a1, T& a4, const T* co, int j, T m4, int lane,
                                            bool sa_on) {
  ghost_add<T>(a0, lane ? co[2] : co[0]);
  ghost_add<T>(a1, lane ? co[3] : co[1]);
  if (sa_on) bwd_sa<T>(a4, ((const T*)d.gprim)[-1 - j], m4);
}

// Where a cell's ring reads and writes go, known before its level begins
struct RingAt {
  int nb[2], nb4[2], put, put4;
};
template <class T>
__device__ __forceinline__ RingAt ring_at(const LaneRec<T>& rc, int q, int lane) {
  RingAt a;
  const int slot = q & (Smem<T>::SLOTS - 1);
#pragma unroll
  for (int e = 0; e < 2; e++) {
    a.nb4[e] = max(rc.slot[e], 0);
    a.nb[e] = a.nb4[e] * 12 + 2 * lane;
    asm volatile("" : "+r"(a.nb[e]), "+r"(a.nb4[e]));   // here, not after the level barrier
  }
  a.put4 = slot;
  a.put = slot * 12;
  asm volatile("" : "+r"(a.put), "+r"(a.put4));
  return a;
}

// The increments of the cell at position p (its record in rc). rare: the kinds that take the
// general path (with the side slots' in a cluster). co2(): the third entry's
// coefficients in memory. Called by whole warps; a thread without a cell of its own (valid =
// false) works on a copy of another's and stores nothing.
template <class T, bool FWD, int C, class Co2>
__device__ __forceinline__ LaneOut<T> lane_cell(const Dev& d, T* ring, T* ring4, int rare, const LaneRec<T>& rc,
                                                const RingAt& at, int p, int lane, bool valid, bool sa_on, Co2 co2) {
  T acc0 = rc.a0, acc1 = rc.a1, acc4 = rc.a4;
  LaneNb<T> nb[2];
#pragma unroll
  for (int e = 0; e < 2; e++)
    ring_read_at<T>(nb[e], ring_of<T, C>(ring, at.nb4[e]) + at.nb[e], ring_of<T, C>(ring4, at.nb4[e]) + at.nb4[e]);
  if (!(rc.kind & rare)) {
#pragma unroll
    for (int e = 0; e < 2; e++) apply_entry<T, FWD>(acc0, acc1, acc4, rc.co[e], nb[e], sa_on);
    if (rc.kind & KIND_THIRD) {
      alignas(16) T c[4];
      load_co<T>(c, co2());
      ring_read<T, C>(nb[0], ring, ring4, rc.slot[2], lane);
      apply_entry<T, FWD>(acc0, acc1, acc4, c, nb[0], sa_on);
    }
  } else if (!(rc.kind & KIND_CSR)) {
    const SweepRec<T>* recs = (const SweepRec<T>*)(FWD ? d.frec : d.brec);
    const int* js = (FWD ? d.fj : d.bj)[p].j;
    const int slots = rare & KIND_SIDE ? Smem<T>::SLOTS : Smem<T>::ALL;
#pragma unroll 1
    for (int e = 0; e < (rc.kind & KIND_COUNT); e++) {
      const int sl = e == 0 ? rc.slot[0] : e == 1 ? rc.slot[1] : rc.slot[2];
      alignas(16) T c[4];
      load_co<T>(c, recs[p].co[e]);
      if (!FWD && sl == SLOT_GHOST) {
        apply_ghost<T>(d, acc0, acc1, acc4, c, js[e], rc.m4, lane, sa_on);
        continue;
      }
      LaneNb<T> b;
      if ((unsigned)sl < (unsigned)slots) ring_read<T, C>(b, ring, ring4, sl, lane);
      else global_read<T>(b, d, (const T*)(FWD ? d.dWs : d.dW), js[e], lane);
      apply_entry<T, FWD>(acc0, acc1, acc4, c, b, sa_on);
    }
  } else {
    T acc[3] = {FWD ? acc0 : (T)0, FWD ? acc1 : (T)0, FWD ? acc4 : (T)0};
    csr_sum<T, FWD, C>(d, ring, ring4, rare & KIND_SIDE ? Smem<T>::SLOTS : Smem<T>::ALL, p, lane, sa_on, acc);
    acc0 = acc[0]; acc1 = acc[1]; acc4 = acc[2];
  }
  __syncwarp();
  const LaneOut<T> o = lane_finish<T, FWD>(rc, acc0, acc1, acc4, lane, sa_on);
  if (valid) {
    ring_put<T>(ring + at.put, ring4 + at.put4, o, lane);
    if (rc.spill) {
      if (C == 1 && (rc.spill & SPILL_OWN)) store_own<T, FWD>(d, FWD ? rc.pb : rc.i, o, lane);
      if (rc.spill & SPILL_READ) store_spill<T, FWD>(d, rc.i, o, lane);
    }
  }
  return o;
}

// the first position at or after b that belongs to cluster block r (positions q are dealt
// round the C blocks: q % C == r)
template <int C>
__device__ __forceinline__ int first_own(int b, int r) {
  return b + ((r - b) & (C - 1));
}

// The forward sweep's last step: what the wall and symmetry ghosts add to the backward sums
// (they need the cells' own forward increments only). Ghosts that come first in a cell's
// order make the sum's start, in the same additions; later ones leave their terms in their
// entries.
template <class T>
__device__ __forceinline__ void ghost_pass(const Dev& d, int s, int first, int step, bool sa_on) {
  const T* sc = (const T*)d.sc_b;
  const int g1 = d.gent_ptr[s + 1], nbs = d.nbs;
  for (int g = d.gent_ptr[s] + first; g < g1; g += step) {
    const int p = d.gent_pos[g];
    SweepRec<T>* rec = (SweepRec<T>*)d.brec + p;
    T ws[5], t[4], a[4] = {(T)0, (T)0, (T)0, (T)0}, a4 = (T)0;
#pragma unroll
    for (int v = 0; v < 5; v++) ws[v] = rec->m[v];
    int lead = -1;                                     // entries before the first interior one
    for (int k = d.bs_ptr[p]; k < d.bs_ptr[p + 1]; k++) {
      if (d.bs_slot[k] != SLOT_GHOST) {
        if (lead < 0) lead = k - d.bs_ptr[p];
        continue;
      }
      const int f = -1 - d.bs_j[k];
      const T sa = sc[3 * nbs + k];
      const T w4 = ghost_terms<T>(d, f, ws, sc[k], sc[nbs + k], sc[2 * nbs + k], t);
      if (lead < 0) {
#pragma unroll
        for (int v = 0; v < 4; v++) ghost_add<T>(a[v], t[v]);
        if (sa_on) bwd_sa<T>(a4, sa, w4);
      } else {
        T* co = rec->co[k - d.bs_ptr[p] - lead];
#pragma unroll
        for (int v = 0; v < 4; v++) co[v] = t[v];
        ((T*)d.gprim)[f] = d.fbc[f] == 2 ? sa : -sa;   // the face's ghost values have been used
      }
    }
#pragma unroll
    for (int v = 0; v < 4; v++) rec->start[v] = a[v];
    rec->pad0[0] = a4;
  }
}

// Level barriers (named, 1 and 2 by the level's parity): the warps that worked on a level
// arrive, the others wait.
__device__ __forceinline__ void bar_wait(int id, int threads) {
  asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;\n" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.cta.shared.s32 %0, [%1];\n" : "=r"(v) : "r"((unsigned)__cvta_generic_to_shared(p)) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
  asm volatile("st.release.cta.shared.s32 [%0], %1;\n" ::"r"((unsigned)__cvta_generic_to_shared(p)), "r"(v) : "memory");
}

// The sweep of one solve. Positions q are counted from the solve's first; level k is
// [lv(k), lv(k + 1)). With one block per solve the warps have roles:
//  - cell warps: two threads per cell of a level; SETS sets of them take the levels in turn. A
//    set reads its next records (from shared memory as far as they have landed, the others
//    from global memory) before it waits for the level before, so with two sets nothing but
//    the ring reads, the arithmetic and the ring stores lies between two levels;
//  - store warps: the increments of level k to global memory during level k + 1, if the two
//    levels fit the ring together (their slots are then not reused before level k + 2); the
//    cell warps store wider levels themselves;
//  - the side warp fetches increments that left the ring: it reads them during level k for
//    level k + 2 and puts them into the side slots during level k + 1;
//  - the copy warp: a chunk's buffer is free once all its positions lie in finished levels;
//    it issues chunks as buffers become free and counts the records that have landed (chunks of
//    a level wider than the buffers that it has finished without are passed over). It
//    runs beside the level barriers, and nobody waits for it. A chunk that has not landed
//    after wait_limit tries marks the solve IGKS_TIMEOUT (the update leaves its state
//    untouched); the warp then waits for the other copies in flight and ends.
template <class T, bool FWD, int C, int SETS>
__device__ __forceinline__ void sweep_narrow(const Dev& d) {
  using S = Smem<T>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* ring = (T*)smem_raw;
  T* ring4 = (T*)(smem_raw + S::ring4);
  const SweepRec<T>* srec = (const SweepRec<T>*)(smem_raw + S::rec);
  int* slv = (int*)(smem_raw + S::lvl);
  const unsigned bar0 = (unsigned)__cvta_generic_to_shared(smem_raw + S::bar);
  int* progress = (int*)(smem_raw + S::flag);
  int* landed_p = progress + 1;
  const int s = d.g_solve0 + blockIdx.x / C, r = blockIdx.x % C;   // one cluster of C blocks per solve
  if (d.st[s].state != 0 || d.flow[s].scheme == 1) return;         // uniform over the cluster
  if (!FWD && d.tmo[s]) return;                                    // the forward sweep of this solve gave up
  if (d.n_broad && (d.broad[s] != 0) != (C > 1)) return;           // the other launch sweeps it
  // (without SA its coefficients and 1/a_ii are zero and so are its increments: on the FP32
  // pipes the row is computed all the same, which costs less than the branches)
  const bool sa_on = std::is_same<T, double>::value ? d.flow[s].sa_on != 0 : true;
  const int* glv = FWD ? d.fwd_lvl : d.bwd_lvl;
  const int* lsp = FWD ? d.lvl_solve_ptr : d.blvl_solve_ptr;
  const int l0 = lsp[s], nl = lsp[s + 1] - 1 - l0;
  if (nl <= 0) return;
  glv += l0;
  const int pbase = glv[0], np = glv[nl] - pbase;
  const SweepRec<T>* grec = (const SweepRec<T>*)(FWD ? d.frec : d.brec) + pbase;
  const int tid = threadIdx.x;
  constexpr int NST = 32 * STORE_WARPS;
  const int nct = C == 1 ? (int)blockDim.x - NST - 64 : (int)blockDim.x;   // cell threads
  const int nbar = nct + NST + 32;                                 // threads of a level barrier
  const bool lvs = nl + 3 < LVL_SMEM;                              // level offsets in shared memory
  if (lvs)
    for (int k = tid; k <= nl + 2; k += blockDim.x) slv[k] = glv[min(k, nl)] - pbase;
  if (C == 1 && tid < S::NCHUNK) mbar_init(bar0 + 8 * tid, 1);
  if (C == 1) asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  if (tid == 0) { *progress = 0; *landed_p = 0; }
  if (tid < 13) (tid < 12 ? ring + 12 * S::ZERO : ring4 + S::ZERO - 12)[tid] = (T)0;
  __syncthreads();
  if constexpr (C > 1) cg::this_cluster().sync();                  // every block runs before any remote read
  auto lv = [&](int k) { return lvs ? slv[k] : glv[min(k, nl)] - pbase; };
  if (tid < nct) {
    const int set = tid / (nct / SETS), t = tid - set * (nct / SETS);
    const int lane = t & 1, w0 = (t & 31) / 2 * C, own = C * (t >> 1), step = C * (nct / SETS) / 2;
    constexpr int rare = C == 1 ? KIND_RARE : KIND_RARE | KIND_SIDE;   // (no side warp in a cluster)
    LaneRec<T> rc;
    auto fetch = [&](int q, int landed) {
      if (q < landed) load_rec<T, FWD>(rc, srec + q % S::NREC, lane);
      else load_rec<T, FWD>(rc, grec + q, lane);
    };
    for (int k = set; k < nl; k += SETS) {
      const int b = lv(k), e = lv(k + 1);
      int q = first_own<C>(b, r) + own;
      const int landed = C == 1 ? ld_acquire(landed_p) : 0;
      RingAt at;
      auto next = [&] {                  // the record of position q and its places in the ring
        fetch(min(q, e - 1), landed);
        at = ring_at<T>(rc, q, lane);
      };
      const bool act = q - w0 < e;       // a warp works if its first cell exists
      if (act) next();
      if (C == 1 && k > 0) bar_wait(2 - (k & 1), nbar);            // level k - 1 is finished
      bool global = false;               // increments stored to global memory that others may read
      if (act) do {                      // more than one round in a level wider than the set
        const bool valid = q < e;
        const int qc = min(q, e - 1);
        const LaneOut<T> o = lane_cell<T, FWD, C>(
            d, ring, ring4, rare, rc, at, pbase + qc, lane, valid, sa_on,
            [&] { return qc < landed ? srec[qc % S::NREC].co[2] : grec[qc].co[2]; });
        if constexpr (C > 1) {           // no store warps
          const T p0 = shfl_pair(o.w0), p1 = shfl_pair(o.w1);
          const T w[4] = {o.w0, o.w1, p0, p1};
          if (valid && lane == 0) store_inc<T, FWD>(d, FWD ? rc.pb : rc.i, w, o.w4);
        }
        global |= (rc.spill & SPILL_READ) != 0;
        q += step;
        if (q - w0 >= e) break;
        next();
      } while (true);
      if (C == 1 && global) __threadfence_block();
      if constexpr (C > 1) cg::this_cluster().sync();   // release/acquire over the cluster's shared and global writes
      else if (SETS > 1) bar_arrive(1 + (k & 1), nbar);
      else if (k == nl - 1) bar_wait(1 + (k & 1), nbar);
    }
    if (SETS > 1 && set != (nl - 1) % SETS) bar_wait(1 + ((nl - 1) & 1), nbar);
  } else if (tid < nct + NST) {
    const int t = tid - nct;
    auto at = [&](int q) { return FWD ? grec[q].st.pb : grec[q].st.i; };
    constexpr int ROUNDS = sizeof(T) == 4 ? 2 : 3;                 // positions whose targets are read a level ahead
    int b = 0, e = 0, en = lv(1), next[ROUNDS];
#pragma unroll
    for (int j = 0; j < ROUNDS; j++) next[j] = t + j * NST < en ? at(t + j * NST) : 0;
    for (int k = 0; k <= nl; k++) {                                // stores level k - 1
      if (t == 0) st_release(progress, k);                         // levels below k are finished
      const bool mine = en - b <= S::SLOTS;                        // (else SPILL_OWN)
      auto put = [&](int q, int x) {
        const int slot = q & (S::SLOTS - 1);
        alignas(16) T w[4];
        load_co<T>(w, ring + slot * 12 + 8);
        store_inc<T, FWD>(d, x, w, ring4[slot]);
      };
#pragma unroll
      for (int j = 0; j < ROUNDS; j++) {
        const int x = next[j];
        if (e + t + j * NST < en) next[j] = at(e + t + j * NST);
        if (mine && b + t + j * NST < e) put(b + t + j * NST, x);
      }
      if (mine)
        for (int q = b + t + ROUNDS * NST; q < e; q += NST) put(q, at(q));
      if (k == nl) break;
      bar_wait(1 + (k & 1), nbar);
      b = e; e = en; en = lv(k + 2);
    }
  } else if (tid < nct + NST + 32) {
    const int t = tid - nct - NST, n = d.nc_pad;
    static_assert(SIDE == 32, "one side slot a thread");
    const int* sp = (FWD ? d.fside_ptr : d.bside_ptr) + l0;
    const int* sj = FWD ? d.fside_j : d.bside_j;
    const T* dF = (const T*)d.dF;
    const T* dWv = (const T*)(FWD ? d.dWs : d.dW);
    // side slots, a step a level: offsets (level k + 4), cell (k + 3), increments (k + 2), slot (k + 1)
    int pa = 0, pb = 0, j = -1, jv = -1;
    T v[13];
    if (nl > 3) { pa = sp[3]; pb = sp[4]; }
    for (int k = 0; k < nl; k++) {
      if (jv >= 0) {
        const int slot = S::SLOTS + ((k + 1) & 1) * SIDE + t;
#pragma unroll
        for (int c = 0; c < 12; c++) ring[slot * 12 + c] = v[c];
        ring4[slot] = v[12];
      }
      jv = j;
      if (jv >= 0) {
#pragma unroll
        for (int c = 0; c < 4; c++) {
          v[c] = dF[2 * c * n + jv];
          v[4 + c] = dF[(2 * c + 1) * n + jv];
          v[8 + c] = dWv[inc_at<T>(n, c, jv)];
        }
        v[12] = dWv[inc_at<T>(n, 4, jv)];
      }
      j = pa + t < pb ? sj[pa + t] : -1;
      if (k + 5 <= nl) { pa = sp[k + 4]; pb = sp[k + 5]; }
      else pa = pb;
      bar_wait(1 + (k & 1), nbar);
    }
  } else if ((tid & 31) == 0) {
    constexpr int CHUNK = S::CHUNK;
    const int nchunk = (np + CHUNK - 1) / CHUNK;
    const unsigned urec = (unsigned)__cvta_generic_to_shared(smem_raw + S::rec);
    int issued = 0, landed = 0, seen = -1, idle = 0;
    unsigned phase = 0;                                            // of each buffer's mbarrier
    auto wait = [&](int q) {
      const int c = q % S::NCHUNK;
      const bool ok = mbar_wait(bar0 + 8 * c, phase >> c & 1, d.wait_limit);
      phase ^= 1u << c;
      return ok;
    };
    while (landed < nchunk && idle < d.wait_limit) {
      const int k = ld_acquire(progress);
      idle = k == seen ? idle + 1 : 0;
      if (k != seen) {
        seen = k;
        if (k >= nl) break;                                        // the sweep is over
        const int first = lv(k) / CHUNK, upto = min(first + S::NCHUNK, nchunk);
        if (landed == issued && first > issued) issued = landed = first;   // finished from global memory
        // the buffers were read by generic loads: order those before the async proxy's writes
        if (issued < upto) asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        for (; issued < upto; issued++) {
          if (FWD && d.starve_test && issued == 1) continue;
          // (a buffer's last chunk, read from global memory where it came late, may be in flight)
          if (issued - S::NCHUNK >= landed) break;
          const int c = issued % S::NCHUNK, q = issued * CHUNK, m = min(CHUNK, np - q);
          const unsigned bytes = (unsigned)(m * sizeof(SweepRec<T>));
          mbar_expect(bar0 + 8 * c, bytes);
          bulk_g2s(urec + (unsigned)(c * CHUNK * sizeof(SweepRec<T>)), grec + q, bytes, bar0 + 8 * c);
        }
      }
      if (landed < issued) {
        if (!wait(landed)) {
          d.tmo[s] = 1;
          landed++;                                                // the others in flight land below
          break;
        }
        landed++;
        st_release(landed_p, landed * CHUNK);
      } else {
        __nanosleep(40);
      }
    }
    for (; landed < issued; landed++)                              // let the copies in flight land
      if (!(FWD && d.starve_test && landed == 1)) wait(landed);
  }
  if constexpr (FWD) {
    if constexpr (C == 1) __syncthreads();                         // the increments stored above
    else cg::this_cluster().sync();
    ghost_pass<T>(d, s, r * (int)blockDim.x + tid, C * (int)blockDim.x, sa_on);
  }
}

// Cell threads of one set at most: what lets the registers of both sets fit (FP32 96 a
// thread, the 8-byte types 128). A level wider than a set takes rounds.
constexpr int SETS = 2;
template <class T>
constexpr int SET_THREADS = sizeof(T) == 4 ? 224 : 192;
template <class T>
constexpr int block_threads(int set) { return SETS * set + 32 * STORE_WARPS + 64; }
template <class T, bool FWD>
__global__ void __launch_bounds__(block_threads<T>(SET_THREADS<T>), 1)
k_sweep_block(const __grid_constant__ Dev d) { sweep_narrow<T, FWD, 1, SETS>(d); }
template <class T, bool FWD, int C>
__global__ void __launch_bounds__(NARROW_THREADS) k_sweep_cluster(const __grid_constant__ Dev d) { sweep_narrow<T, FWD, C, 1>(d); }

// ---- wide schedule: one launch per level, all solves ----
template <class T>
__global__ void k_sweep_fwd_level(Dev d, int b, int e) {
  chain_wait();
  const int k = b + blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= e) return;
  const int i = d.wfwd_cells[k];
  const int s = d.cell_solve[i];
  if (d.st[s].state != 0 || d.flow[s].scheme == 1) return;
  fwd_cell<T>(d, i, d.flow[s].sa_on);
}

template <class T>
__global__ void k_sweep_bwd_level(Dev d, int b, int e) {
  chain_wait();
  const int k = b + blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= e) return;
  const int i = d.wbwd_cells[k];
  const int s = d.cell_solve[i];
  if (d.st[s].state != 0 || d.flow[s].scheme == 1) return;
  bwd_cell<T>(d, i, d.flow[s].sa_on);
}

constexpr int WIDE_BLOCK = 128;

void launch_update(const Dev& d, int precision, cudaStream_t s) {
  if (precision == 1) launch_chained(d.chained, k_update<float>, d.g_nblk, CELL_BLOCK, 0, s, d);
  else if (precision == 2) launch_chained(d.chained, k_update<df64>, d.g_nblk, CELL_BLOCK, 0, s, d);
  else launch_chained(d.chained, k_update<double>, d.g_nblk, CELL_BLOCK, 0, s, d);
}

template <class T, bool FWD>
static void set_smem_t() {
  const int bytes = (int)Smem<T>::total;
  cudaFuncSetAttribute(k_sweep_block<T, FWD>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  cudaFuncSetAttribute(k_sweep_cluster<T, FWD, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  cudaFuncSetAttribute(k_sweep_cluster<T, FWD, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  cudaFuncSetAttribute(k_sweep_cluster<T, FWD, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

void setup_sweeps() {
  set_smem_t<double, true>();
  set_smem_t<double, false>();
  set_smem_t<float, true>();
  set_smem_t<float, false>();
  set_smem_t<df64, true>();
  set_smem_t<df64, false>();
}

// one cluster of C blocks per solve
template <class T, bool FWD, int C>
static void launch_cluster(const Dev& d, int threads, cudaStream_t s) {
  void (*k)(Dev) = k_sweep_cluster<T, FWD, C>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(d.g_nsolve * C));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = Smem<T>::total;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k, d);
}

template <class T, bool FWD>
static void launch_narrow(const Dev& d, int threads, cudaStream_t s) {
  if (d.n_broad) launch_cluster<T, FWD, BROAD_CLUSTER>(d, threads, s);
  if (d.n_broad == d.g_nsolve) return;
  switch (d.sweep_cluster) {
    case 2: launch_cluster<T, FWD, 2>(d, threads, s); break;
    case 4: launch_cluster<T, FWD, 4>(d, threads, s); break;
    case 8: launch_cluster<T, FWD, 8>(d, threads, s); break;
    default:   // one block per solve: the cells' threads, the store, side and copy warps
      k_sweep_block<T, FWD><<<d.g_nsolve, block_threads<T>(std::min(threads, SET_THREADS<T>)), Smem<T>::total, s>>>(d);
      break;
  }
}

void launch_sweep_prep(const Dev& d, int precision, cudaStream_t s) {
  if (precision == 1) launch_chained(d.chained, k_sweep_prep<float>, d.g_nblk, CELL_BLOCK, 0, s, d);
  else if (precision == 2) launch_chained(d.chained, k_sweep_prep<df64>, d.g_nblk, CELL_BLOCK, 0, s, d);
  else launch_chained(d.chained, k_sweep_prep<double>, d.g_nblk, CELL_BLOCK, 0, s, d);
}

void launch_sweep_fwd(const Dev& d, int precision, int threads, cudaStream_t s) {
  if (d.wide) {
    for (int l = 0; l < d.n_wfwd; l++) {
      const int b = d.h_wfwd_ptr[l], e = d.h_wfwd_ptr[l + 1];
      const int g = (e - b + WIDE_BLOCK - 1) / WIDE_BLOCK;
      if (precision == 1) launch_chained(d.chained, k_sweep_fwd_level<float>, g, WIDE_BLOCK, 0, s, d, b, e);
      else if (precision == 2) launch_chained(d.chained, k_sweep_fwd_level<df64>, g, WIDE_BLOCK, 0, s, d, b, e);
      else launch_chained(d.chained, k_sweep_fwd_level<double>, g, WIDE_BLOCK, 0, s, d, b, e);
    }
    return;
  }
  if (precision == 1) launch_narrow<float, true>(d, threads, s);
  else if (precision == 2) launch_narrow<df64, true>(d, threads, s);
  else launch_narrow<double, true>(d, threads, s);
}

void launch_sweep_bwd(const Dev& d, int precision, int threads, cudaStream_t s) {
  if (d.wide) {
    for (int l = 0; l < d.n_wbwd; l++) {
      const int b = d.h_wbwd_ptr[l], e = d.h_wbwd_ptr[l + 1];
      const int g = (e - b + WIDE_BLOCK - 1) / WIDE_BLOCK;
      if (precision == 1) launch_chained(d.chained, k_sweep_bwd_level<float>, g, WIDE_BLOCK, 0, s, d, b, e);
      else if (precision == 2) launch_chained(d.chained, k_sweep_bwd_level<df64>, g, WIDE_BLOCK, 0, s, d, b, e);
      else launch_chained(d.chained, k_sweep_bwd_level<double>, g, WIDE_BLOCK, 0, s, d, b, e);
    }
    return;
  }
  if (precision == 1) launch_narrow<float, false>(d, threads, s);
  else if (precision == 2) launch_narrow<df64, false>(d, threads, s);
  else launch_narrow<double, false>(d, threads, s);
}

}  // namespace igks
