// The base edge flux: shared by the base edge kernel and by the correction edge
// kernels, which add it to their own part.
#pragma once
#include "common.h"

namespace swedg {

__device__ __forceinline__ double tide_value(const Phys& ph, double t) {
  if (ph.tide_period <= 0.0) return ph.tide_amp;
  return ph.tide_amp * sin(2.0 * 3.14159265358979323846 * t / ph.tide_period + ph.tide_phase);
}

// ---------------------------------------------------------------------------
// Base edge flux.  For the P1 parts of both sides: traces at the two Gauss
// points, the LF flux (Sect. 2)
//   A_hat = 1/2 ((A(c) + A(c+)).n + lambda (c - c+)),
//   A.n = (q.n,  U (u.n) + g nx (xi^2/2 + xi h_b),  V (u.n) + g ny (...)),
// with lambda from the element means (Eq. 10, Sect. 3), stored pre-weighted
// by |E| w_g at the points in the left element's direction.
// ---------------------------------------------------------------------------
// Traces of xi, U, V and w = u.n (P1 parts) of one side at the two Gauss
// points.  Mode 1 is the constant sqrt 2 on every edge, so its trace is shared.
struct Tr2 { double xi[2], U[2], V[2], w[2]; double xi0, w0; };

// P1 traces of one side at the two points of the base rule (edge direction of
// the left element), from the scaled basis table: no FP64 multiply for the
// basis values.  w is u . (|E| w_g / 2) n, the weighted normal velocity.
__device__ __forceinline__ void p1_traces(const DevMesh& m, const double* __restrict__ cb,
                                          const double* __restrict__ ub, int64_t ne, int64_t e, int k, bool reverse,
                                          double nxw, double nyw, Tr2& t) {
  const double m0 = m.geo[G_M0 * ne + e];
  const double2 p0 = *reinterpret_cast<const double2*>(m.etb + (3 * e + k) * 4);
  const double2 p1 = *reinterpret_cast<const double2*>(m.etb + (3 * e + k) * 4 + 2);
  const double b10 = reverse ? p1.x : p0.x, b20 = reverse ? p1.y : p0.y;
  const double b11 = reverse ? p0.x : p1.x, b21 = reverse ? p0.y : p1.y;
  double c[3][3], w[3];
#pragma unroll
  for (int f = 0; f < 3; ++f)
#pragma unroll
    for (int i = 0; i < 3; ++i) c[f][i] = cb[(f * 3 + i) * ne + e];
#pragma unroll
  for (int i = 0; i < 3; ++i) w[i] = ub[i * ne + e] * nxw + ub[(3 + i) * ne + e] * nyw;
  double* out[3] = {t.xi, t.U, t.V};
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    const double a0 = c[f][0] * m0;
    out[f][0] = a0 + c[f][1] * b10 + c[f][2] * b20;
    out[f][1] = a0 + c[f][1] * b11 + c[f][2] * b21;
    if (f == 0) t.xi0 = a0;
  }
  t.w0 = w[0] * m0;
  t.w[0] = t.w0 + w[1] * b10 + w[2] * b20;
  t.w[1] = t.w0 + w[1] * b11 + w[2] * b21;
}

__device__ __forceinline__ void base_flux(const DevMesh& m, const Phys& ph, const Stage& stg, int64_t ed, int L, int R,
                                          int info, const double* __restrict__ cb, const double* __restrict__ ub,
                                          double (&F)[6], double (&jump)[2]) {
  const int64_t ne = m.ne, nE = m.nedge;
  const int kL = info & 3, kR = (info >> 2) & 3, bc = info >> 4;
  // the flux comes out weighted by wl = |E| w_g / 2 through the weighted
  // normal (nxw, nyw) = wl n, which also weights w = u.n and so lambda
  const double nxw = m.egeo[E_NXW * nE + ed], nyw = m.egeo[E_NYW * nE + ed];
  const double hmid = m.egeo[E_HMID * nE + ed];
  Tr2 a, b;
  p1_traces(m, cb, ub, ne, L, kL, false, nxw, nyw, a);
  const double unL = a.w0, HL = a.xi0 + hmid;
  double unR, HR;
  if (R >= 0) {
    p1_traces(m, cb, ub, ne, R, kR, true, nxw, nyw, b);
    unR = b.w0;
    HR = b.xi0 + hmid;
  } else if (bc == 2) {
    const double xh = tide_value(ph, stage_time(stg, m.emem[ed]));
    b = a;
    b.xi[0] = xh; b.xi[1] = xh;
    unR = unL;
    HR = xh + hmid;
  } else {
    // mirror state: q+ = q - 2 (q.n) n, (u.n)+ = -(u.n), xi+ = xi
    const double nx = m.egeo[E_NX * nE + ed], ny = m.egeo[E_NY * nE + ed];
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const double qn2 = -2.0 * (a.U[g] * nx + a.V[g] * ny);
      b.xi[g] = a.xi[g];
      b.U[g] = a.U[g] + qn2 * nx;
      b.V[g] = a.V[g] + qn2 * ny;
      b.w[g] = -a.w[g];
    }
    unR = -unL;
    HR = HL;
  }
  // lambda of Eq. (10) from the means (Sect. 3); max sqrt = sqrt max; times wl
  const double wl = m.egeo[E_WLEN * nE + ed];
  const double lam = fmax(fabs(unL), fabs(unR)) + wl * sqrt(ph.g * fmax(HL, HR));
  // momentum rows as U (w + lambda) + U+ (w+ - lambda) + P n: the two
  // factors are shared by both rows
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    const double hb = m.egeo[(E_HG0 + g) * nE + ed];
    const double P = ph.g * (a.xi[g] * (0.5 * a.xi[g] + hb) + b.xi[g] * (0.5 * b.xi[g] + hb));
    const double wa = a.w[g] + lam, wb = b.w[g] - lam;
    jump[g] = b.xi[g] - a.xi[g];
    F[0 * 2 + g] = (a.U[g] + b.U[g]) * nxw + (a.V[g] + b.V[g]) * nyw - lam * jump[g];
    F[1 * 2 + g] = a.U[g] * wa + b.U[g] * wb + P * nxw;
    F[2 * 2 + g] = a.V[g] * wa + b.V[g] * wb + P * nyw;
  }
}

}  // namespace swedg
