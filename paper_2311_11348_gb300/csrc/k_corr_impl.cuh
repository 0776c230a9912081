// Correction part of the order-separated scheme (Sect. 3, Eq. 13 and the
// text after it): every term with a test index or a coefficient index of
// degree >= 2.  Included by k_corr64.cu (FP64 correction) and k_corr32.cu
// (FP32 correction), which define CORR_T and CORR_NS before including it.
//
//   k_usolve_corr<K>   truncated auxiliary system uH = q for one order group
//                      (K x K symmetric, LDL^T), also writes the degree-1
//                      modes, the element's trace record for the edge kernel,
//                      in the first stage of a CFL step its CFL bound, and
//                      the correction of the base modes rc (volume terms of
//                      the degree-1 test modes)
//   k_edge_corr<PM>    edges with max(p_L, p_R) = PM >= 2: traces as Legendre
//                      coefficients along the edge, the moments of the LF
//                      flux, projected onto both sides' higher test modes,
//                      and the whole two-point flux for the base modes (Fb;
//                      FP32: the FP64 base flux plus the two-point equivalent
//                      of the correction flux)
//   k_elem_corr<K>     volume terms as contractions with the reference
//                      tensors of Eq. (13) (compile-time sparsity), source,
//                      the edges' projected fluxes and the SSP-RK update of
//                      the higher modes (test modes q >= 3)
//
// With CORR_TC defined (k_corr_tc.cu) the element update of the orders 3 and 4
// is that file's tensor-core kernel.
#include <algorithm>
#include <cstdio>
#include <vector>

#include "base_edge.cuh"
#include "kernels.h"
#include "tables.h"

namespace swedg {
namespace CORR_NS {

using T = CORR_T;
constexpr bool kF32 = sizeof(T) == 4;

// The FP32 correction reads FP32 copies of the base state, velocity and
// geometry (written once per element by the base kernels), so it runs no
// conversions on the FP64 pipe.
__device__ __forceinline__ const T* base_c(const StateDev& s) {
  if constexpr (kF32) return (const T*)s.cb32; else return (const T*)s.cb;
}
__device__ __forceinline__ const T* base_u(const VelDev& u) {
  if constexpr (kF32) return (const T*)u.ub32; else return (const T*)u.ub;
}
__device__ __forceinline__ const T* geo_t(const DevMesh& m) {
  if constexpr (kF32) return (const T*)m.geo32; else return (const T*)m.geo;
}
__device__ __forceinline__ const T* egeo_t(const DevMesh& m) {
  if constexpr (kF32) return (const T*)m.egeo32; else return (const T*)m.egeo;
}

__host__ __device__ constexpr int pk(int i, int j) { return i <= j ? j * (j + 1) / 2 + i : i * (i + 1) / 2 + j; }
__host__ __device__ constexpr int imax(int a, int b) { return a > b ? a : b; }
// Structural zeros of the reference tensors.  Mode i is phihat_(a,b), a + b =
// deg i, b = i - K(deg i - 1): a Legendre polynomial P_a in the collapsed
// coordinate across the triangle times a Jacobi polynomial in the other one.
// T[n][i][j] vanishes unless the degrees satisfy the triangle inequality
// (phi_i is orthogonal to every polynomial of lower degree), the Legendre
// indices satisfy it too and have an even sum (the integral of P_a P_a' P_a''),
// and for a constant factor unless the other two agree (orthonormality): 546
// of the 2250 entries T[m < 10][i][j] remain for K = 15.
// d_x phihat_q has only the modes of lower degree with a smaller Legendre index of
// the other parity; (d_y - d_x / 2) phihat_q, the derivative along the line of
// constant collapsed coordinate, those with a_m <= a_q of the same parity.
__host__ __device__ constexpr int leg_of(int i) {
  const int d = deg_of(i);
  return d - (i - (d == 0 ? 0 : Kof(d - 1)));
}
__host__ __device__ constexpr bool tri_ok(int a, int b, int c) { return a <= b + c && b <= a + c && c <= a + b; }
__host__ __device__ constexpr bool tnz(int n, int i, int j) {
  if (n == 0) return i == j;
  if (i == 0) return n == j;
  if (j == 0) return n == i;
  return tri_ok(deg_of(n), deg_of(i), deg_of(j)) && tri_ok(leg_of(n), leg_of(i), leg_of(j)) &&
         (leg_of(n) + leg_of(i) + leg_of(j)) % 2 == 0;
}
__host__ __device__ constexpr bool dxnz(int q, int m) {
  return deg_of(m) < deg_of(q) && leg_of(m) < leg_of(q) && (leg_of(q) - leg_of(m)) % 2 == 1;
}
__host__ __device__ constexpr bool dsnz(int q, int m) {
  return deg_of(m) < deg_of(q) && leg_of(m) <= leg_of(q) && (leg_of(q) - leg_of(m)) % 2 == 0;
}
// truncation of the auxiliary system (Sect. 3): K(max(deg i, deg j))
__host__ __device__ constexpr int ktr(int i, int j) { return Kof(imax(deg_of(i), deg_of(j))); }

__constant__ T cT[KMAX][120];       // T[n][i][j], (i, j) packed symmetric
__constant__ T cDx[KMAX][10];       // D_x[q][m]: d_x phihat_q = sum_m D_x[q][m] phihat_m, deg m < 4
__constant__ T cDs[KMAX][10];       // D_y[q][m] - D_x[q][m] / 2, alike
__constant__ T cEL[3][KMAX][5];     // phihat_i(gamma_k(s)) = sum_l cEL[k][i][l] P_l(2 s - 1), l <= deg i
__constant__ T cGP[3][4][5];        // per PM-2: P_l at the points t > 0 (then the middle one) of the npts_for(PM) rule on [-1,1]
__constant__ T cGW[3][4];           // their weights (the rule's weights on [0,1])

#ifdef CORR_LANES
// Terms of the entries S_ij = sum_n H_n T[n][i][j] (j <= i < 15, n < ktr(i, j), structural
// zeros left out; 390 of them) dealt to 16 lanes for k_usolve_lanes, the longest entries first,
// each to the lane with the fewest terms so far: step s of lane t adds H_n t to
// its running sum, and stores it at pk(i, j) after the entry's last term.
constexpr int UL_STEPS = 32;
struct UsolveTerms {
  double t[UL_STEPS][16];
  int code[UL_STEPS][16];  // n | (destination << 8, 255 while the sum goes on)
  int steps;
};
__device__ UsolveTerms gUsolve;

static void usolve_terms(UsolveTerms* U) {
  constexpr int K = 15;
  const RefTables& R = tables();
  struct Entry { int i, j, nz; };
  std::vector<Entry> es;
  for (int i = 0; i < K; ++i)
    for (int j = 0; j <= i; ++j) {
      int nz = 0;
      for (int n = 0; n < ktr(i, j); ++n) nz += tnz(n, i, j);
      es.push_back({i, j, nz});
    }
  std::stable_sort(es.begin(), es.end(), [](const Entry& a, const Entry& b) { return a.nz > b.nz; });
  for (int s = 0; s < UL_STEPS; ++s)
    for (int t = 0; t < 16; ++t) { U->t[s][t] = 0; U->code[s][t] = 255 << 8; }
  int used[16] = {};
  for (const Entry& e : es) {
    const int t = (int)(std::min_element(used, used + 16) - used);
    int left = e.nz;
    for (int n = 0; n < ktr(e.i, e.j); ++n) {
      if (!tnz(n, e.i, e.j)) continue;
      U->t[used[t]][t] = R.T[n][e.i][e.j];
      U->code[used[t]++][t] = n | (--left == 0 ? pk(e.i, e.j) : 255) << 8;
    }
  }
  U->steps = *std::max_element(used, used + 16);  // 25
}
#endif

void upload_tables() {
  const RefTables& R = tables();
  static T t[KMAX][120], dx[KMAX][10], ds[KMAX][10], el[3][KMAX][5], gp[3][4][5], gw[3][4];
  for (int n = 0; n < KMAX; ++n)
    for (int j = 0; j < KMAX; ++j)
      for (int i = 0; i <= j; ++i) t[n][pk(i, j)] = (T)R.T[n][i][j];
  for (int q = 0; q < KMAX; ++q)
    for (int m = 0; m < 10; ++m) {
      dx[q][m] = (T)R.D[0][q][m];
      ds[q][m] = (T)R.Ds[q][m];
    }
  for (int k = 0; k < 3; ++k)
    for (int i = 0; i < KMAX; ++i)
      for (int l = 0; l < 5; ++l) el[k][i][l] = (T)R.EL[k][i][l];
  for (int pm = 2; pm <= 4; ++pm) {
    const int N = npts_for(pm), H = N / 2;
    for (int j = 0; j < 4; ++j) {
      const bool in = j < H || (j == H && N % 2);  // points t > 0, then the middle one
      for (int l = 0; l < 5; ++l) gp[pm - 2][j][l] = in ? (T)R.GL[N][N - 1 - j][l] : (T)0;
      gw[pm - 2][j] = in ? (T)R.ew[N][N - 1 - j] : (T)0;
    }
  }
#ifdef CORR_LANES
  static UsolveTerms ut;
  usolve_terms(&ut);
  cudaMemcpyToSymbol(gUsolve, &ut, sizeof ut);
#endif
  cudaMemcpyToSymbol(cT, t, sizeof t);
  cudaMemcpyToSymbol(cDx, dx, sizeof dx);
  cudaMemcpyToSymbol(cDs, ds, sizeof ds);
  cudaMemcpyToSymbol(cEL, el, sizeof el);
  cudaMemcpyToSymbol(cGP, gp, sizeof gp);
  cudaMemcpyToSymbol(cGW, gw, sizeof gw);
}

static inline int nblocks(int64_t n, int t) { return (int)((n + t - 1) / t); }

// 16-byte accesses to 4 consecutive values (FP64: two of them)
__device__ __forceinline__ void st4(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
__device__ __forceinline__ void st4(double* p, double a, double b, double c, double d) {
  *reinterpret_cast<double2*>(p) = make_double2(a, b);
  *reinterpret_cast<double2*>(p + 2) = make_double2(c, d);
}
__device__ __forceinline__ void ld4(const float* p, float& a, float& b, float& c, float& d) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  a = v.x; b = v.y; c = v.z; d = v.w;
}
__device__ __forceinline__ void ld4(const double* p, double& a, double& b, double& c, double& d) {
  const double2 v = *reinterpret_cast<const double2*>(p), w = *reinterpret_cast<const double2*>(p + 2);
  a = v.x; b = v.y; c = w.x; d = w.y;
}

// Load all K modes of field f (base rows from the FP64 base state, higher rows
// from the group's correction array).
template <int K>
__device__ __forceinline__ void load_modes(T (&out)[K], const T* __restrict__ base, int64_t ne, int64_t e,
                                           const T* __restrict__ high, int64_t n, int64_t l, int f) {
  sfor<0, K>([&](auto i) {
    if constexpr (i < 3) out[i] = base[(f * 3 + i) * ne + e];
    else out[i] = high[(f * (K - 3) + (i - 3)) * n + l];
  });
}

// ---------------------------------------------------------------------------
// Volume terms of Eq. (13) of the higher test modes, in two steps.  The
// derivative of a basis function is a combination of the modes of lower degree,
// d_k phihat_q = sum_m D_k[q][m] phihat_m, so G_k[q][i][j] = sum_m D_k[q][m]
// T[m][i][j]: instead of one contraction with G per test mode, the products
//   Zuu_m = sum_ij T[m][i][j] U_i u_j,  Zuv, Zvu, Zvv likewise,
//   P_m   = sum_ij T[m][i][j] xi_i (xi_j / 2 + [i >= 3, j < 3] hb_j)
// are formed once for the K(p - 1) modes m below the element's degree, and
// every test mode combines them with its two rows of D.  With J^{-1} applied to
// the products (La = J0 + J2 / 2, Lb = J1 + J3 / 2 belong to D_x, J2, J3 to
// D_s = D_y - D_x / 2) and E1 = Zuu + g P, E4 = Zvv + g P,
//   r_xi[q] = sum_m D_x[q][m] (La U_m + Lb V_m) + D_s[q][m] (J2 U_m + J3 V_m)
//   r_U [q] = (1/s) sum_m D_x[q][m] (La E1 + Lb Zuv) + D_s[q][m] (J2 E1 + J3 Zuv)
//   r_V [q] = (1/s) sum_m D_x[q][m] (La Zvu + Lb E4) + D_s[q][m] (J2 Zvu + J3 E4)
// This is 2,300 multiply-adds for K = 15 (10: 760, 6: 200) where the G tensors
// of every test mode took 10,200 (2,900, 540).
// The bottom term g xi h_b keeps only the products with a higher elevation
// mode i >= 3: the rest, g (xi_lin h_b) with xi_lin the degree-1 part of xi,
// integrates by parts to its own boundary integral (the gradient of
// xi_lin h_b is linear, so phi_q of degree >= 2 is orthogonal to it): the
// correction edge kernel moves that integral into the edge flux, where it
// meets the flux's own g xi_lin h_b term and leaves g h_b times the jump of
// xi_lin, formed in FP64.  In FP32 the two O(g |xi| h_b) integrals otherwise
// cancel to a residual several orders of magnitude smaller and carry their
// rounding error into it.
// ---------------------------------------------------------------------------
// the products of one mode M: z = {Zuu + g P, Zuv, Zvu, Zvv + g P}
template <int K, int M>
__device__ __forceinline__ void products(T (&z)[4], const T (&xi)[K], const T (&U)[K], const T (&V)[K],
                                         const T (&u)[K], const T (&v)[K], const T (&xh)[3], T g) {
  T z0 = 0, z1 = 0, z2 = 0, z3 = 0, P = 0;
  sfor<0, K>([&](auto i) {
    constexpr bool any = [] {
      for (int j = 0; j < K; ++j)
        if (tnz(M, decltype(i)::value, j)) return true;
      return false;
    }();
    if constexpr (any) {
      T a = 0, b = 0, w = 0;
      sfor<0, K>([&](auto j) {
        if constexpr (tnz(M, i, j)) {
          const T t = cT[M][pk(i, j)];
          a = fma(u[j], t, a);
          b = fma(v[j], t, b);
          // each unordered pair of P once: xi_i xi_j, on the diagonal half of it
          if constexpr (j < i) w = fma(i >= 3 && j < 3 ? xh[j < 3 ? j : 0] : xi[j], t, w);
          if constexpr (j == i) w = fma((T)0.5 * xi[i], t, w);
        }
      });
      z0 = fma(U[i], a, z0); z1 = fma(U[i], b, z1);
      z2 = fma(V[i], a, z2); z3 = fma(V[i], b, z3);
      P = fma(xi[i], w, P);
    }
  });
  z[0] = fma(g, P, z0);
  z[1] = z1;
  z[2] = z2;
  z[3] = fma(g, P, z3);
}

// orders whose element update runs on the tensor cores (for K = 6 the GEMMs
// would be a few columns)
#ifdef CORR_TC
__host__ __device__ constexpr bool on_tc(int K) { return K >= 10; }
#else
__host__ __device__ constexpr bool on_tc(int K) { return false; }
#endif

// ---------------------------------------------------------------------------
// auxiliary system of one order group:  M u = U, M v = V,
//   M[i][j] = (1/s) sum_{n < K(max deg)} H_n T[n][i][j],  H = xi + h_b.
// Solved as S u = s U with S = s M by an unpivoted LDL^T factorisation.
// With rc given, the same thread then forms the correction of the base modes
// (the volume terms of the degree-1 test modes with a coefficient of degree
// >= 2) from the velocity it has just solved for, so that the base element
// kernel can take it without waiting for the correction element kernel.
// ---------------------------------------------------------------------------
template <int K>
__device__ __forceinline__ void usolve_corr_body(const DevMesh& m, int64_t g0, int64_t n, const Phys& ph,
                                                 const StateDev& c, const T* __restrict__ ch, double* __restrict__ ub,
                                                 float* __restrict__ ub32, T* __restrict__ uh,
                                                 T* __restrict__ tr, T* __restrict__ trv,
                                                 unsigned* status, unsigned long long* dmin,
                                                 double* __restrict__ rc, int64_t rc_off, int64_t nrc) {
  const int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  double u00 = 0.0, v00 = 0.0, H0d = 0.0;  // mode 0 of u and v as stored, and of the depth (FP64)
  if (l < n) {
    const int64_t e = g0 + l, ne = m.ne;
    constexpr int KH = K - 3, NP = K * (K + 1) / 2;
    const T* cb = base_c(c);
    const T* geo = geo_t(m);
    T H[K];
    load_modes<K>(H, cb, ne, e, ch, n, l, 0);
    H[0] += geo[G_HB0 * ne + e];
    H[1] += geo[G_HB1 * ne + e];
    H[2] += geo[G_HB2 * ne + e];
    // depth check on the FP64 mean (base modes are FP64 in every mode)
    H0d = c.cb[e] + m.geo[G_HB0 * ne + e];
    if (!(H0d * m.geo[G_RS * ne + e] * 1.4142135623730951 > ph.h_min)) {
      atomicOr(status, (unsigned)ST_DEPTH);
      atomicOr(m.mstatus + m.mem[e], (unsigned)ST_DEPTH);
    }
    const T sv = geo[G_S * ne + e];
    T A[NP];
    sfor<0, K>([&](auto j) {
      sfor<0, j + 1>([&](auto i) {
        T acc = 0;
        sfor<0, ktr(i, j)>([&](auto nn) {
          if constexpr (tnz(nn, i, j)) acc = fma(H[nn], cT[nn][pk(i, j)], acc);
        });
        A[pk(i, j)] = acc;
      });
    });
    T rd[K];  // 1/d_j
    if constexpr (!kF32 && K == 15) {
      // LDL^T: row j's products L_jk d_k are shared by every row below it
      T dg[K];
      sfor<0, K>([&](auto j) {
        T ld[K];
        T dj = A[pk(j, j)];
        sfor<0, j>([&](auto k) {
          ld[k] = A[pk(j, k)] * dg[k];
          dj = fma(-A[pk(j, k)], ld[k], dj);
        });
        dg[j] = dj;
        rd[j] = (T)1 / dj;
        sfor<j + 1, K>([&](auto i) {
          T w = A[pk(i, j)];
          sfor<0, j>([&](auto k) { w = fma(-A[pk(i, k)], ld[k], w); });
          A[pk(i, j)] = w * rd[j];
        });
      });
    } else {
      // row j holds W_jk = L_jk d_k until its turn, then L_jk: one product per
      // entry fewer (FP64, K = 15 spills more registers this way: 95 against 77 us
      // for up to 10,000 elements)
      sfor<0, K>([&](auto j) {
        T dj = A[pk(j, j)];
        sfor<0, j>([&](auto k) {
          const T L = A[pk(j, k)] * rd[k];
          dj = fma(-A[pk(j, k)], L, dj);
          A[pk(j, k)] = L;
        });
        rd[j] = (T)1 / dj;
        sfor<j + 1, K>([&](auto i) {
          T w = A[pk(i, j)];
          sfor<0, j>([&](auto k) { w = fma(-A[pk(i, k)], A[pk(j, k)], w); });
          A[pk(i, j)] = w;
        });
      });
    }
    T x[2][K];
    load_modes<K>(x[0], cb, ne, e, ch, n, l, 1);
    load_modes<K>(x[1], cb, ne, e, ch, n, l, 2);
    const T s = sv;
    sfor<0, 2>([&](auto r) {
      sfor<0, K>([&](auto i) { sfor<0, i>([&](auto k) { x[r][i] = fma(-A[pk(i, k)], x[r][k], x[r][i]); }); });
      sfor<0, K>([&](auto i) { x[r][i] *= rd[i]; });
      sfor<0, K>([&](auto ii) {
        constexpr int i = K - 1 - ii;
        sfor<0, ii>([&](auto kk) {
          constexpr int k = K - 1 - kk;
          x[r][i] = fma(-A[pk(k, i)], x[r][k], x[r][i]);
        });
      });
      sfor<0, K>([&](auto i) {
        const T v = x[r][i] * s;
        if constexpr (i < 3) {
          ub[(r * 3 + i) * ne + e] = (double)v;
          if constexpr (kF32) ub32[(r * 3 + i) * ne + e] = v;
          if constexpr (i == 0) {
            if constexpr (r == 0) u00 = (double)v; else v00 = (double)v;
          }
        } else {
          uh[(r * KH + (i - 3)) * n + l] = v;
        }
      });
    });
    T xi[K], U[K], V[K];
    load_modes<K>(xi, cb, ne, e, ch, n, l, 0);
    load_modes<K>(U, cb, ne, e, ch, n, l, 1);
    load_modes<K>(V, cb, ne, e, ch, n, l, 2);
    // this element's trace record for the correction edges (VelDev::tr)
    sfor<0, K>([&](auto i) {
      st4(tr + (l * K + i) * 4, xi[i], U[i], V[i], x[0][i] * s);
      trv[l * K + i] = x[1][i] * s;
    });
    if (rc) {
      // test modes of degree 1 have a constant gradient, so by orthonormality
      // their volume terms are sums over the modes alone (i >= 3 here)
      T e1 = 0, e2 = 0, e3 = 0, e4 = 0, px = 0;
      sfor<3, K>([&](auto j) {
        const T uu = x[0][j] * s, vv = x[1][j] * s;  // the velocity modes as stored above
        e1 = fma(U[j], uu, e1); e2 = fma(U[j], vv, e2);
        e3 = fma(V[j], uu, e3); e4 = fma(V[j], vv, e4);
        px = fma(xi[j], xi[j], px);
      });
      const T hg = (T)0.5 * (T)ph.g;
      e1 = fma(hg, px, e1);
      e4 = fma(hg, px, e4);
      const T x1 = geo[G_GQ1X * ne + e], y1 = geo[G_GQ1Y * ne + e];
      const T x2 = geo[G_GQ2X * ne + e], y2 = geo[G_GQ2Y * ne + e];
      rc[0 * nrc + rc_off + l] = (double)fma(x1, e1, y1 * e2);
      rc[1 * nrc + rc_off + l] = (double)fma(x2, e1, y2 * e2);
      rc[2 * nrc + rc_off + l] = (double)fma(x1, e3, y1 * e4);
      rc[3 * nrc + rc_off + l] = (double)fma(x2, e3, y2 * e4);
    }
  }
  if (dmin) {  // uniform over the grid: every thread of the block is here
    const bool in = l < n;
    const int64_t x = in ? g0 + l : 0;
    cfl_fold(dmin, in, m.mem[x], u00, v00, H0d, m.geo[G_RS * m.ne + x], ph.g, m.geo[G_DIAM * m.ne + x], m.p[x]);
  }
}

// The compiler's register allocation (FP32: 72, 128, 233 registers for K =
// 6, 10, 15), and for K = 15 in FP32 a second build in 168 registers (3
// blocks per SM) for launch shapes that cap the base grids: the few base blocks
// leave room for more of its warps.
template <int K>
__global__ void __launch_bounds__(128) k_usolve_corr(DevMesh m, int64_t g0, int64_t n, Phys ph, StateDev c,
                                                     const T* __restrict__ ch, double* __restrict__ ub,
                                                     float* __restrict__ ub32, T* __restrict__ uh,
                                                     T* __restrict__ tr, T* __restrict__ trv,
                                                     unsigned* status, unsigned long long* dmin,
                                                     double* __restrict__ rc, int64_t rc_off, int64_t nrc) {
  usolve_corr_body<K>(m, g0, n, ph, c, ch, ub, ub32, uh, tr, trv, status, dmin, rc, rc_off, nrc);
}
template <int K>
__global__ void __launch_bounds__(128, 3) k_usolve_corr15(DevMesh m, int64_t g0, int64_t n, Phys ph, StateDev c,
                                                         const T* __restrict__ ch, double* __restrict__ ub,
                                                         float* __restrict__ ub32, T* __restrict__ uh,
                                                         T* __restrict__ tr, T* __restrict__ trv,
                                                         unsigned* status, unsigned long long* dmin,
                                                         double* __restrict__ rc, int64_t rc_off, int64_t nrc) {
  usolve_corr_body<K>(m, g0, n, ph, c, ch, ub, ub32, uh, tr, trv, status, dmin, rc, rc_off, nrc);
}

// The solve of FP64 groups of order 4 with 16 lanes per element, for small groups:
// one thread runs 1,700 FP64 instructions one after the other, 64 cycles each.
// Lane i holds row i; the entries are summed by the lanes in shares of equal
// length and the elimination broadcasts L_kj d_j from lane to lane, about 300
// instructions per warp of two elements (twice the total).  Every operation on an
// element is the same, in the same order, as in the one-thread form, so the
// results are too.  74 to 76 us for any group up to 10,000 elements on one thread;
// here 24 us for 512, 74 for 5,000, 115 for 10,000 (GB300, alone); beside the other groups'
// kernels, which share the FP64 pipe, it pays up to about 3,000.
#ifdef CORR_LANES
constexpr int64_t UL_MAX = 3000;
constexpr int UL_BLOCK = 128, UL_EL = UL_BLOCK / 16;
__global__ void __launch_bounds__(UL_BLOCK) k_usolve_lanes(DevMesh m, int64_t g0, int64_t n, Phys ph, StateDev c,
                                                           const T* __restrict__ ch, double* __restrict__ ub,
                                                           T* __restrict__ uh,
                                                           T* __restrict__ tr, T* __restrict__ trv, unsigned* status,
                                                           unsigned long long* dmin, double* __restrict__ rc,
                                                           int64_t rc_off, int64_t nrc) {
  constexpr int K = 15, KH = K - 3, NP = K * (K + 1) / 2;
  __shared__ T sA[UL_EL][NP], sH[UL_EL][16], sx[UL_EL][5][16];
  const unsigned full = 0xffffffffu;
  const int g = threadIdx.x >> 4, i = threadIdx.x & 15;
  const int64_t l = blockIdx.x * (int64_t)UL_EL + g, ne = m.ne;
  const bool live = l < n, row = live && i < K;
  const int64_t e = g0 + (live ? l : 0);
  const T* cb = base_c(c);
  const T* geo = geo_t(m);
  T xi = 0, x[2] = {0, 0};
  if (row) {
    if (i < 3) {
      xi = cb[i * ne + e]; x[0] = cb[(3 + i) * ne + e]; x[1] = cb[(6 + i) * ne + e];
    } else {
      xi = ch[(i - 3) * n + l]; x[0] = ch[(KH + i - 3) * n + l]; x[1] = ch[(2 * KH + i - 3) * n + l];
    }
  }
  const T U = x[0], V = x[1];
  double H0d = 0.0;
  if (live && i == 0) {  // depth check on the FP64 mean
    H0d = c.cb[e] + m.geo[G_HB0 * ne + e];
    if (!(H0d * m.geo[G_RS * ne + e] * 1.4142135623730951 > ph.h_min)) {
      atomicOr(status, (unsigned)ST_DEPTH);
      atomicOr(m.mstatus + m.mem[e], (unsigned)ST_DEPTH);
    }
  }
  sH[g][i] = row && i < 3 ? xi + geo[(G_HB0 + i) * ne + e] : xi;
  __syncwarp();
  {
    const UsolveTerms& tb = gUsolve;
    const int steps = tb.steps;
    T acc = 0;
    for (int s = 0; s < steps; ++s) {
      const int code = tb.code[s][i], dst = code >> 8;
      acc = fma(sH[g][code & 255], tb.t[s][i], acc);
      if (dst != 255) {
        sA[g][dst] = acc;
        acc = 0;
      }
    }
  }
  __syncwarp();
  // row i of the lower triangle (lanes without a row: the identity)
  T a[K], rdi = 1;
  sfor<0, K>([&](auto j) { a[j] = row && j <= i ? sA[g][pk(i < K ? i : 0, j)] : (T)(j == i); });
  sfor<0, K>([&](auto j) {
    const T d = __shfl_sync(full, a[j], j, 16), rd = (T)1 / d;
    if (i == j) rdi = rd;
    const T lij = a[j] * rd, ld = lij * d;  // L_ij, L_ij d_j (i > j)
    sfor<j + 1, K>([&](auto k) {
      const T ldk = __shfl_sync(full, ld, k, 16);
      if (i >= k) a[k] = fma(-lij, ldk, a[k]);
    });
    if (i > j) a[j] = lij;
  });
  sfor<0, K>([&](auto j) {
    if (row && j < i) sA[g][pk(i < K ? i : 0, j)] = a[j];
  });
  __syncwarp();
  sfor<0, 2>([&](auto r) {
    sfor<0, K>([&](auto j) {
      const T xj = __shfl_sync(full, x[r], j, 16);
      if (i > j) x[r] = fma(-a[j], xj, x[r]);
    });
    x[r] *= rdi;
  });
  sfor<0, K>([&](auto k) { a[k] = row && i < k ? sA[g][pk(i < K ? i : 0, k)] : (T)0; });  // column i of L
  sfor<0, 2>([&](auto r) {
    sfor<0, K>([&](auto kk) {
      constexpr int k = K - 1 - kk;
      const T xk = __shfl_sync(full, x[r], k, 16);
      if (i < k) x[r] = fma(-a[k], xk, x[r]);
    });
  });
  const T s = geo[G_S * ne + e];
  const T uu = x[0] * s, vv = x[1] * s;
  if (row) {
    if (i < 3) {
      ub[i * ne + e] = (double)uu;
      ub[(3 + i) * ne + e] = (double)vv;
    } else {
      uh[(i - 3) * n + l] = uu;
      uh[(KH + i - 3) * n + l] = vv;
    }
    st4(tr + (l * K + i) * 4, xi, U, V, uu);
    trv[l * K + i] = vv;
  }
  if (rc) {  // see usolve_corr_body; lane q < 4 forms rc[q], lanes 0 .. 4 the five sums
    sx[g][0][i] = U; sx[g][1][i] = V; sx[g][2][i] = uu; sx[g][3][i] = vv; sx[g][4][i] = xi;
    __syncwarp();
    const int pa = i == 4 ? 4 : i >> 1 & 1, pb = i == 4 ? 4 : 2 + (i & 1);  // U u, U v, V u, V v, xi xi
    T sum = 0;
    if (i < 5)
      for (int j = 3; j < K; ++j) sum = fma(sx[g][pa][j], sx[g][pb][j], sum);
    const T px = __shfl_sync(full, sum, 4, 16);
    if (i == 0 || i == 3) sum = fma((T)0.5 * (T)ph.g, px, sum);
    const T ea = __shfl_sync(full, sum, i >> 1 << 1 & 15, 16), eb = __shfl_sync(full, sum, (i >> 1 << 1 | 1) & 15, 16);
    if (live && i < 4) {
      const T gx = geo[(i & 1 ? G_GQ2X : G_GQ1X) * ne + e], gy = geo[(i & 1 ? G_GQ2Y : G_GQ1Y) * ne + e];
      rc[i * nrc + rc_off + l] = (double)fma(gx, ea, gy * eb);
    }
  }
  if (dmin)  // uniform over the grid
    cfl_fold(dmin, live && i == 0, m.mem[e], (double)uu, (double)vv, H0d, m.geo[G_RS * ne + e], ph.g,
             m.geo[G_DIAM * ne + e], m.p[e]);
}
#endif

template <int K>
static int usolve_group(cudaStream_t st, const DevMesh& m, const Groups& G, int p, const Phys& ph, StateDev c,
                        VelDev u, unsigned* status, unsigned long long* dmin, void* rc) {
  const int64_t g0 = G.start[p], n = G.start[p + 1] - g0;
  if (n == 0) return 0;
  const int64_t nrc = G.start[5] - G.start[2], rc_off = g0 - G.start[2];
  const int ct = spread_threads(n, launch_shape().corr_threads);
#ifdef CORR_LANES
  if (K == 15 && n <= UL_MAX) {
    k_usolve_lanes<<<nblocks(n, UL_EL), UL_BLOCK, 0, st>>>(m, g0, n, ph, c, (const T*)c.ch[p], u.ub, (T*)u.uh[p],
                                                           (T*)u.tr[p], (T*)u.trv[p], status, dmin, (double*)rc,
                                                           rc_off, nrc);
    count_launch();
    SWE_CUDA_OK(cudaGetLastError());
    return 0;
  }
#endif
  bool capped = false;
  if constexpr (K == 15 && kF32) {
    capped = launch_shape().base_bpsm > 0;
    if (capped)
      k_usolve_corr15<K><<<nblocks(n, ct), ct, 0, st>>>(m, g0, n, ph, c, (const T*)c.ch[p], u.ub, u.ub32,
                                                        (T*)u.uh[p], (T*)u.tr[p], (T*)u.trv[p], status, dmin,
                                                        (double*)rc, rc_off, nrc);
  }
  if (!capped)
    k_usolve_corr<K><<<nblocks(n, ct), ct, 0, st>>>(m, g0, n, ph, c, (const T*)c.ch[p], u.ub, u.ub32,
                                                      (T*)u.uh[p], (T*)u.tr[p], (T*)u.trv[p], status, dmin,
                                                      (double*)rc, rc_off, nrc);
  count_launch();
  SWE_CUDA_OK(cudaGetLastError());
  return 0;
}

int launch_usolve_corr(GroupStreams gs, const DevMesh& m, const Groups& G, const Phys& ph, StateDev c, VelDev u,
                       unsigned* status, unsigned long long* dmin, void* rc) {
  int r = usolve_group<6>(gs.s[0], m, G, 2, ph, c, u, status, dmin, rc);
  if (!r) r = usolve_group<10>(gs.s[1], m, G, 3, ph, c, u, status, dmin, rc);
  if (!r) r = usolve_group<15>(gs.s[2], m, G, 4, ph, c, u, status, dmin, rc);
  return r;
}

// ---------------------------------------------------------------------------
// correction edge flux.  Along an edge every trace is a polynomial of the
// side's degree; with t = 2 s - 1 in the left element's parameter s it is held as
// Legendre coefficients (the right side runs the edge the other way: its odd
// coefficients change sign), and the test functions see a flux only through its
// moments m_l = int_0^1 F P_l(t) ds, l <= the side's degree.  Linear terms of the
// flux go from coefficients to moments directly (m_l = F_l / (2 l + 1)), so do
// the products with the linear h_b; only the products U w, V w and xi^2 are
// formed at the npts_for(PM) Gauss points, in pairs +-t whose even and odd
// parts are shared.  With w = u.n the momentum flux is
//   F_U = U_L w_L + U_R w_R + lambda (U_L - U_R) + g nx (xi_L^2 / 2 + xi_R^2 / 2 + h_b (xi_L + xi_R)).
// The test modes of degree >= 2 see this flux with its g xi_lin h_b terms
// replaced by g h_b times the jump of xi_lin (the volume term's share, see
// products).
// FP64 writes the moments of degree <= 1 of the whole flux as the edge's
// two-point flux.
// FP32 splits every trace into its P1 part (b) and the higher part (h): the
// correction's share of the base modes, from
//   U w - U_b w_b = U_h w + U_b w_h,  xi^2 / 2 - xi_b^2 / 2 = xi_h (xi_b + xi_h / 2),
// carries no cancellation against the base flux; the products of two P1 parts
// reach the higher test modes through their three moments in closed form.  The
// same thread computes the base flux in FP64 and stores the sum, one flux for
// both sides of the edge: a separate array cost the base element kernel 18
// FP64 additions and 18 loads per element.
// All fluxes are weighted by |E| / 4 (the weight of the two-point base rule)
// through the normal.
// FP64 is bound by its instruction count (about 350, 640, 1,100 per edge of
// pmax = 2, 3, 4 with one side an order lower, against 700, 1,450, 3,000 and the base
// flux for traces and projections mode by mode at every point): 229, 379, 620 us for
// 249,000 edges between elements of order 2, 3, 4 (GB300, alone), 0.9, 1.5, 2.5 ns
// per edge where the other form took 1.6, 2.9, 5.8.  FP32 waits on the gathers of
// the two trace records and of the FP64 base state: 70, 82, 108 us for the same
// edges with the FP64 base flux; 117, 126, 128 registers, so that every pmax
// runs 4 blocks per SM.
// ---------------------------------------------------------------------------
template <int PM>
struct SideC {
  T x[PM + 1];                       // the higher part of the elevation
  T U[PM + 1], V[PM + 1], w[PM + 1];  // FP64: the whole trace; FP32: its higher part
  T xl[2], Ul[2], Vl[2], wl[2];      // the P1 part (FP64: only xl is kept apart)
  T un, xm;                                      // mean normal velocity and mean elevation
};

template <int PM>
__device__ __forceinline__ void side_coefs(const DevMesh& m, const Groups& G, const StateDev& c, const VelDev& u,
                                           int64_t e, int p, int k, bool reverse, T nxw, T nyw, SideC<PM>& S) {
  const int64_t ne = m.ne;
  const int K = Kof(p);
  const T rs = geo_t(m)[G_RS * ne + e];
  const T* cbt = base_c(c);
  const T* ubt = base_u(u);
  // an element of order >= 2 reads its trace record (16 + 4 bytes per mode),
  // an element of order <= 1 its base modes from the base state and velocity
  const T* r4 = nullptr;
  const T* rv = nullptr;
  if (p >= 2) {  // selects, not a runtime index into the parameter arrays (that would copy them to the stack)
    const int64_t s0 = p == 2 ? G.start[2] : p == 3 ? G.start[3] : G.start[4];
    const int64_t l = e - s0;
    r4 = (const T*)(p == 2 ? u.tr[2] : p == 3 ? u.tr[3] : u.tr[4]) + l * K * 4;
    rv = (const T*)(p == 2 ? u.trv[2] : p == 3 ? u.trv[3] : u.trv[4]) + l * K;
  }
  sfor<0, PM + 1>([&](auto l) { S.x[l] = S.U[l] = S.V[l] = S.w[l] = 0; });
  S.xl[1] = S.Ul[1] = S.Vl[1] = S.wl[1] = 0;
  sfor<0, Kof(PM)>([&](auto i) {
    if (i >= K && i >= 3) return;
    T cx, cU, cV, cu, cv;
    if (p >= 2) {
      ld4(r4 + i * 4, cx, cU, cV, cu);
      cv = rv[i];
    } else if constexpr (i < 3) {
      cx = cbt[(0 * 3 + i) * ne + e]; cU = cbt[(1 * 3 + i) * ne + e]; cV = cbt[(2 * 3 + i) * ne + e];
      cu = ubt[(0 * 3 + i) * ne + e]; cv = ubt[(1 * 3 + i) * ne + e];
    }
    const T cw = cu * nxw + cv * nyw;
    if constexpr (i == 0) {
      const T b = cEL[0][0][0];  // the constant mode, the same on every edge
      S.xl[0] = cx * b; S.Ul[0] = cU * b; S.Vl[0] = cV * b; S.wl[0] = cw * b;
      S.xm = S.xl[0] * rs;
      S.un = S.wl[0] * rs;
    } else {
      sfor<0, deg_of(i) + 1>([&](auto l) {
        const T b = cEL[k][i][l];
        if constexpr (i < 3) {
          S.xl[l] += cx * b; S.Ul[l] += cU * b; S.Vl[l] += cV * b; S.wl[l] += cw * b;
        } else {
          S.x[l] += cx * b; S.U[l] += cU * b; S.V[l] += cV * b; S.w[l] += cw * b;
        }
      });
    }
  });
  const T rso = reverse ? -rs : rs;  // odd coefficients change sign on the reversed edge
  if constexpr (!kF32) {
    sfor<0, 2>([&](auto l) { S.U[l] += S.Ul[l]; S.V[l] += S.Vl[l]; S.w[l] += S.wl[l]; });
  }
  sfor<0, PM + 1>([&](auto l) {
    const T f = l % 2 ? rso : rs;
    S.x[l] *= f; S.U[l] *= f; S.V[l] *= f; S.w[l] *= f;
  });
  S.xl[0] *= rs;
  S.xl[1] *= rso;
  if constexpr (kF32) {
    S.Ul[0] *= rs; S.Vl[0] *= rs; S.wl[0] *= rs;
    S.Ul[1] *= rso; S.Vl[1] *= rso; S.wl[1] *= rso;
  }
}

// values at the points +t and -t of pair j (the middle point: j = N / 2, N odd, in vp) of sum_l c[l] P_l
template <int PM, int J>
__device__ __forceinline__ void at_pair(const T (&c)[PM + 1], T& vp, T& vm) {
  constexpr int GI = PM - 2;
  T ev = c[0] + c[2] * cGP[GI][J][2];
  if constexpr (PM >= 4) ev += c[4] * cGP[GI][J][4];
  if constexpr (2 * J + 1 == npts_for(PM)) {
    vp = vm = ev;
  } else if constexpr (PM >= 3) {
    const T od = c[1] * cGP[GI][J][1] + c[3] * cGP[GI][J][3];
    vp = ev + od;
    vm = ev - od;
  } else {
    vp = ev + c[1] * cGP[GI][J][1];
    vm = ev - c[1] * cGP[GI][J][1];
  }
}

// r += the three moments (l = 0, 1, 2) of the product of two linear functions
__device__ __forceinline__ void add_lin2(T& r0, T& r1, T& r2, const T (&a)[2], const T (&b)[2]) {
  const T p = a[1] * b[1];
  r0 += a[0] * b[0] + p * (T)(1.0 / 3.0);
  r1 += (a[0] * b[1] + a[1] * b[0]) * (T)(1.0 / 3.0);
  r2 += p * (T)(2.0 / 15.0);
}

template <int PM>
__device__ __forceinline__ void edge_corr_body(const DevMesh& m, const int32_t* __restrict__ list, int64_t nl,
                                               const Groups& G, const Phys& ph, const Stage& stg, const StateDev& c,
                                               const VelDev& u, const EdgeFlux& fx) {
  constexpr int N = npts_for(PM), GI = PM - 2;
  void* const* Pf = fx.Pf;
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= nl) return;
  const int64_t ed = list[idx], nE = m.nedge;
  const int L = m.eL[ed], R = m.eR[ed], info = m.einfo[ed];
  const int kL = info & 3, kR = (info >> 2) & 3, bc = info >> 4;
  const int pL = m.p[L], pR = R >= 0 ? m.p[R] : 0;
  const T* eg = egeo_t(m);
  const T nxw = eg[E_NXW * nE + ed], nyw = eg[E_NYW * nE + ed], wl = eg[E_WLEN * nE + ed];
  const T h0 = eg[E_HMID * nE + ed], h1 = (T)0.5 * (eg[E_HB * nE + ed] - eg[E_HA * nE + ed]);
  const T g = (T)ph.g;
  // jump of the degree-1 elevation along the edge, j0 + j1 t (zero on land): it
  // carries the volume term g xi_lin h_b of the higher test modes (moved here,
  // see products), and in FP32 lambda (xi_L - xi_R) of the P1 parts too, whose FP32
  // traces would leave the rounding of xi times lambda (smooth state over deep
  // water: elevation rows of degree 2 - 4 2.9e-4 that way, 5.0e-5 with this jump)
  T j0 = 0, j1 = 0;
  double F[6];
  if constexpr (kF32) {
    // the base flux, in FP64, with the jump at its two points t = -+1 / sqrt 3
    double jump[2];
    base_flux(m, ph, stg, ed, L, R, info, c.cb, u.ub, F, jump);
    j0 = (T)(0.5 * (jump[0] + jump[1]));
    j1 = (T)(0.8660254037844386 * (jump[1] - jump[0]));
  }
  SideC<PM> a, b;
  side_coefs<PM>(m, G, c, u, L, pL, kL, false, nxw, nyw, a);
  if (R >= 0) {
    side_coefs<PM>(m, G, c, u, R, pR, kR, true, nxw, nyw, b);
  } else if (bc == 2) {
    const T xh = (T)tide_value(ph, stage_time(stg, m.emem[ed]));
    b = a;
    sfor<0, PM + 1>([&](auto l) { b.x[l] = 0; });
    b.xl[0] = xh;
    b.xl[1] = 0;
    b.xm = xh;
  } else {
    const T nx = eg[E_NX * nE + ed], ny = eg[E_NY * nE + ed];
    b = a;
    sfor<0, PM + 1>([&](auto l) {
      const T qn = 2 * (a.U[l] * nx + a.V[l] * ny);
      b.U[l] = a.U[l] - qn * nx;
      b.V[l] = a.V[l] - qn * ny;
      b.w[l] = -a.w[l];
    });
    sfor<0, 2>([&](auto l) {
      const T qn = 2 * (a.Ul[l] * nx + a.Vl[l] * ny);
      b.Ul[l] = a.Ul[l] - qn * nx;
      b.Vl[l] = a.Vl[l] - qn * ny;
      b.wl[l] = -a.wl[l];
    });
    b.un = -a.un;
  }
  if constexpr (!kF32) {
    if (R >= 0 || bc == 2) {
      j0 = b.xl[0] - a.xl[0];
      j1 = b.xl[1] - a.xl[1];
    }
  }
  // lambda of Eq. (10) from the element means (Sect. 3), weighted like w
  const T lam = fmax(fabs(a.un), fabs(b.un)) + wl * sqrt(g * fmax(a.xm + h0, b.xm + h0));
  // the linear terms: the elevation row and the jump terms lambda (c_L - c_R).
  // lambda (about sqrt(g h)) is orders of magnitude above w, so products with w
  // +- lambda would drop w's low bits and leave lambda (U_L - U_R) to the
  // difference of two rounded products.  That saves 12 FP64 instructions per edge
  // of pmax = 2 (0.5 % of an FP64 step, nothing in FP32) and costs accuracy: error
  // of a mixed step of p 1 - 3 over deep water 7.4e-10 instead of 5.6e-10, of the
  // FP64 momentum rows of p 0 - 4 3.6e-15 instead of 3.3e-15 (against 80 bits).
  T ax[PM + 1], bx[PM + 1];  // FP64: the whole elevation; FP32: its higher part, as U, V, w
  T m0[PM + 1], m1[PM + 1], m2[PM + 1], lc[PM + 1];
  sfor<0, PM + 1>([&](auto l) {
    constexpr T c = (T)(1.0 / (2 * l + 1));
    lc[l] = lam * c;
    ax[l] = a.x[l];
    bx[l] = b.x[l];
    if constexpr (!kF32 && l < 2) {
      ax[l] += a.xl[l];
      bx[l] += b.xl[l];
    }
    m0[l] = ((a.U[l] + b.U[l]) * nxw + (a.V[l] + b.V[l]) * nyw) * c + lc[l] * (ax[l] - bx[l]);
    m1[l] = lc[l] * (a.U[l] - b.U[l]);
    m2[l] = lc[l] * (a.V[l] - b.V[l]);
  });
  T z0[2], z1[3], z2[3];  // FP32: moments of the P1 parts' flux (elevation row; momentum rows)
  if constexpr (kF32) {
    sfor<0, 2>([&](auto l) {
      constexpr T c = (T)(1.0 / (2 * l + 1));
      z0[l] = ((a.Ul[l] + b.Ul[l]) * nxw + (a.Vl[l] + b.Vl[l]) * nyw) * c - lc[l] * (l == 0 ? j0 : j1);
      z1[l] = lc[l] * (a.Ul[l] - b.Ul[l]);
      z2[l] = lc[l] * (a.Vl[l] - b.Vl[l]);
    });
    z1[2] = z2[2] = 0;
  }
  // the products, at the Gauss points
  const T gnx = g * nxw, gny = g * nyw;
  sfor<0, (N + 1) / 2>([&](auto J) {
    constexpr bool mid = 2 * J + 1 == N;
    T f1[2] = {0, 0}, f2[2] = {0, 0}, pp[2] = {0, 0};
    auto side = [&](const SideC<PM>& S, const T (&sx)[PM + 1]) {
      T x[2], U[2], V[2], w[2];
      at_pair<PM, J>(sx, x[0], x[1]);
      at_pair<PM, J>(S.U, U[0], U[1]);
      at_pair<PM, J>(S.V, V[0], V[1]);
      at_pair<PM, J>(S.w, w[0], w[1]);
      sfor<0, mid ? 1 : 2>([&](auto s) {
        if constexpr (kF32) {
          const T t = s == 0 ? cGP[GI][J][1] : -cGP[GI][J][1];
          const T xb = S.xl[0] + S.xl[1] * t, Ub = S.Ul[0] + S.Ul[1] * t, Vb = S.Vl[0] + S.Vl[1] * t;
          const T wf = S.wl[0] + S.wl[1] * t + w[s];
          f1[s] += U[s] * wf + Ub * w[s];
          f2[s] += V[s] * wf + Vb * w[s];
          pp[s] += x[s] * (xb + (T)0.5 * x[s]);
        } else {
          f1[s] += U[s] * w[s];
          f2[s] += V[s] * w[s];
          pp[s] += x[s] * x[s];
        }
      });
    };
    side(a, ax);
    side(b, bx);
    sfor<0, mid ? 1 : 2>([&](auto s) {
      const T P = kF32 ? pp[s] : (T)0.5 * pp[s];
      f1[s] += P * gnx;
      f2[s] += P * gny;
    });
    const T wgt = cGW[GI][J];
    if constexpr (mid) {
      f1[0] *= wgt;
      f2[0] *= wgt;
      sfor<0, PM + 1>([&](auto l) {
        if constexpr (l % 2 == 0) {
          m1[l] += f1[0] * cGP[GI][J][l];
          m2[l] += f2[0] * cGP[GI][J][l];
        }
      });
    } else {
      const T e1 = wgt * (f1[0] + f1[1]), o1 = wgt * (f1[0] - f1[1]);
      const T e2 = wgt * (f2[0] + f2[1]), o2 = wgt * (f2[0] - f2[1]);
      sfor<0, PM + 1>([&](auto l) {
        m1[l] += (l % 2 ? o1 : e1) * cGP[GI][J][l];
        m2[l] += (l % 2 ? o2 : e2) * cGP[GI][J][l];
      });
    }
  });
  // h_b (xi_h,L + xi_h,R): the product with the linear h_b shifts the moments by one
  // (the higher part is held apart: whole minus P1 part would carry the rounding
  // of the whole times g h_b into the higher momentum modes)
  {
    T S[PM + 1];
    sfor<0, PM + 1>([&](auto l) { S[l] = a.x[l] + b.x[l]; });
    sfor<0, PM + 1>([&](auto l) {
      T s1 = 0;
      if constexpr (l > 0) s1 += S[l > 0 ? l - 1 : 0] * (T)((double)l / (2 * l - 1));
      if constexpr (l < PM) s1 += S[l < PM ? l + 1 : 0] * (T)((double)(l + 1) / (2 * l + 3));
      const T hs = (h0 * S[l] + h1 * s1) * (T)(1.0 / (2 * l + 1));
      m1[l] += gnx * hs;
      m2[l] += gny * hs;
    });
  }
  // the base modes' two-point flux: in FP64 with the g xi_lin h_b terms
  T f2[6];
  {
    T q1[2] = {m1[0], m1[1]}, q2[2] = {m2[0], m2[1]};
    if constexpr (!kF32) {
      const T s0 = a.xl[0] + b.xl[0], s1 = a.xl[1] + b.xl[1];
      const T y0 = h0 * s0 + h1 * s1 * (T)(1.0 / 3.0), y1 = (h0 * s1 + h1 * s0) * (T)(1.0 / 3.0);
      q1[0] += gnx * y0; q1[1] += gnx * y1;
      q2[0] += gny * y0; q2[1] += gny * y1;
    }
    const T r3 = (T)1.7320508075688772;  // the points of the two-point rule are +-1 / sqrt 3
    f2[0] = m0[0] - r3 * m0[1]; f2[1] = m0[0] + r3 * m0[1];
    f2[2] = q1[0] - r3 * q1[1]; f2[3] = q1[0] + r3 * q1[1];
    f2[4] = q2[0] - r3 * q2[1]; f2[5] = q2[0] + r3 * q2[1];
    sfor<0, 6>([&](auto i) { fx.Fb[i * nE + ed] = kF32 ? F[i] + (double)f2[i] : (double)f2[i]; });
  }
  if constexpr (kF32) {  // the P1 parts' share of the higher test modes
    T zp[3] = {0, 0, 0};
    add_lin2(z1[0], z1[1], z1[2], a.Ul, a.wl);
    add_lin2(z1[0], z1[1], z1[2], b.Ul, b.wl);
    add_lin2(z2[0], z2[1], z2[2], a.Vl, a.wl);
    add_lin2(z2[0], z2[1], z2[2], b.Vl, b.wl);
    add_lin2(zp[0], zp[1], zp[2], a.xl, a.xl);
    add_lin2(zp[0], zp[1], zp[2], b.xl, b.xl);
    m0[0] += z0[0];
    m0[1] += z0[1];
    sfor<0, 3>([&](auto l) {
      m1[l] += z1[l] + (T)0.5 * gnx * zp[l];
      m2[l] += z2[l] + (T)0.5 * gny * zp[l];
    });
  }
  // moments of h_b times the jump (a quadratic)
  const T mj[3] = {h0 * j0 + h1 * j1 * (T)(1.0 / 3.0), (h0 * j1 + h1 * j0) * (T)(1.0 / 3.0), h1 * j1 * (T)(2.0 / 15.0)};
  // the flux projected onto the higher test modes of each side once here,
  //   P[k][f][q] = -+ (2/s) sum_l cEL[k][q][l] (+-1)^l (m_l +- n_f g mj_l)
  // (left: minus, +J; right: plus, odd l reversed, -J; the 2 undoes the weight
  // |E| / 4), stored in the element's own slot of its order group (local edge
  // k), so that the element kernel reads one value per edge, field and mode,
  // consecutive elements contiguous
  auto project = [&](int side, int64_t el, int k, int pside, T sg) {
    const int Kside = Kof(pside), KH = Kside - 3;
    const int64_t s0 = pside == 2 ? G.start[2] : pside == 3 ? G.start[3] : G.start[4];
    const int64_t ns = (pside == 2 ? G.start[3] : pside == 3 ? G.start[4] : G.start[5]) - s0;
    T* P = (T*)(pside == 2 ? Pf[2] : pside == 3 ? Pf[3] : Pf[4]) + (el - s0);
    const T jx = side ? -gnx : gnx, jy = side ? -gny : gny;
    const T sgo = side ? -sg : sg;
    T y0[PM + 1], y1[PM + 1], y2[PM + 1];
    sfor<0, PM + 1>([&](auto l) {
      const T f = l % 2 ? sgo : sg;
      y0[l] = f * m0[l];
      if constexpr (l < 3) {
        y1[l] = f * (m1[l] + jx * mj[l]);
        y2[l] = f * (m2[l] + jy * mj[l]);
      } else {
        y1[l] = f * m1[l];
        y2[l] = f * m2[l];
      }
    });
    sfor<3, Kof(PM)>([&](auto q) {
      if (q < Kside) {
        T acc[3] = {0, 0, 0};
        sfor<0, deg_of(q) + 1>([&](auto l) {
          const T bq = cEL[k][q][l];
          acc[0] += y0[l] * bq;
          acc[1] += y1[l] * bq;
          acc[2] += y2[l] * bq;
        });
        P[((k * 3 + 0) * KH + (q - 3)) * ns] = acc[0];
        P[((k * 3 + 1) * KH + (q - 3)) * ns] = acc[1];
        P[((k * 3 + 2) * KH + (q - 3)) * ns] = acc[2];
      }
    });
  };
  const T* geo = geo_t(m);
  if (pL >= 2) project(0, L, kL, pL, (T)-2 * geo[G_RS * m.ne + L]);
  if (R >= 0 && pR >= 2) project(1, R, kR, pR, (T)2 * geo[G_RS * m.ne + R]);
}

template <int PM>
__global__ void __launch_bounds__(128) k_edge_corr(DevMesh m, const int32_t* __restrict__ list, int64_t nl, Groups G,
                                                   Phys ph, Stage stg, StateDev c, VelDev u, EdgeFlux fx) {
  edge_corr_body<PM>(m, list, nl, G, ph, stg, c, u, fx);
}

template <int PM>
static int edge_group(cudaStream_t st, const DevMesh& m, const CorrEdges& ce, const Groups& G, const Phys& ph,
                      const Stage& stg, StateDev c, VelDev u, EdgeFlux fx) {
  const int64_t nl = ce.n[PM];
  if (nl == 0) return 0;
  const int ct = spread_threads(nl, launch_shape().corr_threads);
  k_edge_corr<PM><<<nblocks(nl, ct), ct, 0, st>>>(m, ce.list[PM], nl, G, ph, stg, c, u, fx);
  count_launch();
  SWE_CUDA_OK(cudaGetLastError());
  return 0;
}

int launch_edge_corr(GroupStreams gs, const DevMesh& m, const CorrEdges& ce, const Groups& G, const Phys& ph,
                     const Stage& stg, StateDev c, VelDev u, EdgeFlux fx) {
  int r = edge_group<2>(gs.s[0], m, ce, G, ph, stg, c, u, fx);
  if (!r) r = edge_group<3>(gs.s[1], m, ce, G, ph, stg, c, u, fx);
  if (!r) r = edge_group<4>(gs.s[2], m, ce, G, ph, stg, c, u, fx);
  return r;
}


// ---------------------------------------------------------------------------
// correction element update of one order group (K = K(p), p >= 2), test modes
// q >= 3: volume terms, source g grad h_b xi_q, bottom friction and Coriolis, the
// projections of the full edge fluxes (which the correction edge kernel left in
// the element's slots) and the SSP-RK combination.
//
//
// k_elem_corr_split: a block of KL = K(p - 1) warps works on 32 elements, warp m
// forming the products of mode m and, from shared memory, the test modes 3 + m,
// 3 + m + KL, ....  The form of every FP64 group: one FP64 instruction takes a warp
// 64 cycles whatever its parallelism inside the warp and four warps fill an
// SM's pipe (19 cycles each), so what counts is the instruction count and
// that few elements still give every scheduler a warp.  FP64, 165,888 elements
// alone: K = 6, 10, 15 117, 389, 1045 us (GB300), 75 - 85 % of what the pipe
// can issue; the contraction per test mode took about 250, 1260, 4450.
// k_elem_corr (FP32, large groups): one thread per element, each coefficient
// loaded once, the 3 (K - 3) results in registers.  It is straight-line code (55
// KB for K = 15) and waits for instruction fetches: 19, 48, 108 us for 165,888
// elements of K = 6, 10, 15 (the split form 23, 108, 316: ten code bodies at once
// on an SM), but 20 us for 512 of K = 15 (split 11).  The forms cross where the
// split form's threads fill the device about once (n KL = 60,000: K = 15
// between 5,000 and 10,000 elements, K = 10 between 10,000 and 20,000).
// ---------------------------------------------------------------------------
// source, edges and RK combination of one higher test mode: r = volume terms
template <int K>
__device__ __forceinline__ void finish_mode(const Stage& stg, const Phys& ph, int64_t n, int64_t l, int q,
                                            T (&r)[3], T xq, T Uq, T Vq, T uq, T vq, T gdx, T gdy, T tau, T dt,
                                            const T* __restrict__ pe, const T* __restrict__ chN,
                                            T* __restrict__ chO) {
  constexpr int KH = K - 3;
  r[1] = fma(gdx, xq, r[1]);
  r[2] = fma(gdy, xq, r[2]);
  if (ph.src) {
    r[1] += fma((T)ph.f_c, Vq, -(tau * uq));
    r[2] -= fma((T)ph.f_c, Uq, tau * vq);
  }
  const T* P = pe + (q - 3) * n + l;
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int f = 0; f < 3; ++f) r[f] += P[(k * 3 + f) * KH * n];
  const T a = (T)stg.a, b = (T)stg.b;
  const T cs3[3] = {xq, Uq, Vq};
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    const int64_t ix = (f * KH + (q - 3)) * n + l;
    const T y = fma(dt, r[f], cs3[f]);
    chO[ix] = stg.rhs_only ? r[f] : fma(b, y, stg.a != 0.0 ? a * chN[ix] : (T)0);
  }
}

// bottom friction coefficient tau from the element means (Sect. 3), 0 without source terms
__device__ __forceinline__ T friction(const DevMesh& m, const Phys& ph, int64_t e, T rs, T xi0, T u0, T v0) {
  if (!ph.src) return 0;
  const T ra = (T)1.4142135623730951 * rs;
  const T Hm = (xi0 + geo_t(m)[G_HB0 * m.ne + e]) * ra;
  const T um = u0 * ra, vm = v0 * ra;
  return (T)ph.fric_lin * Hm + (T)ph.fric_quad * sqrt(um * um + vm * vm);
}

#define ELEM_CORR_PARAMS                                                                                          \
  DevMesh m, int64_t g0, int64_t n, Phys ph, Stage stg, const T *__restrict__ cbS, const T *__restrict__ chS,       \
      const T *__restrict__ chN, T *__restrict__ chO, const T *__restrict__ ub, const T *__restrict__ uh,           \
      const T *__restrict__ pe

// The factors of D_x and D_s in the three equations (without the 1/s of the
// momentum rows) from mode m's momenta and products.  Spelled out in fma, like the
// sums that use them: a group takes one kernel form or the other by its size,
// and an element's result must not depend on it.
__device__ __forceinline__ void row_factors(T (&x)[3], T (&s)[3], T La, T Lb, T J2, T J3, T U, T V, const T (&z)[4]) {
  x[0] = fma(La, U, Lb * V);
  s[0] = fma(J2, U, J3 * V);
  x[1] = fma(La, z[0], Lb * z[1]);
  s[1] = fma(J2, z[0], J3 * z[1]);
  x[2] = fma(La, z[2], Lb * z[3]);
  s[2] = fma(J2, z[2], J3 * z[3]);
}

template <int K>
__global__ void __launch_bounds__(128, K == 6 ? 5 : K == 10 ? 4 : 3) k_elem_corr(ELEM_CORR_PARAMS) {
  const int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (l >= n) return;
  const int64_t e = g0 + l, ne = m.ne;
  constexpr int KL = Kof(deg_of(K - 1) - 1);
  const T* geo = geo_t(m);
  T xi[K], U[K], V[K], u[K], v[K];
  load_modes<K>(xi, cbS, ne, e, chS, n, l, 0);
  load_modes<K>(U, cbS, ne, e, chS, n, l, 1);
  load_modes<K>(V, cbS, ne, e, chS, n, l, 2);
  load_modes<K>(u, ub, ne, e, uh, n, l, 0);
  load_modes<K>(v, ub, ne, e, uh, n, l, 1);
  const T J2 = geo[G_JI2 * ne + e], J3 = geo[G_JI3 * ne + e];
  const T La = geo[G_JI0 * ne + e] + (T)0.5 * J2, Lb = geo[G_JI1 * ne + e] + (T)0.5 * J3;
  const T rs = geo[G_RS * ne + e], g = (T)ph.g;
  const T xh[3] = {xi[0] + geo[G_HB0 * ne + e], xi[1] + geo[G_HB1 * ne + e], xi[2] + geo[G_HB2 * ne + e]};
  T r[3][K];
  sfor<3, K>([&](auto q) { r[0][q] = r[1][q] = r[2][q] = 0; });
  sfor<0, KL>([&](auto M) {
    T z[4];
    products<K, M>(z, xi, U, V, u, v, xh, g);
    T x[3], s[3];
    row_factors(x, s, La, Lb, J2, J3, U[M], V[M], z);
    sfor<3, K>([&](auto q) {
      sfor<0, 3>([&](auto f) {
        if constexpr (dxnz(q, M)) r[f][q] = fma(cDx[q][M], x[f], r[f][q]);
        if constexpr (dsnz(q, M)) r[f][q] = fma(cDs[q][M], s[f], r[f][q]);
      });
    });
  });
  const T gdx = geo[G_GDHX * ne + e], gdy = geo[G_GDHY * ne + e];
  const T tau = friction(m, ph, e, rs, xi[0], u[0], v[0]);
  const T dt = (T)stage_dt(stg, m.mem[e]);
  sfor<3, K>([&](auto q) {
    T rq[3] = {r[0][q], rs * r[1][q], rs * r[2][q]};
    finish_mode<K>(stg, ph, n, l, q, rq, xi[q], U[q], V[q], u[q], v[q], gdx, gdy, tau, dt, pe, chN, chO);
  });
}

// warp of mode M among W: its own, or for K = 15 on five warps a pair of a long and a short mode
template <int K, int W>
__host__ __device__ constexpr int warp_of(int M) {
  constexpr int five[10] = {0, 4, 1, 1, 4, 2, 3, 0, 2, 3};
  return W == 5 ? five[M] : M;
}

template <int K, int W>
__global__ void __launch_bounds__(32 * W, K == 15 && W == 5 ? 2 : 1) k_elem_corr_split(ELEM_CORR_PARAMS) {
  constexpr int KL = Kof(deg_of(K - 1) - 1), KH = K - 3;
  static_assert(W == KL || (K == 15 && W == 5), "warps of a block");
  __shared__ T B[KL][6][32];  // per mode m: the factors of D_x and D_s in the three equations
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t l = blockIdx.x * (int64_t)32 + lane;
  const bool live = l < n;
  const int64_t e = g0 + (live ? l : 0), ne = m.ne;
  const T* geo = geo_t(m);
  const T rs = geo[G_RS * ne + e];
  if (live) {
    T xi[K], U[K], V[K], u[K], v[K];
    load_modes<K>(xi, cbS, ne, e, chS, n, l, 0);
    load_modes<K>(U, cbS, ne, e, chS, n, l, 1);
    load_modes<K>(V, cbS, ne, e, chS, n, l, 2);
    load_modes<K>(u, ub, ne, e, uh, n, l, 0);
    load_modes<K>(v, ub, ne, e, uh, n, l, 1);
    const T J2 = geo[G_JI2 * ne + e], J3 = geo[G_JI3 * ne + e];
    const T La = geo[G_JI0 * ne + e] + (T)0.5 * J2, Lb = geo[G_JI1 * ne + e] + (T)0.5 * J3;
    const T xh[3] = {xi[0] + geo[G_HB0 * ne + e], xi[1] + geo[G_HB1 * ne + e], xi[2] + geo[G_HB2 * ne + e]};
    sfor<0, KL>([&](auto M) {
      if (w == warp_of<K, W>(M)) {  // uniform over the warp
        T z[4];
        products<K, M>(z, xi, U, V, u, v, xh, (T)ph.g);
        T x[3], s[3];
        row_factors(x, s, La, Lb, J2, J3, U[M], V[M], z);
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          B[M][2 * f][lane] = x[f];
          B[M][2 * f + 1][lane] = s[f];
        }
      }
    });
  }
  __syncthreads();
  if (!live) return;
  const T gdx = geo[G_GDHX * ne + e], gdy = geo[G_GDHY * ne + e];
  const T tau = friction(m, ph, e, rs, cbS[e], ub[e], ub[3 * ne + e]);
  const T dt = (T)stage_dt(stg, m.mem[e]);
  sfor<3, K>([&](auto q) {
    if ((q - 3) % W == w) {  // uniform over the warp
      T r[3];
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        T acc = 0;
        sfor<0, KL>([&](auto M) {
          if constexpr (dxnz(q, M)) acc = fma(cDx[q][M], B[M][2 * f][lane], acc);
          if constexpr (dsnz(q, M)) acc = fma(cDs[q][M], B[M][2 * f + 1][lane], acc);
        });
        r[f] = f == 0 ? acc : rs * acc;
      }
      T uq = 0, vq = 0;
      if (ph.src) {
        uq = uh[(0 * KH + (q - 3)) * n + l];
        vq = uh[(1 * KH + (q - 3)) * n + l];
      }
      finish_mode<K>(stg, ph, n, l, q, r, chS[(0 * KH + (q - 3)) * n + l], chS[(1 * KH + (q - 3)) * n + l],
                     chS[(2 * KH + (q - 3)) * n + l], uq, vq, gdx, gdy, tau, dt, pe, chN, chO);
    }
  });
}

static const T* base_c_host(const StateDev& s) {
  if constexpr (kF32) return (const T*)s.cb32; else return (const T*)s.cb;
}
static const T* base_u_host(const VelDev& u) {
  if constexpr (kF32) return (const T*)u.ub32; else return (const T*)u.ub;
}

template <int K>
static int elem_group(cudaStream_t st, const DevMesh& m, const Groups& G, int p, const Phys& ph, const Stage& stg,
                      StateDev cS, StateDev cN, StateDev cO, VelDev u, EdgeFlux fx) {
  const int64_t g0 = G.start[p], n = G.start[p + 1] - g0;
  if (n == 0) return 0;
  const T *cb = base_c_host(cS), *ub = base_u_host(u), *chS = (const T*)cS.ch[p], *chN = (const T*)cN.ch[p];
  const T *uh = (const T*)u.uh[p], *pe = (const T*)fx.Pf[p];
  T* chO = (T*)cO.ch[p];
  constexpr int KL = Kof(deg_of(K - 1) - 1);
  if (!kF32 || n * KL <= 60000) {
    bool five = false;
    if constexpr (K == 15 && !kF32) {
      five = n > 64 * (int64_t)sm_count();  // two blocks of ten warps per SM and more
      if (five) k_elem_corr_split<K, 5><<<nblocks(n, 32), 160, 0, st>>>(m, g0, n, ph, stg, cb, chS, chN, chO, ub, uh, pe);
    }
    if (!five) k_elem_corr_split<K, KL><<<nblocks(n, 32), 32 * KL, 0, st>>>(m, g0, n, ph, stg, cb, chS, chN, chO, ub, uh, pe);
  } else if constexpr (kF32) {
    const int t = launch_shape().corr_threads;
    k_elem_corr<K><<<nblocks(n, t), t, 0, st>>>(m, g0, n, ph, stg, cb, chS, chN, chO, ub, uh, pe);
  }
  count_launch();
  SWE_CUDA_OK(cudaGetLastError());
  return 0;
}

int launch_elem_corr(GroupStreams gs, const DevMesh& m, const Groups& G, const Phys& ph, const Stage& stg,
                     StateDev cS, StateDev cN, StateDev cO, VelDev u, EdgeFlux fx) {
  int r = elem_group<6>(gs.s[0], m, G, 2, ph, stg, cS, cN, cO, u, fx);
  if constexpr (!on_tc(10)) {
    if (!r) r = elem_group<10>(gs.s[1], m, G, 3, ph, stg, cS, cN, cO, u, fx);
    if (!r) r = elem_group<15>(gs.s[2], m, G, 4, ph, stg, cS, cN, cO, u, fx);
  }
  return r;
}

}  // namespace CORR_NS
}  // namespace swedg
