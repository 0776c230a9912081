// swe_rhs_p1_noalloc: the base right-hand side of an all-P1 mesh with no
// device allocation at all (the paper has no counterpart; see swedg.h).
//
// Some callers cannot allocate device memory: code that runs inside a
// region whose memory is budgeted up front (an embedding application that
// hands the solver fixed buffers and forbids cudaMalloc/cudaFree on its
// streams), or a host process that must not grow its device footprint after
// start-up.  For them the intermediate arrays of this one computation -- the
// auxiliary velocity u and the moments of every edge's Lax-Friedrichs flux --
// live in file-scope __device__ arrays of fixed size, g_na_scratch and g_na_ok,
// which every GPU that loads the library holds until the process exits.  The caller passes inputs and outputs; nothing else is
// allocated, by this file or by any library it calls.
//
// Sect. 2-3 of the paper for p = 1 with land walls, in the vertex values of the
// linear fields (equal to the modal form in exact arithmetic): with every
// quantity at the vertices the traces on an edge are its two ends' values, the
// element's gradients and the edge normals are coordinate differences, and
// the areas cancel, so that the only square roots are one per element (the scale
// of its orthonormal basis) and one per edge (lambda), and there is no division
// but the solve's.  FP64 instructions bound these kernels (GB300: 19 cycles of
// an SM each, 64 of the warp): about 95 per element in k_na_usolve, 106 per edge,
// 130 per element in k_na_elem, where the modal form with its geometry formed at
// every visit took 1,900 per element; 72 -> 42 us for 20,000 elements (GB300).
#include <cuda.h>

#include <cmath>
#include <mutex>

#include "../../include/swedg.h"
#include "common.h"

namespace swedg {
namespace na {

constexpr int64_t NMAX = SWE_NOALLOC_MAX_ELEMENTS;
// per element: u, v at the three vertices, then the edge flux's moments
// [3 fields][2 ends][3 local edges]
constexpr int64_t PER_ELEM = 6 + 18;
static __device__ __align__(256) double g_na_scratch[PER_ELEM * NMAX];
static __device__ __align__(256) unsigned char g_na_ok[NMAX];  // 1: a usable element (see elem_ok)

// Set-up once per device context (with that device current): the device
// addresses of the scratch arrays.  The context is identified by its driver
// id, so a context re-created after cudaDeviceReset is set up again; a mutex
// serialises the set-up of host threads that call at the same time.
struct Scratch {
  double* v = nullptr;
  unsigned char* ok = nullptr;
};
struct DevState {
  bool ready = false;
  unsigned long long ctx_id = 0;
  Scratch scratch;
};
static DevState g_dev[64];
static std::mutex g_setup_mutex;

typedef CUresult (*PFN_ctxGetCurrent)(CUcontext*);
typedef CUresult (*PFN_ctxGetId)(CUcontext, unsigned long long*);

// driver id of the current context, 0 when there is none (or no driver entry)
static unsigned long long current_ctx_id() {
  static PFN_ctxGetCurrent get_current = nullptr;
  static PFN_ctxGetId get_id = nullptr;
  static bool looked_up = false;
  if (!looked_up) {
    void* f1 = nullptr;
    void* f2 = nullptr;
    cudaDriverEntryPointQueryResult q1, q2;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f1, 12000, cudaEnableDefault, &q1) == cudaSuccess &&
        cudaGetDriverEntryPointByVersion("cuCtxGetId", &f2, 12000, cudaEnableDefault, &q2) == cudaSuccess &&
        q1 == cudaDriverEntryPointSuccess && q2 == cudaDriverEntryPointSuccess) {
      get_current = (PFN_ctxGetCurrent)f1;
      get_id = (PFN_ctxGetId)f2;
    }
    looked_up = true;
  }
  if (!get_current || !get_id) return 0;
  CUcontext ctx = nullptr;
  unsigned long long id = 0;
  if (get_current(&ctx) != CUDA_SUCCESS || ctx == nullptr || get_id(ctx, &id) != CUDA_SUCCESS) return 0;
  return id;
}

static int setup(int dev, Scratch* scratch) {
  if (dev < 0 || dev >= 64) return SWE_EINVAL;
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  const unsigned long long id0 = current_ctx_id();
  if (g_dev[dev].ready && id0 != 0 && id0 == g_dev[dev].ctx_id) {
    *scratch = g_dev[dev].scratch;
    return 0;
  }
  // the symbol lookup also makes the device's primary context current
  void *p = nullptr, *q = nullptr;
  g_dev[dev].ready = false;
  if (cudaGetSymbolAddress(&p, g_na_scratch) != cudaSuccess || p == nullptr) return SWE_ECUDA;
  if (cudaGetSymbolAddress(&q, g_na_ok) != cudaSuccess || q == nullptr) return SWE_ECUDA;
  g_dev[dev].scratch.v = (double*)p;
  g_dev[dev].scratch.ok = (unsigned char*)q;
  g_dev[dev].ctx_id = current_ctx_id();
  g_dev[dev].ready = true;
  *scratch = g_dev[dev].scratch;
  return 0;
}

struct P2 {
  double x, y;
};

__device__ __forceinline__ P2 vertex(const double* __restrict__ xy, int64_t v) {
  return P2{xy[2 * v], xy[2 * v + 1]};  // 8-byte loads: the caller's array may start anywhere
}

// An element is used only when its vertex ids lie in [0, nv) and it is
// counter-clockwise with positive area (det J_e > 0); any other element gets
// NaN rows and is a land edge to its neighbours.
__device__ __forceinline__ bool elem_ok(const double* __restrict__ xy, const int32_t (&v)[3], int64_t nv, double& det) {
  if (!(v[0] >= 0 && v[1] >= 0 && v[2] >= 0 && v[0] < nv && v[1] < nv && v[2] < nv)) return false;
  const P2 a = vertex(xy, v[0]), b = vertex(xy, v[1]), c = vertex(xy, v[2]);
  det = (b.x - a.x) * (c.y - a.y) - (c.x - a.x) * (b.y - a.y);
  return det > 0.0;
}

// The element across local edge k of e, with e's local edge number kn in the
// neighbour's list, or -1 (land): a neighbour id outside [0, ne), an unusable
// neighbour, or one whose own list does not name e.  Both the edge and the
// element kernel decide through this one function, so every flux slot an
// element reads was written by the same call.
__device__ __forceinline__ int64_t mutual_nbr(const int32_t* __restrict__ nbr, const unsigned char* __restrict__ ok,
                                              int64_t ne, int64_t e, int k, int& kn) {
  const int64_t n = nbr[3 * e + k];
  if (n < 0 || n >= ne || n == e || !ok[n]) return -1;
  for (int j = 0; j < 3; ++j)
    if (nbr[3 * n + j] == e) { kn = j; return n; }
  return -1;
}

// The degree-1 modes at the vertices are (sqrt 2, -+sqrt 12, -2), (.., +sqrt 12,
// -2), (sqrt 2, 0, 4) over s = sqrt det: vertex values of one field's modes.
constexpr double kR2 = 1.4142135623730951, kR12 = 3.4641016151377544;
__device__ __forceinline__ void to_vertices(const double* c, int64_t ne, double rs, double (&n)[3]) {
  const double c2 = (2.0 * rs) * c[2 * ne], c1 = (kR12 * rs) * c[ne];
  const double a = (kR2 * rs) * c[0], b = a - c2;
  n[0] = b - c1;
  n[1] = b + c1;
  n[2] = fma(2.0, c2, a);
}

// The element's fields at its vertices, into rhs (the caller's output array serves
// as their buffer until k_na_elem overwrites it; a call with rhs == c works
// too, k_na_elem reads nothing else of c), and the auxiliary system of Sect. 3:
// sum_k u_k int H lambda_j lambda_k = int U lambda_j with H linear, a 3 x 3
// symmetric system with entries 2 S + 4 H_j and 2 S - H_l (times det / 120) for
// S = H_0 + H_1 + H_2, solved with its adjugate.
__global__ void __launch_bounds__(64) k_na_usolve(int64_t nv, int64_t ne, const double* __restrict__ xy,
                                                  const double* __restrict__ hv, const int32_t* __restrict__ tri,
                                                  const double* c, double* rhs, double* __restrict__ scr,
                                                  unsigned char* __restrict__ ok) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= ne) return;
  const int32_t v[3] = {tri[3 * e], tri[3 * e + 1], tri[3 * e + 2]};
  double det = 0.0;
  const bool good = elem_ok(xy, v, nv, det);
  ok[e] = good;
  if (!good) return;
  const double rs = rsqrt(det);
  double f[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i) to_vertices(c + 3 * i * ne + e, ne, rs, f[i]);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) rhs[(3 * i + j) * ne + e] = f[i][j];
  const double H0 = hv[v[0]] + f[0][0], H1 = hv[v[1]] + f[0][1], H2 = hv[v[2]] + f[0][2];
  const double S2 = 2.0 * (H0 + H1 + H2);
  const double a = fma(4.0, H0, S2), d = fma(4.0, H1, S2), h = fma(4.0, H2, S2);
  const double b = S2 - H2, cc = S2 - H1, g = S2 - H0;  // entries (0,1), (0,2), (1,2)
  const double C00 = d * h - g * g, C01 = cc * g - b * h, C02 = b * g - cc * d;
  const double C11 = a * h - cc * cc, C12 = b * cc - a * g, C22 = a * d - b * b;
  const double r = 5.0 / (a * C00 + b * C01 + cc * C02);
#pragma unroll
  for (int i = 1; i < 3; ++i) {  // int U lambda_j = det / 24 (U_0 + U_1 + U_2 + U_j)
    const double s = f[i][0] + f[i][1] + f[i][2];
    const double b0 = (s + f[i][0]) * r, b1 = (s + f[i][1]) * r, b2 = (s + f[i][2]) * r;
    scr[(3 * (i - 1) + 0) * NMAX + e] = C00 * b0 + C01 * b1 + C02 * b2;
    scr[(3 * (i - 1) + 1) * NMAX + e] = C01 * b0 + C11 * b1 + C12 * b2;
    scr[(3 * (i - 1) + 2) * NMAX + e] = C02 * b0 + C12 * b1 + C22 * b2;
  }
}

// One side of an edge: xi, U, V, w = u.N at its two ends A, B (N the scaled
// normal), and the element means of w and xi.
struct Side {
  double x[2], U[2], V[2], w[2], wm, xm;
};
__device__ __forceinline__ Side side(const double* f, const double* __restrict__ scr, int64_t ne, int64_t e, int ia,
                                     int ib, int ic, double Nx, double Ny) {
  Side s;
  const int i[2] = {ia, ib};
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    s.x[a] = f[i[a] * ne + e];
    s.U[a] = f[(3 + i[a]) * ne + e];
    s.V[a] = f[(6 + i[a]) * ne + e];
    s.w[a] = scr[i[a] * NMAX + e] * Nx + scr[(3 + i[a]) * NMAX + e] * Ny;
  }
  const double wc = scr[ic * NMAX + e] * Nx + scr[(3 + ic) * NMAX + e] * Ny;
  s.wm = (s.w[0] + s.w[1] + wc) * (1.0 / 3.0);
  s.xm = (s.x[0] + s.x[1] + f[ic * ne + e]) * (1.0 / 3.0);
  return s;
}

// LF flux (Sect. 2) of every edge, as its moments with the two linear functions
// that are 1 at one end: for products of two linear functions a b these are
// |E| / 12 (2 a_A b_A + (a_A + a_B)(b_A + b_B)) and alike for B, for a linear F
// |E| / 6 (2 F_A + F_B); a half of each is taken for the flux average.  Stored
// once in the slot of the lower-numbered element.  A block takes the 3 ET edges
// of ET elements and first packs those it owns (half of them on average): an
// FP64 instruction takes its 64 cycles for one active lane as for 32.
constexpr int ET = 40, BT = 64;
__global__ void __launch_bounds__(BT) k_na_edge(int64_t ne, const double* __restrict__ xy,
                                                const double* __restrict__ hv, const int32_t* __restrict__ tri,
                                                const int32_t* __restrict__ nbr, const double* f, double g,
                                                double* __restrict__ scr, const unsigned char* __restrict__ ok) {
  __shared__ int32_t own[3 * ET], own_n[3 * ET];  // local edge of the block << 2 | neighbour's local edge; neighbour
  __shared__ int count[(3 * ET + 31) / 32 + 1];
  const int64_t e0 = blockIdx.x * (int64_t)ET;
  const int lane = threadIdx.x & 31;
  constexpr int NC = (3 * ET + BT - 1) / BT;
  int kn[NC], mine[NC], rank[NC];
  int64_t nn[NC];
#pragma unroll
  for (int r = 0; r < NC; ++r) {
    const int t = r * BT + threadIdx.x;
    const int64_t e = e0 + t / 3;
    kn[r] = 0;
    nn[r] = -1;
    mine[r] = 0;
    if (t < 3 * ET && e < ne && ok[e]) {
      nn[r] = mutual_nbr(nbr, ok, ne, e, t % 3, kn[r]);
      mine[r] = nn[r] < 0 || nn[r] > e;  // else owned by the neighbour
    }
    const unsigned m = __ballot_sync(0xffffffffu, mine[r]);
    rank[r] = __popc(m & ((1u << lane) - 1u));
    if (lane == 0 && t / 32 < (3 * ET + 31) / 32) count[t / 32] = __popc(m);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int s = 0;
    for (int i = 0; i < (3 * ET + 31) / 32; ++i) {
      const int x = count[i];
      count[i] = s;
      s += x;
    }
    count[(3 * ET + 31) / 32] = s;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < NC; ++r)
    if (mine[r]) {
      const int t = r * BT + threadIdx.x, p = count[t / 32] + rank[r];
      own[p] = t << 2 | kn[r];
      own_n[p] = (int32_t)nn[r];
    }
  __syncthreads();
  const int total = count[(3 * ET + 31) / 32];
  for (int p = threadIdx.x; p < total; p += BT) {
    const int t = own[p] >> 2, kr = own[p] & 3, k = t % 3;
    const int64_t e = e0 + t / 3, n = own_n[p];
    const int ia = k == 2 ? 0 : k + 1, ib = k == 0 ? 2 : k - 1;
    const int32_t va = tri[3 * e + ia], vb = tri[3 * e + ib];
    const P2 A = vertex(xy, va), B = vertex(xy, vb);
    // |E| / 24 times the unit normal carries the weights of the momentum rows
    const double Nx = (B.y - A.y) * (1.0 / 24.0), Ny = (A.x - B.x) * (1.0 / 24.0);
    const double hA = hv[va], hB = hv[vb], hm = 0.5 * (hA + hB), N2 = Nx * Nx + Ny * Ny;
    Side a = side(f, scr, ne, e, ia, ib, k, Nx, Ny), b;
    if (n >= 0) {  // the neighbour runs the edge the other way
      b = side(f, scr, ne, n, kr == 0 ? 2 : kr - 1, kr == 2 ? 0 : kr + 1, kr, Nx, Ny);
    } else {  // land: mirror state
      const double r = 2.0 / N2;
      b = a;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const double qn = (a.U[q] * Nx + a.V[q] * Ny) * r;
        b.U[q] = a.U[q] - qn * Nx;
        b.V[q] = a.V[q] - qn * Ny;
        b.w[q] = -a.w[q];
      }
      b.wm = -a.wm;
    }
    const double lam = fmax(fabs(a.wm), fabs(b.wm)) + sqrt(N2 * (g * (fmax(a.xm, b.xm) + hm)));
    double* F = scr + 6 * NMAX + e;
    // elevation row: linear
    double FA = (a.U[0] + b.U[0]) * Nx + (a.V[0] + b.V[0]) * Ny + lam * (a.x[0] - b.x[0]);
    double FB = (a.U[1] + b.U[1]) * Nx + (a.V[1] + b.V[1]) * Ny + lam * (a.x[1] - b.x[1]);
    F[(0 * 3 + k) * NMAX] = 2.0 * fma(2.0, FA, FB);
    F[(1 * 3 + k) * NMAX] = 2.0 * fma(2.0, FB, FA);
    // momentum rows: U w + U+ w+ + (P + P+) N, and lambda (U - U+) as a linear
    // term: w +- lambda in the products would drop the low bits of w, which is
    // orders of magnitude below lambda (40 us instead of 42, and noise of
    // lambda |U| instead of |w U| in the momentum rows)
    const double lam2 = 2.0 * lam;
    const double UA = a.U[0] - b.U[0], UB = a.U[1] - b.U[1], VA = a.V[0] - b.V[0], VB = a.V[1] - b.V[1];
    const double wa = a.w[0] + a.w[1], wb = b.w[0] + b.w[1];
    const double xa = a.x[0] + a.x[1], xb = b.x[0] + b.x[1];
    const double gNx = g * Nx, gNy = g * Ny, hs = hA + hB;
    const double PA = a.x[0] * fma(0.5, a.x[0], hA) + b.x[0] * fma(0.5, b.x[0], hA);
    const double PB = a.x[1] * fma(0.5, a.x[1], hB) + b.x[1] * fma(0.5, b.x[1], hB);
    const double PS = xa * fma(0.5, xa, hs) + xb * fma(0.5, xb, hs);
    const double XA = a.U[0] * a.w[0] + b.U[0] * b.w[0] + PA * gNx, XB = a.U[1] * a.w[1] + b.U[1] * b.w[1] + PB * gNx;
    const double XS = (a.U[0] + a.U[1]) * wa + (b.U[0] + b.U[1]) * wb + PS * gNx;
    F[(2 * 3 + k) * NMAX] = fma(lam2, fma(2.0, UA, UB), fma(2.0, XA, XS));
    F[(3 * 3 + k) * NMAX] = fma(lam2, fma(2.0, UB, UA), fma(2.0, XB, XS));
    const double YA = a.V[0] * a.w[0] + b.V[0] * b.w[0] + PA * gNy, YB = a.V[1] * a.w[1] + b.V[1] * b.w[1] + PB * gNy;
    const double YS = (a.V[0] + a.V[1]) * wa + (b.V[0] + b.V[1]) * wb + PS * gNy;
    F[(4 * 3 + k) * NMAX] = fma(lam2, fma(2.0, VA, VB), fma(2.0, YA, YS));
    F[(5 * 3 + k) * NMAX] = fma(lam2, fma(2.0, VB, VA), fma(2.0, YB, YS));
  }
}

// Volume, source and edge terms as loads R_j = (.., lambda_j) at the vertices, then
// the modal rows sum_j phi_q(v_j) R_j.  With d_j = det grad lambda_j (coordinate
// differences) and the vertex sums the areas cancel: int a b = det / 24
// (sum a sum b + sum a_j b_j), grad h_b = sum h_j d_j / det.
__global__ void __launch_bounds__(64) k_na_elem(int64_t ne, const double* __restrict__ xy,
                                                const double* __restrict__ hv, const int32_t* __restrict__ tri,
                                                const int32_t* __restrict__ nbr, double g,
                                                const double* __restrict__ scr, const unsigned char* __restrict__ ok,
                                                double* rhs) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= ne) return;
  if (!ok[e]) {  // unusable element: NaN rows, nothing read
    for (int i = 0; i < 9; ++i) rhs[i * ne + e] = __longlong_as_double(0x7ff8000000000000LL);
    return;
  }
  const int32_t v[3] = {tri[3 * e], tri[3 * e + 1], tri[3 * e + 2]};
  const P2 p[3] = {vertex(xy, v[0]), vertex(xy, v[1]), vertex(xy, v[2])};
  const double dx[3] = {p[1].y - p[2].y, p[2].y - p[0].y, p[0].y - p[1].y};
  const double dy[3] = {p[2].x - p[1].x, p[0].x - p[2].x, p[1].x - p[0].x};
  const double h[3] = {hv[v[0]], hv[v[1]], hv[v[2]]};
  double f[3][3], u[2][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) f[i][j] = rhs[(3 * i + j) * ne + e];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) u[i][j] = scr[(3 * i + j) * NMAX + e];
  // the edges' moments, collected at the vertices (- for the flux's own direction)
  double R[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    int kn = 0;
    const int64_t n = mutual_nbr(nbr, ok, ne, e, k, kn);
    const bool right = n >= 0 && n < e;  // the flux is stored by the neighbour, in its direction
    const double* F = scr + 6 * NMAX + (right ? n : e);
    const int ko = right ? kn : k;
    const unsigned long long neg = right ? 0ull : 0x8000000000000000ull;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double a = F[((2 * i + (right ? 1 : 0)) * 3 + ko) * NMAX], b = F[((2 * i + (right ? 0 : 1)) * 3 + ko) * NMAX];
      R[i][(k + 1) % 3] += __longlong_as_double(__double_as_longlong(a) ^ neg);
      R[i][(k + 2) % 3] += __longlong_as_double(__double_as_longlong(b) ^ neg);
    }
  }
  const double xs = f[0][0] + f[0][1] + f[0][2], Us = f[1][0] + f[1][1] + f[1][2], Vs = f[2][0] + f[2][1] + f[2][2];
  const double us = u[0][0] + u[0][1] + u[0][2], vs = u[1][0] + u[1][1] + u[1][2];
  double Axx = Us * us, Axy = Us * vs, Ayx = Vs * us, Ayy = Vs * vs;
  double q[3], P = 0.0;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    Axx += f[1][j] * u[0][j]; Axy += f[1][j] * u[1][j];
    Ayx += f[2][j] * u[0][j]; Ayy += f[2][j] * u[1][j];
    q[j] = fma(0.5, f[0][j], h[j]);
    P += f[0][j] * q[j];
  }
  P = g * fma(xs, q[0] + q[1] + q[2], P);
  constexpr double r24 = 1.0 / 24.0;
  Axx = (Axx + P) * r24; Axy *= r24; Ayx *= r24; Ayy = (Ayy + P) * r24;
  const double g24 = g * r24, hx = g24 * (h[0] * dx[0] + h[1] * dx[1] + h[2] * dx[2]);
  const double hy = g24 * (h[0] * dy[0] + h[1] * dy[1] + h[2] * dy[2]);
  const double U6 = Us * (1.0 / 6.0), V6 = Vs * (1.0 / 6.0);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const double xj = xs + f[0][j];
    R[0][j] += dx[j] * U6 + dy[j] * V6;
    R[1][j] += dx[j] * Axx + dy[j] * Axy + hx * xj;
    R[2][j] += dx[j] * Ayx + dy[j] * Ayy + hy * xj;
  }
  const double det = dy[2] * dx[1] - dy[1] * dx[2];
  const double rs = rsqrt(det), t0 = kR2 * rs, t1 = kR12 * rs, t2 = 2.0 * rs;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const double s = R[i][0] + R[i][1];
    rhs[(3 * i + 0) * ne + e] = t0 * (s + R[i][2]);
    rhs[(3 * i + 1) * ne + e] = t1 * (R[i][1] - R[i][0]);
    rhs[(3 * i + 2) * ne + e] = t2 * fma(2.0, R[i][2], -s);
  }
}

}  // namespace na
}  // namespace swedg

using namespace swedg;

extern "C" int swe_rhs_p1_noalloc(int64_t nv, const double* xy, const double* hv, int64_t ne, const int32_t* tri,
                                  const int32_t* nbr, const double* c, double g, double* rhs_out, void* stream) {
  if (ne < 1 || ne > na::NMAX || nv < 3 || !xy || !hv || !tri || !nbr || !c || !rhs_out || !(g > 0.0) ||
      !(g < INFINITY))
    return SWE_EINVAL;
  // an error left by earlier work on this thread is reported, not mistaken for ours later
  if (cudaGetLastError() != cudaSuccess) return SWE_ECUDA;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return SWE_ECUDA;
  na::Scratch scr;
  const int rc = na::setup(dev, &scr);
  if (rc) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  const int T = 64;
  const unsigned nb = (unsigned)((ne + T - 1) / T);
  na::k_na_usolve<<<nb, T, 0, s>>>(nv, ne, xy, hv, tri, c, rhs_out, scr.v, scr.ok);
  if (cudaGetLastError() != cudaSuccess) return SWE_ECUDA;
  na::k_na_edge<<<(unsigned)((ne + na::ET - 1) / na::ET), na::BT, 0, s>>>(ne, xy, hv, tri, nbr, rhs_out, g, scr.v, scr.ok);
  if (cudaGetLastError() != cudaSuccess) return SWE_ECUDA;
  na::k_na_elem<<<nb, T, 0, s>>>(ne, xy, hv, tri, nbr, g, scr.v, scr.ok, rhs_out);
  return cudaGetLastError() == cudaSuccess ? 0 : SWE_ECUDA;
}
