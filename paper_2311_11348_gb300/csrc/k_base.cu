// Base part of the order-separated scheme (Sect. 3): every term whose test
// index and coefficient indices are modes of degree <= 1, on every element,
// in FP64.  Plus the layout conversions, the CFL reduction, the time update
// and the diagnostics.
//
// Kernels (one thread per element or per edge, on few elements a warp per field; FP64-pipe bound on GB300):
//   k_usolve_base  auxiliary system uH = q (Sect. 3) for p <= 1 elements
//                  (and, in the first stage of a step, the CFL bounds of its
//                  elements: min over elements, exact, order independent)
//   k_edge_base    Lax-Friedrichs flux (Sect. 2) of the P1 traces at the two
//                  Gauss points of the edges between elements of order <= 1,
//                  lambda of Eq. (10) from means
//   k_elem_base    volume + source terms (Eq. 13 with the degree-1 tensors in
//                  closed form), edge projections, rc and the SSP-RK stage
//                  combination of the base modes
#include <cfloat>

#include "base_edge.cuh"
#include "kernels.h"
#include "tables.h"


namespace swedg {

__constant__ double cTs[2];  // T[1][1][2] and T[2][2][2] over phihat_1

void upload_base_tables() {
  const RefTables& R = tables();
  const double Ts[2] = {R.T[1][1][2] / R.phi0, R.T[2][2][2] / R.phi0};
  cudaMemcpyToSymbol(cTs, Ts, sizeof Ts);
}

static inline int nblocks(int64_t n, int t) { return (int)((n + t - 1) / t); }

static int g_sm_count = 152;
void set_sm_count(int n) { g_sm_count = n > 0 ? n : 152; }
int sm_count() { return g_sm_count; }

// Threads per block of a kernel over n units: t, halved (down to a warp) while the
// blocks would not cover the SMs twice.  An FP64 instruction takes a warp 64 cycles and
// its SM 19, so four warps in one block run a kernel of few units at half
// the speed of the same four on four SMs.
int spread_threads(int64_t n, int t) {
  while (t > 32 && nblocks(n, t) < 2 * g_sm_count) t = (t / 2 + 31) / 32 * 32;
  return t;
}

// Grid of the FP64-pipe-bound base kernels.  `per_sm` > 0 resident blocks per SM
// once the work is more than one unit per thread of that grid: a few warps
// per SM keep the FP64 pipe busy, and the rest of the SM stays free for the
// concurrent FP32 correction.
struct BaseGrid {
  int blocks, threads, chunk;
};
static BaseGrid base_grid(int64_t n, const LaunchShape& L) {
  const int64_t blocks = (int64_t)g_sm_count * L.base_bpsm, threads = blocks * L.base_threads;
  if (L.base_bpsm <= 0 || n <= threads) {
    const int t = spread_threads(n, L.base_threads);
    return {nblocks(n, t), t, 0};
  }
  // tiles of chunk * threads units, smaller ones where a block would take less than four
  int c = L.base_chunk;
  while (c > 1 && n < 4 * c * threads) c /= 2;
  return {(int)blocks, L.base_threads, c};
}

template <typename T>
__device__ __forceinline__ T* chp(void* p) { return reinterpret_cast<T*>(p); }

// Work distribution of the base kernels over n units (edges or elements).
// chunk == 0 or work == nullptr: equal grid-stride shares.  Otherwise every block
// takes tiles of chunk * blockDim.x consecutive units from an atomic ticket
// counter (work[0]) until none are left -- the next ticket is fetched while the
// current tile runs -- so a block on an SM that the concurrent correction
// kernels keep busy simply takes fewer tiles; the last block to finish (counted
// in work[1]) resets both counters for the next launch on the stream.  Every unit is
// computed by one thread with the same arithmetic whatever the schedule, so
// results do not depend on it.
template <typename F>
__device__ __forceinline__ void for_units(int64_t n, int chunk, unsigned* work, F&& f) {
  const bool dyn = chunk > 0 && work != nullptr;
  __shared__ unsigned s_ticket;
  const int64_t tile = dyn ? (int64_t)chunk * blockDim.x : (int64_t)gridDim.x * blockDim.x;
  const int64_t ntiles = (n + tile - 1) / tile;
  // static: tile t is the t-th grid-wide stride, every block takes each t
  // with its own offset blockIdx.x * blockDim.x; dynamic: tile t is chunk *
  // blockDim.x consecutive units, taken from the ticket counter
  int64_t t = 0;
  if (dyn) {
    if (threadIdx.x == 0) s_ticket = atomicAdd(work, 1u);
    __syncthreads();
    t = s_ticket;
  }
  const int64_t off = dyn ? threadIdx.x : blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int per = dyn ? chunk : 1;
#pragma unroll 1
  while (t < ntiles) {
    if (dyn) {
      __syncthreads();  // every thread has read the ticket
      if (threadIdx.x == 0) s_ticket = atomicAdd(work, 1u);
    }
    const int64_t base = t * tile + off;
#pragma unroll 1
    for (int k = 0; k < per; ++k) {
      const int64_t i = base + (int64_t)k * blockDim.x;
      if (i < n) f(i);
    }
    if (dyn) {
      __syncthreads();  // the next ticket has arrived
      t = s_ticket;
    } else {
      ++t;
    }
  }
  if (dyn && threadIdx.x == 0) {
    // this block takes no more tickets; the last one out resets the counters
    __threadfence();
    if (atomicAdd(work + 1, 1u) == gridDim.x - 1) {
      work[0] = 0u;
      work[1] = 0u;
      __threadfence();
    }
  }
}

// ---------------------------------------------------------------------------
// layout conversion: caller layout <-> internal state.  Caller layouts: the
// full c[3][15][ne_user] (off == nullptr), or packed element by element,
// element u's 3 K(p_u) values (field-major) from off[u] (modes < K(p_u) only).
// One thread per element in the caller's order: the caller's side, the larger
// one, is then read and written in whole lines, and neighbours of one order
// are neighbours in the internal order too.  The packed layout goes through
// shared memory, a block's elements being one contiguous piece of it.  (One thread
// per internal element left a sector of the caller's array to up to four
// warps: 765 us out and 295 us in for 2,097,152 elements in the full layout.)
// ---------------------------------------------------------------------------
constexpr int LT = 64;  // elements per block of the packed conversions (23 KB of shared memory)

// the state value of (internal element e of order p, field f, mode i < K(p)), as a reference
template <typename TC>
struct StateAt {
  const StateDev& st;
  TC* h;
  int64_t ne, e, n, l;
  int K;
  __device__ __forceinline__ StateAt(const StateDev& s, const Groups& G, int64_t ne_, int64_t e_, int p)
      : st(s), h(nullptr), ne(ne_), e(e_), n(0), l(0), K(Kof(p)) {
    if (p >= 2) {  // selects, not a runtime index into the parameter arrays
      const int64_t a = p == 2 ? G.start[2] : p == 3 ? G.start[3] : G.start[4];
      n = (p == 2 ? G.start[3] : p == 3 ? G.start[4] : G.start[5]) - a;
      l = e - a;
      h = reinterpret_cast<TC*>(p == 2 ? s.ch[2] : p == 3 ? s.ch[3] : s.ch[4]);
    }
  }
  __device__ __forceinline__ double get(int f, int i) const {
    return i < 3 ? st.cb[(f * 3 + i) * ne + e] : (double)h[(f * (K - 3) + (i - 3)) * n + l];
  }
  __device__ __forceinline__ void put(int f, int i, double v) const {
    if (i < 3) {
      st.cb[(f * 3 + i) * ne + e] = v;
      if (st.cb32) st.cb32[(f * 3 + i) * ne + e] = (float)v;
    } else {
      h[(f * (K - 3) + (i - 3)) * n + l] = (TC)v;
    }
  }
};

template <typename TC>
__global__ void k_from_user(DevMesh m, Groups G, const int32_t* __restrict__ inv, const double* __restrict__ cu,
                            StateDev st) {
  const int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (u >= m.ne) return;
  const int64_t e = inv[u];
  const StateAt<TC> S(st, G, m.ne, e, m.p[e]);
#pragma unroll
  for (int f = 0; f < 3; ++f)
#pragma unroll
    for (int i = 0; i < KMAX; ++i) {
      if (i < S.K) S.put(f, i, cu[(f * KMAX + i) * m.ne + u]);
      else if (i < 3) S.put(f, i, 0.0);
    }
}

template <typename TC>
__global__ void k_to_user(DevMesh m, Groups G, const int32_t* __restrict__ inv, StateDev st,
                          double* __restrict__ cu) {
  const int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (u >= m.ne) return;
  const int64_t e = inv[u];
  const StateAt<TC> S(st, G, m.ne, e, m.p[e]);
#pragma unroll
  for (int f = 0; f < 3; ++f)
#pragma unroll
    for (int i = 0; i < KMAX; ++i) cu[(f * KMAX + i) * m.ne + u] = i < S.K ? S.get(f, i) : 0.0;
}

template <typename TC>
__global__ void __launch_bounds__(LT) k_from_packed(DevMesh m, Groups G, const int32_t* __restrict__ inv,
                                                    const int64_t* __restrict__ off, int64_t total,
                                                    const double* __restrict__ cu, StateDev st) {
  __shared__ double buf[LT * 3 * KMAX];
  const int64_t u0 = blockIdx.x * (int64_t)LT, u1 = min(u0 + LT, m.ne), u = u0 + threadIdx.x;
  const int64_t a = off[u0], len = (u1 < m.ne ? off[u1] : total) - a;
#pragma unroll 1
  for (int64_t j = threadIdx.x; j < len; j += 9 * LT) {  // nine loads in flight per thread
    double t[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) t[k] = j + k * LT < len ? cu[a + j + k * LT] : 0.0;
#pragma unroll
    for (int k = 0; k < 9; ++k)
      if (j + k * LT < len) buf[j + k * LT] = t[k];
  }
  __syncthreads();
  if (u >= m.ne) return;
  const int64_t e = inv[u];
  const StateAt<TC> S(st, G, m.ne, e, m.p[e]);
  const double* x = buf + (off[u] - a);
#pragma unroll
  for (int f = 0; f < 3; ++f)
#pragma unroll
    for (int i = 0; i < KMAX; ++i) {
      if (i < S.K) S.put(f, i, x[f * S.K + i]);
      else if (i < 3) S.put(f, i, 0.0);
    }
}

template <typename TC>
__global__ void __launch_bounds__(LT) k_to_packed(DevMesh m, Groups G, const int32_t* __restrict__ inv,
                                                  const int64_t* __restrict__ off, int64_t total, StateDev st,
                                                  double* __restrict__ cu) {
  __shared__ double buf[LT * 3 * KMAX];
  const int64_t u0 = blockIdx.x * (int64_t)LT, u1 = min(u0 + LT, m.ne), u = u0 + threadIdx.x;
  const int64_t a = off[u0], len = (u1 < m.ne ? off[u1] : total) - a;
  if (u < m.ne) {
    const int64_t e = inv[u];
    const StateAt<TC> S(st, G, m.ne, e, m.p[e]);
    double* x = buf + (off[u] - a);
#pragma unroll
    for (int f = 0; f < 3; ++f) {  // a field's loads together, then its stores
      double v[KMAX];
#pragma unroll
      for (int i = 0; i < KMAX; ++i) v[i] = i < S.K ? S.get(f, i) : 0.0;
#pragma unroll
      for (int i = 0; i < KMAX; ++i)
        if (i < S.K) x[f * S.K + i] = v[i];
    }
  }
  __syncthreads();
  for (int64_t j = threadIdx.x; j < len; j += LT) cu[a + j] = buf[j];
}

__global__ void k_sub(const double* __restrict__ a, const double* __restrict__ b, double* __restrict__ out,
                      int64_t n) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) out[i] = a[i] - b[i];
}

int launch_sub(cudaStream_t s, const double* a, const double* b, double* out, int64_t n) {
  if (n == 0) return 0;
  k_sub<<<nblocks(n, 256), 256, 0, s>>>(a, b, out, n);
  count_launch();
  SWE_CUDA_OK(cudaGetLastError());
  return 0;
}

int launch_from_user(cudaStream_t s, const DevMesh& m, const Groups& G, const int32_t* inv, const int64_t* off,
                     int64_t packed_n, int corr_fp32, const double* cu, StateDev st) {
  if (m.ne == 0) return 0;
  if (off) {
    if (corr_fp32) k_from_packed<float><<<nblocks(m.ne, LT), LT, 0, s>>>(m, G, inv, off, packed_n, cu, st);
    else k_from_packed<double><<<nblocks(m.ne, LT), LT, 0, s>>>(m, G, inv, off, packed_n, cu, st);
  } else {
    if (corr_fp32) k_from_user<float><<<nblocks(m.ne, 128), 128, 0, s>>>(m, G, inv, cu, st);
    else k_from_user<double><<<nblocks(m.ne, 128), 128, 0, s>>>(m, G, inv, cu, st);
  }
  count_launch();
  SWE_CUDA_OK(cudaGetLastError());
  return 0;
}

int launch_to_user(cudaStream_t s, const DevMesh& m, const Groups& G, const int32_t* inv, const int64_t* off,
                   int64_t packed_n, int corr_fp32, StateDev st, double* cu) {
  if (m.ne == 0) return 0;
  if (off) {
    if (corr_fp32) k_to_packed<float><<<nblocks(m.ne, LT), LT, 0, s>>>(m, G, inv, off, packed_n, st, cu);
    else k_to_packed<double><<<nblocks(m.ne, LT), LT, 0, s>>>(m, G, inv, off, packed_n, st, cu);
  } else {
    if (corr_fp32) k_to_user<float><<<nblocks(m.ne, 128), 128, 0, s>>>(m, G, inv, st, cu);
    else k_to_user<double><<<nblocks(m.ne, 128), 128, 0, s>>>(m, G, inv, st, cu);
  }
  count_launch();
  SWE_CUDA_OK(cudaGetLastError());
  return 0;
}

// ---------------------------------------------------------------------------
// auxiliary system for p <= 1 (Sect. 3):  M_H u = U, M_H v = V with
//   M_H[i][j] = (1/s) sum_{n < K(i,j)} H_n T[n][i][j],  K(1,1) = 1, else 3.
// The 3 x 3 symmetric system is solved with its adjugate (one division).
// The basis is orthonormal with the constant phihat_1, so T[0][i][j] =
// T[i][0][j] = phihat_1 delta_ij: over phihat_1 the first row and column are
// H_0, H_1, H_2; of the T[n][i][j] with n, i, j >= 1 only T[1][1][2] (in any order)
// and T[2][2][2] are nonzero, mode 1 being odd along the collapsed coordinate (the
// factor comes back in the final scale).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_usolve_base(DevMesh m, int64_t n_end, Phys ph, const double* __restrict__ cb,
                                                     double* __restrict__ ub, float* __restrict__ ub32,
                                                     unsigned* status, unsigned long long* dmin) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  double u0 = 0.0, v0 = 0.0, H0 = 0.0;
  if (e < n_end) {
    const int64_t ne = m.ne;
    H0 = cb[0 * ne + e] + m.geo[G_HB0 * ne + e];
    const double U0 = cb[3 * ne + e], V0 = cb[6 * ne + e];
    if (!(H0 * m.geo[G_M0 * ne + e] > ph.h_min)) {  // mean depth: mode 0 times phi_{e,1} = phihat_1 / s_e
      atomicOr(status, (unsigned)ST_DEPTH);
      atomicOr(m.mstatus + m.mem[e], (unsigned)ST_DEPTH);
    }
    double v[6];
    if (m.p[e] == 0) {
      const double r = 1.0 / (H0 * m.geo[G_M0 * ne + e]);
      v[0] = U0 * r; v[1] = 0.0; v[2] = 0.0;
      v[3] = V0 * r; v[4] = 0.0; v[5] = 0.0;
    } else {
      const double H1 = cb[1 * ne + e] + m.geo[G_HB1 * ne + e];
      const double H2 = cb[2 * ne + e] + m.geo[G_HB2 * ne + e];
      const double U1 = cb[4 * ne + e], U2 = cb[5 * ne + e];
      const double V1 = cb[7 * ne + e], V2 = cb[8 * ne + e];
      // entries of S / phihat_1 with S = s M (the 1/s factor cancels in the
      // adjugate solve up to a final scale)
      const double a = H0, b = H1, c = H2;
      const double d = H0 + H2 * cTs[0];
      const double f = H1 * cTs[0];
      const double h = H0 + H2 * cTs[1];
      // M = (phihat_1 / s) [[a b c][b d f][c f h]];  u = s adj(S') U / (phihat_1 det(S'))
      const double C00 = d * h - f * f, C01 = c * f - b * h, C02 = b * f - c * d;
      const double C11 = a * h - c * c, C12 = b * c - a * f, C22 = a * d - b * b;
      const double det = a * C00 + b * C01 + c * C02;
      const double r = 1.0 / (det * m.geo[G_M0 * ne + e]);
      v[0] = (C00 * U0 + C01 * U1 + C02 * U2) * r; v[1] = (C01 * U0 + C11 * U1 + C12 * U2) * r;
      v[2] = (C02 * U0 + C12 * U1 + C22 * U2) * r; v[3] = (C00 * V0 + C01 * V1 + C02 * V2) * r;
      v[4] = (C01 * V0 + C11 * V1 + C12 * V2) * r; v[5] = (C02 * V0 + C12 * V1 + C22 * V2) * r;
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      ub[i * ne + e] = v[i];
      if (ub32) ub32[i * ne + e] = (float)v[i];
    }
    u0 = v[0];
    v0 = v[3];
  }
  if (dmin) {  // uniform over the grid: every thread of the block is here
    const bool in = e < n_end;
    const int64_t x = in ? e : 0;
    cfl_fold(dmin, in, m.mem[x], u0, v0, H0, m.geo[G_RS * m.ne + x], ph.g, m.geo[G_DIAM * m.ne + x], m.p[x]);
  }
}

int launch_usolve_base(cudaStream_t s, const DevMesh& m, const Groups& G, const Phys& ph, const double* cb,
                       double* ub, float* ub32, unsigned* status, unsigned long long* dmin) {
  const int64_t n = G.start[2];
  if (n == 0) return 0;
  const int ut = spread_threads(n, launch_shape().usolve_threads);
  k_usolve_base<<<nblocks(n, ut), ut, 0, s>>>(m, n, ph, cb, ub, ub32, status, dmin);
  count_launch();
  SWE_CUDA_OK(cudaGetLastError());
  return 0;
}

__global__ void k_reset_min(unsigned long long* dmin, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dmin[i] = (unsigned long long)__double_as_longlong(DBL_MAX);
}

int launch_reset_min(cudaStream_t s, unsigned long long* dmin, int nmem) {
  k_reset_min<<<nblocks(nmem, 128), 128, 0, s>>>(dmin, nmem);
  count_launch();
  SWE_CUDA_OK(cudaGetLastError());
  return 0;
}

// per member: dt = dt_fixed > 0 ? dt_fixed : cfl * min (before the step), and
// the minimum back to DBL_MAX for the next step's reduction (the velocity
// solves of the first stage fold their elements' CFL bounds into it);
// t += dt (after the step)
__global__ void k_set_dt(double* dt_dev, unsigned long long* dmin, double cfl, double dt_fixed, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    dt_dev[i] = dt_fixed > 0.0 ? dt_fixed : cfl * __longlong_as_double((long long)dmin[i]);
    dmin[i] = (unsigned long long)__double_as_longlong(DBL_MAX);
  }
}
__global__ void k_fill(double* p, double v, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = v;
}

int launch_fill(cudaStream_t s, double* p, double v, int n) {
  if (n <= 0) return 0;
  k_fill<<<nblocks(n, 128), 128, 0, s>>>(p, v, n);
  count_launch();
  SWE_CUDA_OK(cudaGetLastError());
  return 0;
}

__global__ void k_advance_time(double* t_dev, const double* dt_dev, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) t_dev[i] += dt_dev[i];
}

int launch_advance_time(cudaStream_t s, double* t_dev, unsigned long long* dmin, double cfl, double dt_fixed,
                        double* dt_dev, int nmem) {
  if (t_dev == nullptr) k_set_dt<<<nblocks(nmem, 128), 128, 0, s>>>(dt_dev, dmin, cfl, dt_fixed, nmem);
  else k_advance_time<<<nblocks(nmem, 128), 128, 0, s>>>(t_dev, dt_dev, nmem);
  count_launch();
  SWE_CUDA_OK(cudaGetLastError());
  return 0;
}

// ---------------------------------------------------------------------------
// Base edge flux (base_edge.cuh) of the edges of list[n], or of all of them
// (list == nullptr, n = nedge).  The correction edges are left out: their kernel
// writes the whole flux.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128) k_edge_base(DevMesh m, Phys ph, Stage stg, const int32_t* __restrict__ list,
                                                   int64_t n, const double* __restrict__ cb,
                                                   const double* __restrict__ ub, double* __restrict__ Fb, int chunk,
                                                   unsigned* work) {
  for_units(n, chunk, work, [&](int64_t unit) {
  const int64_t ed = list ? list[unit] : unit;
  double F[6], jump[2];
  base_flux(m, ph, stg, ed, m.eL[ed], m.eR[ed], m.einfo[ed], cb, ub, F, jump);
#pragma unroll
  for (int i = 0; i < 6; ++i) Fb[i * m.nedge + ed] = F[i];
  });
}

int launch_edge_base(cudaStream_t s, const DevMesh& m, const int32_t* list, int64_t n, const Phys& ph,
                     const Stage& stg, const double* cb, const double* ub, EdgeFlux fx, unsigned* work) {
  if (n == 0) return 0;
  const BaseGrid g = base_grid(n, launch_shape());
  k_edge_base<<<g.blocks, g.threads, 0, s>>>(m, ph, stg, list, n, cb, ub, fx.Fb, g.chunk, work);
  count_launch();
  SWE_CUDA_OK(cudaGetLastError());
  return 0;
}

// ---------------------------------------------------------------------------
// Base element update.  For test modes q of degree 1, grad phi_q is constant,
// so by orthonormality (Eq. 13 restricted to indices <= 3)
//   (A_xi, grad phi_q) = grad phi_q . (U_1, V_1) sqrt|Omega|
//   (A_U , grad phi_q) = d_x phi_q sum_i (U_i u_i + g(xi_i^2/2 + xi_i hb_i))
//                      + d_y phi_q sum_i U_i v_i          (and alike for V),
// the source (r, phi_q) = g grad h_b xi_q (- tau u_q + f_c V_q, - tau v_q -
// f_c U_q with bottom friction and Coriolis), and the edge terms are
// -sum_g F_g phi_q(x_g) over the three edges (sign flipped for the right side).
// ---------------------------------------------------------------------------
// The update of one element.  F: the field whose three modes are computed (0 xi, 1
// U, 2 V), or -1 for all three.  Every multiply-add is written as an fma where the
// compiler could pick one of two contractions, so that both forms give the same bits.
template <int F>
__device__ __forceinline__ void elem_unit(const DevMesh& m, const Phys& ph, const Stage& stg,
                                          const double* __restrict__ cbS, const double* __restrict__ cbN,
                                          double* __restrict__ cbO, float* __restrict__ cbO32,
                                          const double* __restrict__ ub, const double* __restrict__ Fb,
                                          const double* __restrict__ rc, int64_t rc_start, int64_t e) {
  constexpr int F0 = F < 0 ? 0 : F, F1 = F < 0 ? 3 : F + 1;
  const int64_t ne = m.ne, nE = m.nedge;
  const double* geo = m.geo;
  double c[3][3], u[2][3];
#pragma unroll
  for (int f = 0; f < 3; ++f)
#pragma unroll
    for (int i = 0; i < 3; ++i) c[f][i] = cbS[(f * 3 + i) * ne + e];
#pragma unroll
  for (int f = 0; f < 2; ++f)
#pragma unroll
    for (int i = 0; i < 3; ++i) u[f][i] = ub[(f * 3 + i) * ne + e];
  const double rs = geo[G_RS * ne + e], sqa = geo[G_SQA * ne + e], m0 = geo[G_M0 * ne + e];
  const double hb[3] = {geo[G_HB0 * ne + e], geo[G_HB1 * ne + e], geo[G_HB2 * ne + e]};
  double r[3][3];
  // volume terms
  double Axx = 0.0, Axy = 0.0, Ayx = 0.0, Ayy = 0.0, P = 0.0;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    Axx = fma(c[1][i], u[0][i], Axx); Axy = fma(c[1][i], u[1][i], Axy);
    Ayx = fma(c[2][i], u[0][i], Ayx); Ayy = fma(c[2][i], u[1][i], Ayy);
    P = fma(c[0][i], fma(0.5, c[0][i], hb[i]), P);
  }
  Axx = fma(ph.g, P, Axx);
  Ayy = fma(ph.g, P, Ayy);
  const double gdx = geo[G_GDHX * ne + e], gdy = geo[G_GDHY * ne + e];
  const double U0s = c[1][0] * sqa, V0s = c[2][0] * sqa;
  r[0][0] = 0.0;
  r[1][0] = gdx * c[0][0];
  r[2][0] = gdy * c[0][0];
#pragma unroll
  for (int q = 1; q < 3; ++q) {
    const double gx = geo[(q == 1 ? G_GQ1X : G_GQ2X) * ne + e], gy = geo[(q == 1 ? G_GQ1Y : G_GQ2Y) * ne + e];
    r[0][q] = fma(gx, U0s, gy * V0s);
    r[1][q] = fma(gdx, c[0][q], fma(gx, Axx, gy * Axy));
    r[2][q] = fma(gdy, c[0][q], fma(gx, Ayx, gy * Ayy));
  }
  if (F != 0 && ph.src) {
    // bottom friction and Coriolis of Eq. (5); tau from the element means of H
    // and u (Sect. 3), mean = mode 0 / sqrt|Omega| = mode 0 * sqrt 2 / s_e
    const double ra = 1.4142135623730951 * rs;
    const double Hm = (c[0][0] + hb[0]) * ra, um = u[0][0] * ra, vm = u[1][0] * ra;
    const double tau = fma(ph.fric_lin, Hm, ph.fric_quad * sqrt(fma(um, um, vm * vm)));
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      r[1][q] += fma(ph.f_c, c[2][q], -(tau * u[0][q]));
      r[2][q] -= fma(ph.f_c, c[1][q], tau * u[1][q]);
    }
  }
  // edge terms
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int ee = m.eedge[k * ne + e];
    const int64_t ed = ee >> 1;
    const bool right = ee & 1;
    // the basis at the edge's two points, times -1/s_e (left side) or +1/s_e
    // (right side, whose own direction is reversed): table values with the
    // sign bit set by an integer xor, no FP64 multiply
    const unsigned long long neg = right ? 0ull : 0x8000000000000000ull;
    auto sgn = [neg](double x) { return __longlong_as_double(__double_as_longlong(x) ^ neg); };
    const double2 p0 = *reinterpret_cast<const double2*>(m.etb + (3 * e + k) * 4);
    const double2 p1 = *reinterpret_cast<const double2*>(m.etb + (3 * e + k) * 4 + 2);
    const double s0 = sgn(m0);  // mode 1 is the constant phi_{e,1}
    const double b10 = sgn(right ? p1.x : p0.x), b11 = sgn(right ? p0.x : p1.x);
    const double b20 = sgn(right ? p1.y : p0.y), b21 = sgn(right ? p0.y : p1.y);
#pragma unroll
    for (int f = F0; f < F1; ++f) {
      const double A0 = Fb[(f * 2 + 0) * nE + ed], A1 = Fb[(f * 2 + 1) * nE + ed];
      // r += x y + z w is a multiply, an FMA and an add; this way two FMAs: 113
      // FP64 instructions per element instead of 131 (GB300, 524,288 triangles, 6
      // stages: 2,800 -> 2,668 us)
      r[f][0] = fma(s0, A0 + A1, r[f][0]);
      r[f][1] = fma(A1, b11, fma(A0, b10, r[f][1]));
      r[f][2] = fma(A1, b21, fma(A0, b20, r[f][2]));
    }
  }
  // correction of the base modes from the volume terms of p >= 2 elements
  if (F != 0 && !stg.base_only && e >= rc_start) {
    const int64_t nrc = ne - rc_start, lr = e - rc_start;
#pragma unroll
    for (int f = F0 > 1 ? F0 : 1; f < F1; ++f)
#pragma unroll
      for (int q = 1; q < 3; ++q) r[f][q] += rc[((f - 1) * 2 + q - 1) * nrc + lr];
  }
  const int K = m.p[e] == 0 ? 1 : 3;
  const double dt = stage_dt(stg, m.mem[e]), a = stg.a, bb = stg.b;
  const bool euler = a == 0.0 && bb == 1.0;  // the first stage: c + dt r
#pragma unroll
  for (int f = F0; f < F1; ++f)
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int64_t ix = (f * 3 + q) * ne + e;
      double v = 0.0;
      if (q < K) {
        if (stg.rhs_only) v = r[f][q];
        else if (euler) v = fma(dt, r[f][q], c[f][q]);
        else v = fma(bb, fma(dt, r[f][q], c[f][q]), a != 0.0 ? a * cbN[ix] : 0.0);
      }
      cbO[ix] = v;
      if (cbO32) cbO32[ix] = (float)v;
    }
}

// MINB: blocks per SM the register allocation must allow -- 4 (128 registers)
// for uncapped grids, where the kernel's own occupancy is what counts; 3 for
// grids capped at a few blocks per SM beside the correction kernels, where
// the measured step is faster with the unrestricted allocation
template <int MINB>
__global__ void __launch_bounds__(128, MINB) k_elem_base(DevMesh m, Phys ph, Stage stg, const double* __restrict__ cbS,
                                                   const double* __restrict__ cbN, double* __restrict__ cbO,
                                                   float* __restrict__ cbO32, const double* __restrict__ ub,
                                                   const double* __restrict__ Fb, const double* __restrict__ rc, int64_t rc_start, int chunk,
                                                   unsigned* work) {
  for_units(m.ne, chunk, work,
            [&](int64_t e) { elem_unit<-1>(m, ph, stg, cbS, cbN, cbO, cbO32, ub, Fb, rc, rc_start, e); });
}

// Few elements: a block of three warps updates 32 of them, a warp to a field.  A
// lone warp issues an FP64 instruction in 64 cycles and its SM one in 19, so the
// longest field's about 50 instructions in a chain count instead of the 113 of all three
// as long as an SM holds few warps.  Measured per stage (GB300, p = 1, FP64; one
// thread per element -> this form): 512 triangles 19.1 ->
// 17.0 us, 2,048 19.1 -> 17.1, 4,608 19.8 -> 17.7, 8,192 20.4 -> 18.4; p 1 - 4,
// mixed: 512 43.0 -> 41.8, 2,048 44.4 -> 43.5.
// Beside correction kernels, which share the pipe, the repeated common terms
// cost more than the shorter chain gains from about 3,000 elements on (p 1 - 4,
// FP64: 512 and 2,048 elements within 0.2 %, 3,200 and 4,608 0.6 and 1 % slower).
static int64_t field_elems(bool base_only) { return base_only ? 8192 : 2048; }

__global__ void __launch_bounds__(96) k_elem_base_fields(DevMesh m, Phys ph, Stage stg, const double* __restrict__ cbS,
                                                         const double* __restrict__ cbN, double* __restrict__ cbO,
                                                         float* __restrict__ cbO32, const double* __restrict__ ub,
                                                         const double* __restrict__ Fb, const double* __restrict__ rc,
                                                         int64_t rc_start) {
  const int64_t e = blockIdx.x * (int64_t)32 + (threadIdx.x & 31);
  if (e >= m.ne) return;
  const int f = threadIdx.x >> 5;
  if (f == 0) elem_unit<0>(m, ph, stg, cbS, cbN, cbO, cbO32, ub, Fb, rc, rc_start, e);
  else if (f == 1) elem_unit<1>(m, ph, stg, cbS, cbN, cbO, cbO32, ub, Fb, rc, rc_start, e);
  else elem_unit<2>(m, ph, stg, cbS, cbN, cbO, cbO32, ub, Fb, rc, rc_start, e);
}

int launch_elem_base(cudaStream_t s, const DevMesh& m, const Groups& G, const Phys& ph, const Stage& stg,
                     const double* cbS, const double* cbN, double* cbO, float* cbO32, const double* ub, EdgeFlux fx,
                     const void* rc, unsigned* work) {
  if (m.ne == 0) return 0;
  const LaunchShape& L = launch_shape();
  const BaseGrid g = base_grid(m.ne, L);
  if (m.ne <= field_elems(G.start[2] == m.ne))
    k_elem_base_fields<<<nblocks(m.ne, 32), 96, 0, s>>>(m, ph, stg, cbS, cbN, cbO, cbO32, ub, fx.Fb, (const double*)rc,
                                                        G.start[2]);
  else if (L.base_bpsm == 0 || L.base_bpsm >= 4)
    k_elem_base<4><<<g.blocks, g.threads, 0, s>>>(m, ph, stg, cbS, cbN, cbO, cbO32, ub, fx.Fb, (const double*)rc,
                                                  G.start[2], g.chunk, work);
  else
    k_elem_base<3><<<g.blocks, g.threads, 0, s>>>(m, ph, stg, cbS, cbN, cbO, cbO32, ub, fx.Fb, (const double*)rc,
                                                  G.start[2], g.chunk, work);
  count_launch();
  SWE_CUDA_OK(cudaGetLastError());
  return 0;
}

// ---------------------------------------------------------------------------
// p-adaptivity indicator (modal decay of xi, FP64 in every mode):
//   s_e = sum_{deg i = p_e} xi_i^2 / sum_{deg i >= 1} xi_i^2
// p_e + 1 if s_e > theta_up (p_e < p_max), p_e - 1 if s_e < theta_down
// (p_e > p_min).  The new orders are written in the caller's element order.
// ---------------------------------------------------------------------------
template <typename TC>
__global__ void k_indicator(DevMesh m, Groups G, const int32_t* __restrict__ perm, StateDev st, double up,
                            double down, int pmin, int pmax, int8_t* __restrict__ p_user) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= m.ne) return;
  const int64_t ne = m.ne;
  const int p = m.p[e], K = Kof(p);
  double num = 0.0, den = 0.0;
  for (int i = 1; i < K && i < 3; ++i) {
    const double x = st.cb[i * ne + e];
    den += x * x;
    if (p == 1) num += x * x;
  }
  if (p >= 2) {
    const int64_t n = G.start[p + 1] - G.start[p], l = e - G.start[p];
    const TC* h = chp<TC>(st.ch[p]);
    for (int i = 3; i < K; ++i) {
      const double x = (double)h[(i - 3) * n + l];
      den += x * x;
      if (deg_of(i) == p) num += x * x;
    }
  }
  const double s = (p > 0 && den > 0.0) ? num / den : 0.0;
  int q = p;
  if (s > up && p < pmax) q = p + 1;
  else if (s < down && p > pmin) q = p - 1;
  p_user[perm[e]] = (int8_t)q;
}

int launch_indicator(cudaStream_t s, const DevMesh& m, const Groups& G, const int32_t* perm, int corr_fp32,
                     StateDev st, double up, double down, int pmin, int pmax, int8_t* p_user) {
  if (m.ne == 0) return 0;
  if (corr_fp32) k_indicator<float><<<nblocks(m.ne, 256), 256, 0, s>>>(m, G, perm, st, up, down, pmin, pmax, p_user);
  else k_indicator<double><<<nblocks(m.ne, 256), 256, 0, s>>>(m, G, perm, st, up, down, pmin, pmax, p_user);
  count_launch();
  SWE_CUDA_OK(cudaGetLastError());
  return 0;
}

// ---------------------------------------------------------------------------
// status: non-finite values in the state
// ---------------------------------------------------------------------------
template <typename TC>
__global__ void k_check(DevMesh m, Groups G, StateDev st, unsigned* status) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= m.ne) return;
  const int64_t ne = m.ne;
  bool bad = false;
  for (int i = 0; i < 9; ++i) bad |= !isfinite(st.cb[i * ne + e]);
  const int p = m.p[e];
  if (p >= 2) {
    const int K = Kof(p);
    const int64_t n = G.start[p + 1] - G.start[p], l = e - G.start[p];
    const TC* h = chp<TC>(st.ch[p]);
    for (int i = 0; i < 3 * (K - 3); ++i) bad |= !isfinite((double)h[i * n + l]);
  }
  if (bad) {
    atomicOr(status, (unsigned)ST_NONFINITE);
    atomicOr(m.mstatus + m.mem[e], (unsigned)ST_NONFINITE);
  }
}

int launch_check_state(cudaStream_t s, const DevMesh& m, const Groups& G, int corr_fp32, StateDev st,
                       unsigned* status) {
  if (m.ne == 0) return 0;
  if (corr_fp32) k_check<float><<<nblocks(m.ne, 256), 256, 0, s>>>(m, G, st, status);
  else k_check<double><<<nblocks(m.ne, 256), 256, 0, s>>>(m, G, st, status);
  count_launch();
  SWE_CUDA_OK(cudaGetLastError());
  return 0;
}

// ---------------------------------------------------------------------------
// deterministic reductions (fixed tree per block, blocks summed in order)
// ---------------------------------------------------------------------------
__device__ void block_sum_store(double v, double* partial) {
  __shared__ double red[256];
  red[threadIdx.x] = v;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}

__global__ void k_sum_partials(const double* partial, int n, double* out) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    double s = 0.0;
    for (int i = 0; i < n; ++i) s += partial[i];
    *out = s;
  }
}

__global__ void k_mass(DevMesh m, const double* __restrict__ cb, double* partial) {
  double v = 0.0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m.ne; e += (int64_t)gridDim.x * blockDim.x)
    v += m.geo[G_SQA * m.ne + e] * cb[e];
  block_sum_store(v, partial);
}

int launch_mass(cudaStream_t s, const DevMesh& m, const double* cb, double* partial, int nblk, double* out) {
  k_mass<<<nblk, 256, 0, s>>>(m, cb, partial);
  count_launch();
  k_sum_partials<<<1, 32, 0, s>>>(partial, nblk, out);
  count_launch();
  SWE_CUDA_OK(cudaGetLastError());
  return 0;
}

template <typename TC>
__global__ void k_energy(DevMesh m, Groups G, Phys ph, StateDev c, VelDev u, double* partial) {
  double v = 0.0;
  const int64_t ne = m.ne;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < ne; e += (int64_t)gridDim.x * blockDim.x) {
    const int p = m.p[e], K = Kof(p);
    for (int i = 0; i < 3 && i < K; ++i) {
      const double x = c.cb[i * ne + e];
      v += 0.5 * ph.g * x * x + 0.5 * (c.cb[(3 + i) * ne + e] * u.ub[i * ne + e] + c.cb[(6 + i) * ne + e] * u.ub[(3 + i) * ne + e]);
    }
    if (p >= 2) {
      const int64_t n = G.start[p + 1] - G.start[p], l = e - G.start[p];
      const TC* h = chp<TC>(c.ch[p]);
      const TC* uh = chp<TC>(u.uh[p]);
      const int Kh = K - 3;
      for (int i = 0; i < Kh; ++i) {
        const double x = h[i * n + l];
        v += 0.5 * ph.g * x * x + 0.5 * ((double)h[(Kh + i) * n + l] * (double)uh[i * n + l] +
                                         (double)h[(2 * Kh + i) * n + l] * (double)uh[(Kh + i) * n + l]);
      }
    }
  }
  block_sum_store(v, partial);
}

int launch_energy(cudaStream_t s, const DevMesh& m, const Groups& G, int corr_fp32, const Phys& ph, StateDev c,
                  VelDev u, double* partial, int nblk, double* out) {
  if (corr_fp32) k_energy<float><<<nblk, 256, 0, s>>>(m, G, ph, c, u, partial);
  else k_energy<double><<<nblk, 256, 0, s>>>(m, G, ph, c, u, partial);
  count_launch();
  k_sum_partials<<<1, 32, 0, s>>>(partial, nblk, out);
  count_launch();
  SWE_CUDA_OK(cudaGetLastError());
  return 0;
}

}  // namespace swedg
