// FP32 correction with the momentum volume terms of Eq. (13) on the 5th-
// generation tensor cores (tcgen05, TF32 inputs, FP32 accumulation in TMEM).
//
// The correction kernels of k_corr_impl.cuh are instantiated once more here
// (namespace corrtc, FP32, CORR_TC); for the orders with K >= 10 modes the
// element update is k_elem_tc<K>.  It forms the products of k_corr_impl.cuh's
// element update (products), for every mode m below the element's degree
//   Zuu_m = sum_i U_i Wu[m][i], Zuv, Zvu, Zvv alike, P_m = sum_i xi_i Wx[m][i],
//   Wu[m][i] = sum_j T[m][i][j] u_j, Wv of v, Wx of xi / 2,
// in two stages.  Stage one, W, is three GEMMs per tile of 128 elements that
// share one constant operand: rows = elements with their K values u, v or xi / 2,
// columns = pairs (m, i).  T is symmetric, so a pair of two modes below the
// element's degree is one column for both, and pairs with a constant mode need no
// product (T[m][0][j] = phihat_1 delta_mj): 90 columns for K = 15, 35 for K =
// 10.  The thinnest 10 (3) of them, of one or two entries, are summed on the
// CUDA cores instead, which makes the GEMMs N = 80 (32) and lets two (three)
// CTAs share an SM's TMEM, each one's loads and CUDA-core work under the
// others' MMAs.  Stage two, the sums over i and everything that follows
// (D, source, edges, RK), runs on the CUDA cores, each thread reading its own
// element's row of the accumulators from TMEM.  The terms that need no GEMM are
// formed while the MMAs run.
//
// Measured on the 2,097,152-triangle shelf (GB300), orders 3 and 4 of one stage:
// k_elem_tc replaces a contraction over (k, j) with the G tensors of all test
// modes (N = 16 K, 2 K columns per row, four times the MMA work, two passes for K =
// 15, 128 threads per SM) and a second kernel that read its result back from
// memory, 342 us together, by 167 + 132 us.  The tensor pipe is 2 % busy: what is
// left are the loads and the CUDA-core work of 8 to 12 warps per SM.
//
// Precision: every FP32 operand x is split into two TF32 parts, x = h + t
// to within 2^-22 |x|, with h = tf32(x) and t = tf32(x - h) (tf32 = round to
// the nearest value with 10 mantissa bits), and each GEMM runs as the three
// products hh + ht + th into one FP32 accumulator.  The B parts come from the
// FP64 values of T.  The bottom term's products xi_i h_b_j (i >= 3, see
// products) are added on the CUDA cores.
//
// Schedule: persistent CTAs of 128 threads (thread t = element row t of the
// tile) load B once (a bulk TMA copy on an mbarrier), then per tile: the threads
// write the A operands into shared memory; one thread issues the MMAs and commits
// them to an mbarrier; every thread reads its TMEM row and finishes.
//
// Shared-memory operand layout: K-major with the 128-byte swizzle.  A row is
// 32 floats = 128 bytes, the head parts of 16 reduction columns and then their
// tails; groups of 8 rows are 1024 bytes apart (the descriptor's
// stride-dimension byte offset), and the 16-byte unit u of row r is stored at unit
// u ^ (r % 8): (row r, column c) at float offset
//   (r / 8) * 256 + (r % 8) * 32 + (((c / 4) ^ (r % 8)) * 4) + c % 4.
// An MMA step of 8 columns starts 32 bytes further into the rows.
//
// Every mbarrier wait is bounded; a wait that runs out sets ST_TIMEOUT in the
// status word, skips the result and still frees the CTA's TMEM.
#include <algorithm>
#include <cstring>

#define CORR_T float
#define CORR_NS corrtc
#define CORR_TC 1
#include "k_corr_impl.cuh"
#include "tc_issue.h"

namespace swedg {
namespace corrtc {

// orthogonality zeros of G_k[q][i][j], and the base triples
__host__ __device__ constexpr bool gnz(int q, int i, int j) {
  return deg_of(q) == 0 ? false
         : deg_of(q) == 1 ? i == j
                          : (deg_of(i) <= deg_of(j) + deg_of(q) - 1 && deg_of(j) <= deg_of(i) + deg_of(q) - 1);
}
__host__ __device__ constexpr bool base3(int q, int i, int j) { return q < 3 && i < 3 && j < 3; }

constexpr int TC_M = 128;     // elements per tile = MMA M
constexpr int TC_ROW = 32;    // floats of an operand row: 16 head columns, 16 tail columns
constexpr int TC_ABUF = TC_M * TC_ROW;
constexpr uint32_t TC_SPIN = 1u << 22;

// The columns (m, i) of the GEMMs and the pairs left to the CUDA cores.
template <int K>
struct TcPairs {
  int nc = 0, nt = 0;
  int cm[96] = {}, ci[96] = {}, tm[16] = {}, ti[16] = {};
};
template <int K>
__host__ __device__ constexpr TcPairs<K> tc_pairs() {
  constexpr int KL = Kof(deg_of(K - 1) - 1), thin = K == 15 ? 10 : 3;
  TcPairs<K> p;
  for (int size = 1; size <= K; ++size)  // the thinnest pairs first
    for (int m = 1; m < KL; ++m)
      for (int i = m; i < K; ++i) {
        int nz = 0;
        for (int j = 0; j < K; ++j) nz += tnz(m, i, j) ? 1 : 0;
        if (nz != size) continue;
        if (p.nt < thin) {
          p.tm[p.nt] = m;
          p.ti[p.nt++] = i;
        } else {
          p.cm[p.nc] = m;
          p.ci[p.nc++] = i;
        }
      }
  return p;
}
__host__ __device__ constexpr int tc_n(int K) { return K == 15 ? 80 : 32; }        // MMA N
__host__ __device__ constexpr int tc_cols(int K) { return K == 15 ? 256 : 128; }    // TMEM columns per CTA
__host__ __device__ constexpr int tc_ctas(int K) { return K == 15 ? 2 : 3; }        // CTAs per SM
static_assert(tc_pairs<15>().nc == tc_n(15) && tc_pairs<10>().nc == tc_n(10), "GEMM columns");
static_assert(3 * tc_n(15) <= tc_cols(15) && 3 * tc_n(10) <= tc_cols(10), "TMEM columns of one CTA");
static_assert(tc_ctas(15) * tc_cols(15) <= 512 && tc_ctas(10) * tc_cols(10) <= 512, "TMEM columns of an SM");
static_assert(tc_n(15) % 16 == 0 && tc_n(10) % 16 == 0, "MMA N");
__host__ __device__ constexpr int tc_bfloats(int K) { return tc_n(K) * TC_ROW; }
__host__ __device__ constexpr int tc_boff(int K) { return K == 10 ? 0 : tc_bfloats(10); }
constexpr int TC_BTOTAL = tc_bfloats(10) + tc_bfloats(15);
// float offset of (row r, column c) in a K-major operand with the 128-byte swizzle
__host__ __device__ constexpr int tc_at(int r, int c) {
  return (r / 8) * 256 + (r % 8) * 32 + (((c / 4) ^ (r % 8)) * 4) + (c % 4);
}
// shared memory of k_elem_tc<K>: three A operands, B, barriers + TMEM slot
__host__ __device__ constexpr int tc_smem(int K) { return (3 * TC_ABUF + tc_bfloats(K)) * 4 + 64; }
static_assert(tc_ctas(15) * (tc_smem(15) + 1024) <= 227 * 1024 && tc_ctas(10) * (tc_smem(10) + 1024) <= 227 * 1024,
              "shared memory of an SM");

// round to the nearest value with a 10-bit mantissa (ties away from zero)
static inline float tf32_round(float x) {
  uint32_t u;
  std::memcpy(&u, &x, 4);
  u = (u + 0x1000u) & 0xffffe000u;
  float h;
  std::memcpy(&h, &u, 4);
  return h;
}

// The operand of the one-GEMM form of the contraction, G_k over (k, j) (see
// swe_tc_operand_image): two parts of 16 K rows of 32 columns.
int64_t tc_operand_image(int K, float* out, int64_t cap) {
  if (K != 6 && K != 10 && K != 15) return -1;
  const int64_t part_n = 16 * K * TC_ROW, need = 2 * part_n;
  if (!out) return need;
  if (cap < need) return -1;
  const RefTables& R = tables();
  std::fill(out, out + need, 0.0f);
  for (int k = 0; k < 2; ++k)
    for (int q = 0; q < K; ++q)
      for (int i = 0; i < K; ++i)
        for (int j = 0; j < K; ++j) {
          if (!gnz(q, i, j) || base3(q, i, j)) continue;
          const int row = 16 * i + q, col = k * K + j;
          double rest = R.G[k][q][i][j];
          for (int part = 0; part < 2; ++part) {
            const float v = tf32_round((float)rest);
            rest -= (double)v;
            out[part * part_n + tc_at(row, col)] = v;
          }
        }
  return need;
}

// B of k_elem_tc<K>: row c = the pair of column c, T[m][i][j] for j < K, heads then tails
template <int K>
static void tc_b_image(float* out) {
  constexpr TcPairs<K> P = tc_pairs<K>();
  const RefTables& R = tables();
  for (int c = 0; c < P.nc; ++c)
    for (int j = 0; j < K; ++j) {
      if (!tnz(P.cm[c], P.ci[c], j)) continue;
      const double t = R.T[P.cm[c]][P.ci[c]][j];
      const float h = tf32_round((float)t);
      out[tc_at(c, j)] = h;
      out[tc_at(c, 16 + j)] = tf32_round((float)(t - (double)h));
    }
}

// Both B images (host).  Contexts of any device copy them to their own memory
// without a lock, so they are written once, before the first caller gets them.
struct TcOperand {
  float b[TC_BTOTAL] = {};
  TcOperand() {
    tc_b_image<10>(b + tc_boff(10));
    tc_b_image<15>(b + tc_boff(15));
  }
};
const float* tc_operand(size_t* bytes) {
  static const TcOperand op;
  *bytes = sizeof op.b;
  return op.b;
}

template <int K>
static int64_t pair_operand(float* out, int64_t cap, int32_t* pairs) {
  constexpr TcPairs<K> P = tc_pairs<K>();
  constexpr int64_t need = tc_bfloats(K);
  if (!out) return need;
  if (cap < need) return -1;
  size_t bytes = 0;
  std::memcpy(out, tc_operand(&bytes) + tc_boff(K), need * sizeof(float));
  for (int c = 0; pairs && c < P.nc + P.nt; ++c) {
    pairs[2 * c] = c < P.nc ? P.cm[c] : P.tm[c - P.nc];
    pairs[2 * c + 1] = c < P.nc ? P.ci[c] : P.ti[c - P.nc];
  }
  return need;
}
int64_t tc_pair_operand(int K, float* out, int64_t cap, int32_t* pairs) {
  return K == 10 ? pair_operand<10>(out, cap, pairs) : K == 15 ? pair_operand<15>(out, cap, pairs) : -1;
}

// ------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: K-major, 128-byte swizzle (layout type 2),
// SBO 1024 B between groups of 8 rows; LBO is not used by swizzled K-major
// layouts whose K step fits in the 128-byte row (encoded as 1)
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// instruction descriptor of kind::tf32: D FP32, A and B TF32, both K-major, M x N
__host__ __device__ constexpr uint32_t tc_idesc(int M, int N) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mbar_init(uint32_t a, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t a) {
  uint64_t state;
  asm volatile("mbarrier.arrive.shared::cta.b64 %0, [%1];" : "=l"(state) : "r"(a) : "memory");
}
__device__ __forceinline__ bool mbar_wait(uint32_t a, uint32_t parity) {
  for (uint32_t it = 0; it < TC_SPIN; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

// one bulk TMA copy global -> shared, completing on the mbarrier
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ float tf32_rn(float x) { return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xffffe000u); }

// one A row: the K values v (zero to 16), heads and tails, x = h + t to within 2^-22 |x|
template <int K>
__device__ __forceinline__ void write_a_row(float* A, int r, const float (&v)[K], float scale) {
#pragma unroll
  for (int c4 = 0; c4 < 4; ++c4) {
    float h[4], t[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = 4 * c4 + i;
      const float x = c < K ? scale * v[c < K ? c : 0] : 0.0f;
      h[i] = tf32_rn(x);
      t[i] = tf32_rn(x - h[i]);
    }
    *reinterpret_cast<float4*>(A + tc_at(r, 4 * c4)) = make_float4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<float4*>(A + tc_at(r, 16 + 4 * c4)) = make_float4(t[0], t[1], t[2], t[3]);
  }
}

// the five products of one mode
struct Prod {
  float uu, uv, vu, vv, p;
  __device__ __forceinline__ void add(float U, float V, float xi, float wu, float wv, float wx) {
    uu = fmaf(U, wu, uu);
    uv = fmaf(U, wv, uv);
    vu = fmaf(V, wu, vu);
    vv = fmaf(V, wv, vv);
    p = fmaf(xi, wx, p);
  }
};

template <int K>
__global__ void __launch_bounds__(TC_M, tc_ctas(K)) k_elem_tc(ELEM_CORR_PARAMS, const float* __restrict__ bimg,
                                                              unsigned* status) {
  constexpr int KL = Kof(deg_of(K - 1) - 1), N = tc_n(K);
  constexpr TcPairs<K> P = tc_pairs<K>();
  extern __shared__ __align__(1024) unsigned char tc_smem_raw[];
  float* sA = reinterpret_cast<float*>(tc_smem_raw);  // [u, v, xi / 2][128 rows][32]
  float* sB = sA + 3 * TC_ABUF;                        // [N rows][32]
  uint64_t* bars = reinterpret_cast<uint64_t*>(sB + tc_bfloats(K));
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 2);
  const int t = threadIdx.x, w = t >> 5;
  const uint32_t bfull = smem_u32(bars), mdone = smem_u32(bars + 1);
  if (t == 0) {
    mbar_init(bfull, 1);
    mbar_init(mdone, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (w == 0) {
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(tc_cols(K))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  if (t == 0) {  // B, once per CTA
    uint64_t state;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 %0, [%1], %2;"
                 : "=l"(state)
                 : "r"(bfull), "r"((uint32_t)(tc_bfloats(K) * 4))
                 : "memory");
    bulk_g2s(smem_u32(sB), bimg, (uint32_t)(tc_bfloats(K) * 4), bfull);
  }
  // the swizzle XOR acts on address bits 4-9: operands must start on 1024 bytes
  bool ok = (smem_u32(sA) & 1023u) == 0 && (smem_u32(sB) & 1023u) == 0;
  bool blanded = false;
  uint32_t commits = 0;
  const uint32_t idesc = tc_idesc(TC_M, N);
  const uint32_t lane_base = tmem + ((uint32_t)(32 * w) << 16);
  const float* geo = m.geo32;
  const int64_t ne = m.ne;
  const float g = (float)ph.g;
  const float f0 = cT[0][0];  // T[0][0][0] = phihat_1

#pragma unroll 1
  for (int64_t tile = blockIdx.x; tile * TC_M < n; tile += gridDim.x) {
    const int64_t l = tile * TC_M + t;
    const bool live = l < n;
    const int64_t e = g0 + (live ? l : 0);
    float xi[K], U[K], V[K];
    Prod Z[KL];
    float tau = 0.0f;
    {
      float u[K], v[K];
      if (live) {
        load_modes<K>(xi, cbS, ne, e, chS, n, l, 0);
        load_modes<K>(U, cbS, ne, e, chS, n, l, 1);
        load_modes<K>(V, cbS, ne, e, chS, n, l, 2);
        load_modes<K>(u, ub, ne, e, uh, n, l, 0);
        load_modes<K>(v, ub, ne, e, uh, n, l, 1);
      } else {
        sfor<0, K>([&](auto j) { xi[j] = U[j] = V[j] = u[j] = v[j] = 0.0f; });
      }
      write_a_row<K>(sA, t, u, 1.0f);
      write_a_row<K>(sA + TC_ABUF, t, v, 1.0f);
      write_a_row<K>(sA + 2 * TC_ABUF, t, xi, 0.5f);
      // publish the rows to the tensor cores' (async) proxy; the previous tile's
      // TMEM reads are complete (tcgen05.wait::ld) before the barrier
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_fence_before();
      __syncthreads();
      if (t == 0) {
        ok = tc_issue(
            ok, blanded, [&] { return mbar_wait(bfull, 0); },
            [&] {
              tc_fence_after();
              const uint32_t b = smem_u32(sB);
#pragma unroll
              for (int gi = 0; gi < 3; ++gi) {
                const uint32_t a = smem_u32(sA + gi * TC_ABUF), d = tmem + (uint32_t)(gi * N);
#pragma unroll
                for (int st = 0; st < 2; ++st) {  // two steps of 8 columns: 32 bytes further into the rows; tails 64 on
                  const uint32_t o = 32u * st;
                  tc_mma(d, tc_desc(a + o), tc_desc(b + o), idesc, st > 0 ? 1u : 0u);  // h h
                  tc_mma(d, tc_desc(a + o), tc_desc(b + 64u + o), idesc, 1u);           // h t
                  tc_mma(d, tc_desc(a + 64u + o), tc_desc(b + o), idesc, 1u);           // t h
                }
              }
              asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mdone)
                           : "memory");
            },
            [&] { mbar_arrive(mdone); });
      }
      // while the MMAs run: what needs no GEMM.  The constant mode on either side ...
      Prod z0{0.f, 0.f, 0.f, 0.f, 0.f};
      sfor<0, K>([&](auto i) { z0.add(U[i], V[i], xi[i], u[i], v[i], 0.5f * xi[i]); });
      Z[0] = Prod{f0 * z0.uu, f0 * z0.uv, f0 * z0.vu, f0 * z0.vv, f0 * z0.p};
      const float U0 = f0 * U[0], V0 = f0 * V[0], x0 = f0 * xi[0];
      sfor<1, KL>([&](auto M) { Z[M] = Prod{U0 * u[M], U0 * v[M], V0 * u[M], V0 * v[M], x0 * (0.5f * xi[M])}; });
      // ... the thin pairs ...
      sfor<0, P.nt>([&](auto c) {
        constexpr int M = P.tm[c], I = P.ti[c];
        float wu = 0.f, wv = 0.f, wx = 0.f;
        sfor<0, K>([&](auto j) {
          if constexpr (tnz(M, I, j)) {
            const float tt = cT[M][pk(I, j)];
            wu = fmaf(u[j], tt, wu);
            wv = fmaf(v[j], tt, wv);
            wx = fmaf(0.5f * xi[j], tt, wx);
          }
        });
        Z[M].add(U[I], V[I], xi[I], wu, wv, wx);
        if constexpr (I < KL && I != M) Z[I < KL ? I : 0].add(U[M], V[M], xi[M], wu, wv, wx);
      });
      // ... and the bottom term's products with the higher elevation modes
      const float hb[3] = {geo[G_HB0 * ne + e], geo[G_HB1 * ne + e], geo[G_HB2 * ne + e]};
      sfor<1, KL>([&](auto M) {
        sfor<3, K>([&](auto i) {
          sfor<0, 3>([&](auto j) {
            if constexpr (tnz(M, i, j)) Z[M].p = fmaf(xi[i], hb[j] * cT[M][pk(i, j)], Z[M].p);
          });
        });
      });
      tau = friction(m, ph, e, geo[G_RS * ne + e], xi[0], u[0], v[0]);
    }
    const bool done = mbar_wait(mdone, commits & 1u);
    ++commits;
    ok &= done;
    tc_fence_after();
    // block-uniform: tcgen05.ld is a warp-wide instruction and the barriers below need every thread
    const bool got = __syncthreads_and(ok) != 0;
    if (!got) ok = false;
    if (got) {
      sfor<0, N / 16>([&](auto c16) {
        float wu[16], wv[16], wx[16];
        tmem_ld16(lane_base + (uint32_t)(16 * c16), wu);
        tmem_ld16(lane_base + (uint32_t)(N + 16 * c16), wv);
        tmem_ld16(lane_base + (uint32_t)(2 * N + 16 * c16), wx);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        sfor<0, 16>([&](auto k) {
          constexpr int M = P.cm[16 * c16 + k], I = P.ci[16 * c16 + k];
          Z[M].add(U[I], V[I], xi[I], wu[k], wv[k], wx[k]);
          if constexpr (I < KL && I != M) Z[I < KL ? I : 0].add(U[M], V[M], xi[M], wu[k], wv[k], wx[k]);
        });
      });
    }
    if (live && got) {
      const float J2 = geo[G_JI2 * ne + e], J3 = geo[G_JI3 * ne + e], rs = geo[G_RS * ne + e];
      const float La = geo[G_JI0 * ne + e] + 0.5f * J2, Lb = geo[G_JI1 * ne + e] + 0.5f * J3;
      float r[3][K];
      sfor<3, K>([&](auto q) { r[0][q] = r[1][q] = r[2][q] = 0.0f; });
      sfor<0, KL>([&](auto M) {
        const float e1 = Z[M].uu + g * Z[M].p, e2 = Z[M].uv, e3 = Z[M].vu, e4 = Z[M].vv + g * Z[M].p;
        const float x0 = La * U[M] + Lb * V[M], s0 = J2 * U[M] + J3 * V[M];
        const float x1 = rs * (La * e1 + Lb * e2), s1 = rs * (J2 * e1 + J3 * e2);
        const float x2 = rs * (La * e3 + Lb * e4), s2 = rs * (J2 * e3 + J3 * e4);
        sfor<3, K>([&](auto q) {
          if constexpr (dxnz(q, M)) {
            r[0][q] = fmaf(cDx[q][M], x0, r[0][q]);
            r[1][q] = fmaf(cDx[q][M], x1, r[1][q]);
            r[2][q] = fmaf(cDx[q][M], x2, r[2][q]);
          }
          if constexpr (dsnz(q, M)) {
            r[0][q] = fmaf(cDs[q][M], s0, r[0][q]);
            r[1][q] = fmaf(cDs[q][M], s1, r[1][q]);
            r[2][q] = fmaf(cDs[q][M], s2, r[2][q]);
          }
        });
      });
      const float gdx = geo[G_GDHX * ne + e], gdy = geo[G_GDHY * ne + e];
      const float dt = (float)stage_dt(stg, m.mem[e]);
      sfor<3, K>([&](auto q) {
        float rq[3] = {r[0][q], r[1][q], r[2][q]};
        const float uq = ph.src ? uh[(0 * (K - 3) + (q - 3)) * n + l] : 0.0f;
        const float vq = ph.src ? uh[(1 * (K - 3) + (q - 3)) * n + l] : 0.0f;
        finish_mode<K>(stg, ph, n, l, q, rq, xi[q], U[q], V[q], uq, vq, gdx, gdy, tau, dt, pe, chN, chO);
      });
    }
    tc_fence_before();
    // the next tile rewrites A and the accumulators; a failed wait anywhere ends the loop for all
    if (__syncthreads_or(!ok)) {
      ok = false;
      break;
    }
  }
  if (!ok && t == 0) atomicOr(status, (unsigned)ST_TIMEOUT);
  // a commit still in flight (a wait that gave up) completes before TMEM is freed
  if (!ok && commits > 0) mbar_wait(mdone, (commits - 1) & 1u);
  if (t == 0) tc_drain(blanded, [&] { return mbar_wait(bfull, 0); });  // the B copy lands before the CTA exits
  tc_fence_before();
  __syncthreads();
  if (w == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tc_cols(K)) : "memory");
  }
}

static int g_nsm_tc = 152;

template <int K>
static int tc_group(cudaStream_t st, const DevMesh& m, const Groups& G, int p, const Phys& ph, const Stage& stg,
                    StateDev cS, StateDev cN, StateDev cO, VelDev u, EdgeFlux fx, unsigned* status,
                    const float* bimg) {
  const int64_t g0 = G.start[p], n = G.start[p + 1] - g0;
  if (n == 0) return 0;
  const unsigned grid = (unsigned)std::min<int64_t>((n + TC_M - 1) / TC_M, (int64_t)g_nsm_tc * tc_ctas(K));
  k_elem_tc<K><<<grid, TC_M, tc_smem(K), st>>>(m, g0, n, ph, stg, cS.cb32, (const float*)cS.ch[p],
                                               (const float*)cN.ch[p], (float*)cO.ch[p], u.ub32,
                                               (const float*)u.uh[p], (const float*)fx.Pf[p], bimg + tc_boff(K), status);
  count_launch();
  SWE_CUDA_OK(cudaGetLastError());
  return 0;
}

int launch_elem_tc(cudaStream_t st, const DevMesh& m, const Groups& G, const Phys& ph, const Stage& stg, StateDev cS,
                   StateDev cN, StateDev cO, VelDev u, EdgeFlux fx, const float* bimg, unsigned* status) {
  int r = tc_group<15>(st, m, G, 4, ph, stg, cS, cN, cO, u, fx, status, bimg);
  if (!r) r = tc_group<10>(st, m, G, 3, ph, stg, cS, cN, cO, u, fx, status, bimg);
  return r;
}

// Self-test of the bounded waits: an mbarrier that nothing arrives on, waited
// for `spins` times; the wait runs out, the kernel sets ST_TIMEOUT and returns.
__global__ void k_wait_selftest(int64_t spins, unsigned* status) {
  __shared__ __align__(8) uint64_t bar;
  const uint32_t a = smem_u32(&bar);
  if (threadIdx.x == 0) {
    mbar_init(a, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    bool ok = false;
    for (int64_t it = 0; it < spins && !ok; ++it) {
      uint32_t r;
      asm volatile(
          "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
          : "=r"(r)
          : "r"(a), "r"(0u)
          : "memory");
      ok = r != 0;
    }
    if (!ok) atomicOr(status, (unsigned)ST_TIMEOUT);
  }
}

int launch_wait_selftest(cudaStream_t st, int64_t spins, unsigned* status) {
  k_wait_selftest<<<1, 32, 0, st>>>(spins, status);
  count_launch();
  SWE_CUDA_OK(cudaGetLastError());
  return 0;
}

// kernel attributes of the current device (once per device and process)
int set_tc_attributes() {
  int dev = 0;
  SWE_CUDA_OK(cudaGetDevice(&dev));
  SWE_CUDA_OK(cudaFuncSetAttribute(k_elem_tc<10>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc_smem(10)));
  SWE_CUDA_OK(cudaFuncSetAttribute(k_elem_tc<15>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc_smem(15)));
  int nsm = 0;
  SWE_CUDA_OK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  if (nsm > 0) g_nsm_tc = nsm;
  return 0;
}

}  // namespace corrtc
}  // namespace swedg
