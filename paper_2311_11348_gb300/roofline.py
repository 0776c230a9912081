"""Algorithmic operation counts of the libswedg kernel families (bench roofline).

The counts mirror the arithmetic of the kernels (same loops, the same
compile-time sparsity predicates of the reference tensors): an FMA counts as
2 floating-point operations, an add, multiply, division or square root as 1;
loads, conversions and selects count 0.  They are the "algorithmic flops per
unit" of the roofline that bench.py reports:

  family      unit                         arithmetic       count per unit
  usolve      element (p<=1 / p>=2)        FP64 / corr      USOLVE_P1 / usolve_flops(K)
  edge_base   edge with p <= 1 sides       FP64             EDGE_BASE
  elem_base   element                      FP64             ELEM_BASE (first stage ELEM_BASE_EULER)
  edge_corr   edge with max(p_L,p_R) >= 2  corr type        edge_corr_flops(K_L, K_R, pmax, fp64)
  elem_corr   element p >= 2               corr type        elem_corr_flops(K)
  vol_tc      element p >= 3               TF32 tensor      vol_tc_flops(K)

"corr type" is FP64 in the FP64 mode and FP32 in both mixed modes (whose
correction edges also compute the FP64 base flux, EDGE_BASE more).  The
velocity solve of a p >= 2 element also forms the volume terms of the degree-1
test modes.  In the tensor-core mode ("tf32") vol_tc is the element update of
the orders 3 and 4, counted by the MMA work it issues: three GEMMs (u, v, xi / 2)
against the columns of T, each in three TF32 passes (head x head, head x tail,
tail x head) over the 16 reduction columns; elem_corr is then the order 2.
"""
from __future__ import annotations

import numpy as np

DEG = [0, 1, 1, 2, 2, 2, 3, 3, 3, 3, 4, 4, 4, 4, 4]
KP = [1, 3, 6, 10, 15]
SM_COUNT = 152
SM_MAX_GHZ = 2.07
# FP64 pipe of a GB300: 2 DFMA = 4 flop per clock per SM (measured 1.19 TFLOP/s at 1.92 GHz)
FP64_PEAK_TFLOPS = SM_COUNT * 4 * SM_MAX_GHZ / 1e3
# FP32 pipe: 128 FMA = 256 flop per clock per SM
FP32_PEAK_TFLOPS = SM_COUNT * 256 * SM_MAX_GHZ / 1e3
# dense TF32 : BF16 tensor rate of the part (1.1 : 2.25 PFLOP/s nominal)
TF32_OVER_BF16 = 1.1 / 2.25

LEG = [0, 1, 0, 2, 1, 0, 3, 2, 1, 0, 4, 3, 2, 1, 0]  # Legendre index of each mode

USOLVE_P1 = 70   # the 3 x 3 solve with the entries the orthonormal basis fixes left out
EDGE_BASE = 152
ELEM_BASE = 208  # a stage with the full SSP-RK combination
ELEM_BASE_EULER = 181  # the first stage (c + dt r)


def npts(pm):
    return 2 if pm <= 1 else (3 * pm + 2) // 2


def _tri(a, b, c):
    return a <= b + c and b <= a + c and c <= a + b


def tnz(n, i, j):
    """the entries T[n][i][j] that the degrees and the Legendre indices leave nonzero"""
    if n == 0:
        return i == j
    if i == 0:
        return n == j
    if j == 0:
        return n == i
    return _tri(DEG[n], DEG[i], DEG[j]) and _tri(LEG[n], LEG[i], LEG[j]) and (LEG[n] + LEG[i] + LEG[j]) % 2 == 0


def dxnz(q, m):
    return DEG[m] < DEG[q] and LEG[m] < LEG[q] and (LEG[q] - LEG[m]) % 2 == 1


def dsnz(q, m):
    return DEG[m] < DEG[q] and LEG[m] <= LEG[q] and (LEG[q] - LEG[m]) % 2 == 0


def ktr(i, j):
    return KP[max(DEG[i], DEG[j])]


def usolve_flops(K):
    """truncated K x K assembly, LDL^T, two right-hand sides, and the volume
    terms of the test modes 1 and 2 (five sums over the higher modes)"""
    f = 3
    for j in range(K):
        for i in range(j + 1):
            f += 2 * sum(1 for n in range(ktr(i, j)) if tnz(n, i, j))
    for j in range(K):
        f += 3 * j + 1 + (K - 1 - j) * 2 * j
    f += 2 * (K * (K - 1) + K + K * (K - 1) + K)
    return f + 10 * (K - 3) + 18


def elem_corr_flops(K):
    """the products of the modes below the element's degree, their combination
    by the test modes q >= 3, source, the three edges' projected fluxes and the
    RK combination"""
    KL = KP[DEG[K - 1] - 1]
    f = 8
    for m in range(KL):
        for i in range(K):
            nz = [j for j in range(K) if tnz(m, i, j)]
            if nz:
                f += 4 * len(nz) + 2 * sum(1 for j in nz if j < i) + (3 if i in nz else 0) + 10
        f += 4 + 18
    for q in range(3, K):
        f += 6 * sum(dxnz(q, m) + dsnz(q, m) for m in range(KL)) + 2 + 4 + 3 * 3 + 3 * 5
    return f


def vol_tc_flops(K):
    """TF32 MMA flops per element (row of the GEMMs): three GEMMs of N = 80 (K =
    15) or 32 columns over two steps of 8, each in three passes (hh, ht, th); 2
    flops per multiply-add"""
    return 3 * 3 * 2 * (80 if K == 15 else 32) * 8 * 2


def edge_corr_flops(KL, KR, pm, fp64):
    """Legendre coefficients of both sides (xi, U, V, w), the linear row, the jump
    terms and the products with h_b by coefficients, the products at npts(pm) points, their
    moments, and the projections onto the higher test modes of each side"""
    N, L = npts(pm), pm + 1
    f = 60
    for K in (KL, KR):
        f += 3 * K + 8 * sum(DEG[i] + 1 for i in range(K)) + 4 * L
        if K >= 6:
            f += 9 * L + 6 * sum(DEG[q] + 1 for q in range(3, K))
    ev = 6 if pm == 2 else 9 if pm == 3 else 10  # a field at a pair of points
    f += L * (14 + 10) + (N // 2) * (8 * ev) + N * (14 if fp64 else 34) + 4 * L * ((N + 1) // 2)
    return f + (0 if fp64 else 68)


def family_flops(orders, fam, nedge=None, mode="mixed"):
    """flops per SSP-RK3 step (3 stages) of one kernel family on an order map
    (i.i.d. orders: an edge's pmax is the larger of two independent draws)"""
    p = np.asarray(orders)
    ne = len(p)
    n = [int((p == q).sum()) for q in range(5)]
    nedge = nedge or int(round(1.5 * ne))
    cdf = np.cumsum(np.array(n, float) / max(ne, 1))
    st = 3
    if fam == "elem_base":
        return ((st - 1) * ELEM_BASE + ELEM_BASE_EULER) * ne
    if fam == "edge_base":
        return st * EDGE_BASE * nedge * cdf[1] ** 2
    if fam == "dt":
        return 0
    if fam == "usolve":
        return st * (n[1] * USOLVE_P1 + n[0] * 6 + sum(n[q] * usolve_flops(KP[q]) for q in (2, 3, 4)))
    if fam == "elem_corr":
        return st * sum(n[q] * elem_corr_flops(KP[q]) for q in ((2,) if mode == "tf32" else (2, 3, 4)))
    if fam == "vol_tc":
        return st * sum(n[q] * vol_tc_flops(KP[q]) for q in (3, 4))
    if fam == "edge_corr":
        tot = 0.0
        for pm in (2, 3, 4):
            pr = cdf[pm] ** 2 - cdf[pm - 1] ** 2
            tot += pr * nedge * edge_corr_flops(KP[pm], KP[max(1, pm - 1)], pm, mode == "fp64")
        return st * tot
    return None


def edge_corr_fp64_flops(orders, nedge=None):
    """FP64 flops per SSP-RK3 step of the base flux that the correction edge
    kernels carry (edges with max(p_L, p_R) >= 2)"""
    p = np.asarray(orders)
    nedge = nedge or int(round(1.5 * len(p)))
    return 3 * EDGE_BASE * nedge * (1.0 - float((p <= 1).mean()) ** 2)


def pipe_of(fam, mode):
    """which arithmetic pipe bounds a family: 'fp64', 'fp32' or 'tensor'"""
    if fam == "vol_tc":
        return "tensor"
    if fam in ("edge_corr", "elem_corr") and mode in ("mixed", "tf32"):
        return "fp32"
    return "fp64"
