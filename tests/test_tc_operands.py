"""Host-side checks of the tensor-core operands (precision mode
SWE_PREC_MIXED_TF32), no GPU.

swe_tc_pair_operand, what the kernel contracts with: its rows decode to the
oracle's T[m][i][j] of Eq. (13) in two TF32 parts, its pairs of modes cover every
product once, the products formed as the kernel forms them equal the direct
contraction with T, and it is complete and the same for every caller.

swe_tc_operand_image, the layout for callers with contractions of their own with
the G tensors: it decodes to the oracle's G in two TF32 parts, and GEMMs of
velocity and pressure rows against it reproduce the direct volume contraction of
the momentum rows."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

import oracle as O
from paper_2311_11348_gb300 import build, swedg

DEG = [0, 1, 1, 2, 2, 2, 3, 3, 3, 3, 4, 4, 4, 4, 4]


@pytest.fixture(scope="module")
def lib():
    build.build()
    return swedg.load()


def at(r, c):  # K-major, 128-byte swizzle: 16-byte unit c/4 of row r at unit (c/4) ^ (r%8)
    return (r // 8) * 256 + (r % 8) * 32 + (((c // 4) ^ (r % 8)) * 4) + c % 4


def decode(K, img):
    """the two parts of the image as B[part][k][q][i][j]: row 16 i + q, column
    k K + j of a [16 K][32] operand per part; every other entry zero"""
    nb = 16 * K
    assert len(img) == 2 * nb * 32
    B = np.zeros((2, 2, 16, K, K), np.float32)
    seen = np.zeros(len(img), bool)
    for part in range(2):
        base = part * nb * 32
        for i in range(K):
            for q in range(16):
                for k in range(2):
                    for j in range(K):
                        o = base + at(16 * i + q, k * K + j)
                        B[part, k, q, i, j] = img[o]
                        seen[o] = True
    assert not np.any(img[~seen])  # the padding (q >= K, columns >= 2 K) is zero
    return B


def used(q, i, j):
    """structurally nonzero and not a base triple (the FP64 base owns q, i, j < 3)"""
    dq, di, dj = DEG[q], DEG[i], DEG[j]
    if q < 3 and i < 3 and j < 3:
        return False
    if dq == 0:
        return False
    if dq == 1:
        return i == j
    return di <= dj + dq - 1 and dj <= di + dq - 1


@pytest.mark.parametrize("K", [6, 10, 15])
def test_operand_images_hold_G_split_into_tf32_head_and_tail(lib, K):
    B = decode(K, swedg.tc_operand_image(K))
    G = O.tensors()["G"]
    assert np.all(B.view(np.uint32) & 0x1FFF == 0)  # every part is a TF32 value: no bits below the 10-bit mantissa
    S = B.astype(np.float64).sum(0)
    floor = 1e-14 * np.abs(G).max()  # the library's tables agree with the oracle's to this
    for k in range(2):
        for q in range(16):
            for i in range(K):
                for j in range(K):
                    want = G[k, q, i, j] if (q < K and used(q, i, j)) else 0.0
                    tol = 2.0 ** -21 * abs(want) + floor  # the parts sum to G within 2^-22 |G|
                    assert abs(S[k, q, i, j] - want) <= tol, (k, q, i, j)
                    if want:  # part 0 is G rounded to 10 mantissa bits
                        assert abs(B[0, k, q, i, j] - want) <= 2.0 ** -11 * abs(want) + floor


@pytest.mark.parametrize("K", [6, 10, 15])
def test_gemm_decomposition_reproduces_the_volume_contraction(lib, K):
    """GEMMs of per-element rows (2 K values: the contravariant velocities, or g
    J^-1 xi / 2) against the image, giving W, ZU, ZV [i][q]; then the sums over i
    with the element's U, V, xi, and the bottom term's products with the
    higher elevation modes added apart"""
    rng = np.random.default_rng(K)
    n = 7
    xi, U, V, u, v = (rng.standard_normal((n, K)) for _ in range(5))
    hb = rng.standard_normal((n, 3))
    J = rng.standard_normal((n, 4))
    rs = rng.uniform(0.5, 2.0, n)
    g = 9.81
    B = decode(K, swedg.tc_operand_image(K)).astype(np.float64).sum(0)  # [k][q][i][j], q < 16
    Gm = B[:, :K]
    mask = np.array([[[used(q, i, j) for j in range(K)] for i in range(K)] for q in range(K)])
    assert not np.any(Gm[:, ~mask])
    # direct contraction (non-base triples only), physical gradients through J^-1;
    # the bottom term xi_i h_b_j only with a higher elevation mode i >= 3
    pp = 0.5 * xi
    uc = J[:, [0]] * u + J[:, [1]] * v
    vc = J[:, [2]] * u + J[:, [3]] * v
    Px, Py = (np.array([sum(xi[e, i] * (pp[e, j] + (hb[e, j] if i >= 3 and j < 3 else 0.0)) * Gm[k][:, i, j]
                            for i in range(K) for j in range(K)) for e in range(n)]) for k in range(2))
    rU = rs[:, None] * (np.einsum("qij,ei,ej->eq", Gm[0], U, uc) + np.einsum("qij,ei,ej->eq", Gm[1], U, vc)
                        + g * (J[:, [0]] * Px + J[:, [2]] * Py))
    rV = rs[:, None] * (np.einsum("qij,ei,ej->eq", Gm[0], V, uc) + np.einsum("qij,ei,ej->eq", Gm[1], V, vc)
                        + g * (J[:, [1]] * Px + J[:, [3]] * Py))
    # the operand B[(i, q)][(k, j)] and three A operands of 2 K columns
    Bop = np.zeros((16 * K, 2 * K))
    for i in range(K):
        for q in range(16):
            Bop[16 * i + q, :K] = B[0, q, i, :]
            Bop[16 * i + q, K:] = B[1, q, i, :]
    Aw = np.hstack([uc, vc])
    Au = g * np.hstack([J[:, [0]] * pp, J[:, [2]] * pp])
    Av = g * np.hstack([J[:, [1]] * pp, J[:, [3]] * pp])
    W, ZU, ZV = ((A @ Bop.T).reshape(n, K, 16) for A in (Aw, Au, Av))
    ex = np.einsum("qij,ei,ej->eq", Gm[0, :, 3:, :3], xi[:, 3:], hb)
    ey = np.einsum("qij,ei,ej->eq", Gm[1, :, 3:, :3], xi[:, 3:], hb)
    gU = np.einsum("ei,eiq->eq", U, W) + np.einsum("ei,eiq->eq", xi, ZU)
    gV = np.einsum("ei,eiq->eq", V, W) + np.einsum("ei,eiq->eq", xi, ZV)
    gU = rs[:, None] * (gU[:, :K] + g * (J[:, [0]] * ex + J[:, [2]] * ey))
    gV = rs[:, None] * (gV[:, :K] + g * (J[:, [1]] * ex + J[:, [3]] * ey))
    tol = 1e-9 * max(np.abs(rU).max(), np.abs(rV).max())
    assert np.abs(gU - rU).max() <= tol
    assert np.abs(gV - rV).max() <= tol
    assert np.abs(rU[:, 3:]).max() > 0.1  # the test exercises nonzero higher rows


def pair_rows(K):
    """columns' rows of T by part [2][N][16], the columns' pairs and the others"""
    img, cols, thin = swedg.tc_pair_operand(K)
    B = np.array([[[img[at(c, 16 * part + j)] for j in range(16)] for c in range(len(cols))] for part in range(2)])
    assert np.count_nonzero(img) == np.count_nonzero(B)
    return B, cols, thin


@pytest.mark.parametrize("K", [10, 15])
def test_pair_operand_holds_T_split_into_tf32_head_and_tail(lib, K):
    B, cols, _ = pair_rows(K)
    T = O.tensors()["T"]
    want = np.zeros((len(cols), 16))
    want[:, :K] = T[cols[:, 0], cols[:, 1], :K]
    floor = 1e-13 * np.abs(T).max()  # structural zeros: the oracle's quadrature noise
    assert np.all(B.view(np.uint32) & 0x1FFF == 0)
    assert np.all(np.abs(B[0] - want) <= 2.0 ** -11 * np.abs(want) + floor)
    assert np.all(np.abs(B.astype(np.float64).sum(0) - want) <= 2.0 ** -22 * np.abs(want) + floor)
    assert np.all(np.abs(want[np.abs(B[0]) == 0]) <= floor)


@pytest.mark.parametrize("K", [10, 15])
def test_pairs_cover_every_product_of_the_higher_modes_once(lib, K):
    """the pairs (m, i), 1 <= m <= i, m of lower degree, with a nonzero T[m][i][j]; a constant mode needs none"""
    _, cols, thin = pair_rows(K)
    KL = {10: 6, 15: 10}[K]
    T = O.tensors()["T"]
    nz = np.abs(T) > 1e-13 * np.abs(T).max()
    pairs = [tuple(p) for p in np.vstack([cols, thin])]
    assert len(set(pairs)) == len(pairs)
    assert set(pairs) == {(m, i) for m in range(1, KL) for i in range(m, K) if nz[m, i, :K].any()}
    delta = np.sqrt(2.0) * np.eye(K)
    assert np.abs(T[0, :K, :K] - delta).max() < 1e-13 and np.abs(T[:K, 0, :K] - delta).max() < 1e-13


@pytest.mark.parametrize("K", [10, 15])
def test_products_as_the_kernel_forms_them(lib, K):
    """Z_m = sum_ij T[m][i][j] U_i u_j from the columns' GEMM, the other pairs and the constant mode, a pair of
    two modes below the element's degree serving both"""
    B, cols, thin = pair_rows(K)
    KL = {10: 6, 15: 10}[K]
    T = O.tensors()["T"]
    rng = np.random.default_rng(K)
    U, u = rng.standard_normal((2, 5, K))
    W = np.hstack([u @ B.astype(np.float64).sum(0)[:, :K].T, u @ T[thin[:, 0], thin[:, 1], :K].T])
    f0 = np.sqrt(2.0)
    Z = f0 * U[:, :1] * u[:, :KL]
    Z[:, 0] = f0 * (U * u).sum(1)
    for c, (m, i) in enumerate(np.vstack([cols, thin])):
        Z[:, m] += U[:, i] * W[:, c]
        if i < KL and i != m:
            Z[:, i] += U[:, m] * W[:, c]
    want = np.einsum("mij,ei,ej->em", T[:KL, :K, :K], U, u)
    # each entry of T to within 2^-22; the sum of the terms' magnitudes bounds the products' error
    bound = 2.0 ** -22 * np.einsum("mij,ei,ej->em", np.abs(T[:KL, :K, :K]), np.abs(U), np.abs(u))
    assert np.all(np.abs(Z - want) <= bound)


def test_pair_operand_is_written_once(lib):
    """contexts upload it without a lock: every caller, from any thread, gets the complete image"""
    want = {K: swedg.tc_pair_operand(K)[0] for K in (10, 15)}

    def differ(i):
        K = (10, 15)[i % 2]
        return sum(not np.array_equal(swedg.tc_pair_operand(K)[0], want[K]) for _ in range(2000))

    with ThreadPoolExecutor(8) as ex:  # the library call runs without the interpreter's lock
        assert sum(ex.map(differ, range(8))) == 0
