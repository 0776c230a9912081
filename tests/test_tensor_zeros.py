"""The structural zeros of the reference tensors that the correction kernels leave
out at compile time (degree and Legendre-index rules), checked against the
library's tensors: every dropped entry is a zero, and G follows from D and T."""
import numpy as np
import pytest

swedg = pytest.importorskip("paper_2311_11348_gb300.swedg")

MODES = [(d - b, b) for d in range(5) for b in range(d + 1)]
DEG = [a + b for a, b in MODES]
LEG = [a for a, b in MODES]


def tri(a, b, c):
    return a <= b + c and b <= a + c and c <= a + b


def tnz(n, i, j):
    if n == 0:
        return i == j
    if i == 0:
        return n == j
    if j == 0:
        return n == i
    return tri(DEG[n], DEG[i], DEG[j]) and tri(LEG[n], LEG[i], LEG[j]) and (LEG[n] + LEG[i] + LEG[j]) % 2 == 0


def test_dropped_entries_are_zero():
    D, G, T = swedg.reference_tensors()
    keep = np.array([[[tnz(n, i, j) for j in range(15)] for i in range(15)] for n in range(15)])
    # quadrature noise of the largest entries (about 12 for T, 60 for D)
    assert np.abs(T[~keep]).max() < 1e-13 * np.abs(T).max()
    assert int(keep[:10].sum()) == 546
    dx, ds = D[0], D[1] - 0.5 * D[0]
    kx = np.array([[DEG[m] < DEG[q] and LEG[m] < LEG[q] and (LEG[q] - LEG[m]) % 2 == 1 for m in range(15)] for q in range(15)])
    ks = np.array([[DEG[m] < DEG[q] and LEG[m] <= LEG[q] and (LEG[q] - LEG[m]) % 2 == 0 for m in range(15)] for q in range(15)])
    assert np.abs(dx[~kx]).max() < 1e-13 * np.abs(dx).max()
    assert np.abs(ds[~ks]).max() < 1e-13 * np.abs(dx).max()


def test_g_is_the_derivative_expansion_times_t():
    """d_k phi_q = sum_m D_k[q][m] phi_m, so G_k[q][i][j] = sum_m D_k[q][m] T[m][i][j]"""
    D, G, T = swedg.reference_tensors()
    assert np.abs(np.einsum("kqm,mij->kqij", D, T) - G).max() < 1e-13 * np.abs(G).max()
