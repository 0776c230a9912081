"""GPU tests of the correction kernels' dispatch at the sizes where it changes
(rule on the group size) and at ragged ends, against the FP64 oracle.

Tolerances, of the largest entry of each field: FP64 1e-12 (the bound of the
other right-hand side tests); FP32 100 * 2^-24, i.e. one rounding for each of
the about 100 terms an entry sums over its volume and edge parts."""
import os
import sys

import numpy as np
import pytest

sys.path.insert(0, os.path.join(os.path.dirname(__file__), "..", "oracle"))
import oracle as O  # noqa: E402
from paper_2311_11348_gb300 import inputs, swedg  # noqa: E402

pytestmark = pytest.mark.gpu
TOL = {swedg.PREC_FP64: 1e-12, swedg.PREC_MIXED_FP32: 100 * 2.0**-24, swedg.PREC_MIXED_TF32: 100 * 2.0**-24}


def rect(nx, ny):
    """the triangles of nx x ny squares out of a larger split-square mesh, so that any count can be made"""
    n = max(nx, ny)
    xy, tri = inputs.split_square_mesh(n, 1e3, jitter=0.2, seed=7)
    return xy, tri.reshape(n, n, 2, 3)[:nx, :ny].reshape(-1, 3)


def rhs_errors(orders_of, nx, ny, prec, **kw):
    xy, tri = rect(nx, ny)
    hv = inputs.fourier_bathymetry(xy, 1e3, lo=10.0, hi=50.0, seed=2)
    orders = orders_of(len(tri))
    m = O.Mesh(xy, tri, hv, orders)
    c = m.project_state(lambda x, y: (0.3 * np.exp(-((x - 400) ** 2 + (y - 600) ** 2) / 4e4),
                                      2.0 + np.sin(x / 150), 1.0 + np.cos(y / 130)))
    ref = m.rhs(O.Params(g=9.81, **kw), c)
    s = swedg.Solver(g=9.81, precision=prec, friction=(kw.get("fric_lin", 0.0), kw.get("fric_quad", 0.0)),
                     f_c=kw.get("f_c", 0.0))
    s.set_mesh(xy, tri)
    s.set_bathymetry(hv)
    s.set_orders(orders)
    out = s.rhs(c)
    s.close()
    return [float(np.abs(out[f] - ref[f]).max() / np.abs(ref[f]).max()) for f in range(3)]


@pytest.mark.parametrize("p,nx,ny", [(4, 50, 60), (4, 51, 59), (3, 64, 78), (3, 70, 72), (2, 100, 100), (2, 99, 102)])
def test_element_kernel_forms_meet_at_the_size_rule(p, nx, ny):
    """groups just below and above K(p-1) n = 60,000, where the FP32 element update changes its form"""
    for prec in (swedg.PREC_MIXED_FP32, swedg.PREC_MIXED_TF32):
        err = rhs_errors(lambda n: np.full(n, p, np.int8), nx, ny, prec)
        assert max(err) < TOL[prec], err


@pytest.mark.parametrize("prec", [swedg.PREC_FP64, swedg.PREC_MIXED_FP32, swedg.PREC_MIXED_TF32])
@pytest.mark.parametrize("nx,ny", [(1, 1), (3, 5), (4, 4), (11, 3)])
def test_correction_kernels_on_ragged_groups(prec, nx, ny):
    """every order at once, groups of a few elements and around a warp, all source terms"""
    err = rhs_errors(lambda n: (np.arange(n) % 5).astype(np.int8), nx, ny, prec, fric_lin=1e-4, fric_quad=0.009, f_c=1e-2)
    assert max(err) < TOL[prec], err


@pytest.mark.parametrize("prec,p,sizes", [(swedg.PREC_MIXED_FP32, 4, [(50, 60), (40, 50)]),
                                          (swedg.PREC_MIXED_FP32, 3, [(64, 78), (50, 60)]),
                                          (swedg.PREC_MIXED_FP32, 2, [(100, 100), (60, 70)]),
                                          (swedg.PREC_FP64, 4, [(30, 50), (20, 30)]),
                                          (swedg.PREC_FP64, 4, [(69, 70), (20, 30)]),
                                          (swedg.PREC_FP64, 1, [(60, 68), (20, 30)]),
                                          (swedg.PREC_MIXED_FP32, 2, [(32, 32), (20, 30)]),
                                          (swedg.PREC_FP64, 1, [(1, 1), (60, 70)])])
def test_member_alone_and_in_a_union_across_the_size_rules_bitwise(prec, p, sizes):
    """alone the first member's group runs one form of the element update or of the velocity solve, in the union
    another (FP32: K(p-1) n = 60,000; FP64, order 4: 3,000 and 9,728 elements; base
    element update: 8,192 elements, 2,048 beside correction kernels), with all source terms"""
    from paper_2311_11348_gb300.ensemble import Ensemble
    members, states = [], []
    for k, (nx, ny) in enumerate(sizes):
        n = max(nx, ny)
        xy, tri = inputs.split_square_mesh(n, 1e3, jitter=0.2, seed=7 + k)
        tri = np.ascontiguousarray(tri.reshape(n, n, 2, 3)[:nx, :ny].reshape(-1, 3))
        members.append(dict(xy=xy, tri=tri, hv=inputs.fourier_bathymetry(xy, 1e3, lo=10.0, hi=50.0, seed=2 + k),
                            orders=np.full(len(tri), p, np.int8)))
        rng = np.random.default_rng(5 + k)
        K = (p + 1) * (p + 2) // 2
        c = np.zeros((3, swedg.KMAX, len(tri)))
        c[:, :K] = rng.standard_normal((3, K, len(tri))) * 0.1
        states.append(c)
    out = []
    for ms, cs in ((members[:1], states[:1]), (members, states)):
        e = Ensemble(ms, g=9.81, rk_order=3, precision=prec, friction=(1e-4, 0.009), f_c=1e-2)
        e.set_states(cs)
        e.run(2)
        out.append(e.states()[0])
        e.close()
    assert np.isfinite(out[0]).all() and np.array_equal(out[0], out[1])


@pytest.mark.parametrize("nx,ny", [(1, 4), (1, 5), (30, 50), (31, 49)])
def test_velocity_solve_forms_meet_at_the_size_rule(nx, ny):
    """FP64, order 4: one full block of the sixteen-lane form (8 elements), one more, its largest group (3,000)
    and a larger one"""
    err = rhs_errors(lambda n: np.full(n, 4, np.int8), nx, ny, swedg.PREC_FP64)
    assert max(err) < TOL[swedg.PREC_FP64], err


@pytest.mark.parametrize("prec,eps", [(swedg.PREC_FP64, 2.0**-53), (swedg.PREC_MIXED_FP32, 2.0**-24),
                                      (swedg.PREC_MIXED_TF32, 2.0**-24)])
def test_uniform_current_over_deep_water_keeps_the_jump_term_out_of_the_products(prec, eps):
    """A uniform current over a flat bottom has a zero right-hand side away from the walls.  On equal squares both
    sides of an edge have the same traces to the bit, so lambda (U_L - U_R) vanishes and what is left are the
    roundings of the terms U w, about 100 each: 100 eps |U| |u| perimeter / s.  Products of U with w +- lambda would
    leave eps |U| lambda |E| / s, here 9,000 eps |U| |u| |E| / s."""
    n, h, u = 16, 2000.0, (0.013, 0.007)
    xy, tri = inputs.split_square_mesh(n, 1024.0, jitter=0.0, seed=1)
    nbr, _ = swedg.mesh_adjacency(xy, tri)
    orders = (np.arange(len(tri)) % 3 + 2).astype(np.int8)
    s = swedg.Solver(g=9.81, precision=prec)
    s.set_mesh(xy, tri)
    s.set_bathymetry(np.full(len(xy), h))
    s.set_orders(orders)
    se = 64.0  # sqrt det J
    c = np.zeros((3, swedg.KMAX, len(tri)))
    c[1, 0], c[2, 0] = (h * ui * se / np.sqrt(2.0) for ui in u)
    r = s.rhs(c)[1:, 3:, (nbr >= 0).all(axis=1)]
    s.close()
    speed = float(np.hypot(*u))
    bound = 100 * eps * h * speed * speed * (2 + np.sqrt(2.0)) * 64.0 / se
    print(prec, float(np.abs(r).max()) / bound)
    assert np.abs(r).max() <= bound


@pytest.mark.parametrize("prec,eps", [(swedg.PREC_FP64, 2.0**-53), (swedg.PREC_MIXED_FP32, 2.0**-24),
                                      (swedg.PREC_MIXED_TF32, 2.0**-24)])
def test_small_higher_elevation_modes_over_deep_water_keep_their_digits(prec, eps):
    """Still water over a flat bottom with a constant elevation a and tiny higher modes: the higher momentum rows are
    linear in those modes with the factor g (h + a), so the rows for a = 1 and a = 0 differ by (h + a) / h.  On equal
    squares the jump of a vanishes to the bit and the roundings left are those of g a^2 / 2, about 100 of them:
    100 eps g a^2 perimeter / s.  Higher modes taken as whole minus constant would leave eps g h a |E| / s."""
    n, h, se = 16, 8192.0, 64.0  # se = sqrt det J
    xy, tri = inputs.split_square_mesh(n, 1024.0, jitter=0.0, seed=1)
    orders = (np.arange(len(tri)) % 3 + 2).astype(np.int8)
    s = swedg.Solver(g=9.81, precision=prec)
    s.set_mesh(xy, tri)
    s.set_bathymetry(np.full(len(xy), h))
    s.set_orders(orders)
    K = (orders + 1) * (orders + 2) // 2
    c = np.zeros((3, swedg.KMAX, len(tri)))
    c[0, 3:] = 2.0**-20 * np.random.default_rng(4).uniform(-1, 1, (12, len(tri))) * se
    c[0] *= np.arange(swedg.KMAX)[:, None] < K[None]
    c[0] = c[0].astype(np.float32)  # held exactly in every mode
    r0 = s.rhs(c)[1:, 3:]
    c[0, 0] = se / np.sqrt(2.0)
    r1 = s.rhs(c)[1:, 3:]
    s.close()
    bound = 100 * eps * 9.81 * (2 + np.sqrt(2.0)) * 64.0 / se
    d = np.abs(r1 - r0 * (1.0 + 1.0 / h)).max()
    print(prec, d / bound, np.abs(r0).max() / bound)
    assert d <= bound


@pytest.mark.parametrize("prec", [swedg.PREC_FP64, swedg.PREC_MIXED_FP32, swedg.PREC_MIXED_TF32])
def test_still_water_has_elevation_rows_of_fp64_rounding(prec):
    """still water with a constant elevation a over a varying bottom: the elevation flux is lambda times the jump of
    a, whose P1 part every mode forms in FP64: about 100 roundings, 100 2^-53 lambda a perimeter / s"""
    xy, tri = inputs.split_square_mesh(16, 1024.0, jitter=0.2, seed=7)
    hv = inputs.fourier_bathymetry(xy, 1024.0, lo=500.0, hi=4000.0, seed=2)
    orders = (np.arange(len(tri)) % 5).astype(np.int8)
    a, b = xy[tri[:, 1]] - xy[tri[:, 0]], xy[tri[:, 2]] - xy[tri[:, 0]]
    se = np.sqrt(a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0])
    s = swedg.Solver(g=9.81, precision=prec)
    s.set_mesh(xy, tri)
    s.set_bathymetry(hv)
    s.set_orders(orders)
    c = np.zeros((3, swedg.KMAX, len(tri)))
    c[0, 0] = se / np.sqrt(2.0)
    r = np.abs(s.rhs(c)[0]).max(axis=0)
    s.close()
    perimeter = sum(np.linalg.norm(xy[tri[:, (k + 1) % 3]] - xy[tri[:, k]], axis=1) for k in range(3))
    assert np.all(r <= 100 * 2.0**-53 * np.sqrt(9.81 * 4001.0) * perimeter / se)


@pytest.mark.parametrize("prec", [swedg.PREC_FP64, swedg.PREC_MIXED_FP32, swedg.PREC_MIXED_TF32])
def test_rhs_parts_without_higher_coefficients_has_no_correction_of_the_base_elevation(prec):
    """the elevation flux is linear, so with every coefficient of degree >= 2 zero both parts form the same base rows"""
    xy, tri = inputs.split_square_mesh(12, 1e3, jitter=0.2, seed=7)
    orders = (np.arange(len(tri)) % 5).astype(np.int8)
    s = swedg.Solver(g=9.81, precision=prec)
    s.set_mesh(xy, tri)
    s.set_bathymetry(inputs.fourier_bathymetry(xy, 1e3, lo=10.0, hi=50.0, seed=2))
    s.set_orders(orders)
    rng = np.random.default_rng(1)
    c = np.zeros((3, swedg.KMAX, len(tri)))
    c[:, 0] = rng.standard_normal((3, len(tri)))
    c[:, 1:3, orders > 0] = rng.standard_normal((3, 2, int((orders > 0).sum())))
    base, corr = s.rhs_parts(c)
    whole = s.rhs(c)
    s.close()
    assert not corr[0, :3].any()
    assert np.array_equal(base[0, :3], whole[0, :3])
