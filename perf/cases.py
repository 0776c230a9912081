"""Performance cases: the work a user of this framework has it do.

Every case makes a seeded mesh, bathymetry, order map and smooth initial
state, and runs them through the package's public calls (`swedg.Solver`,
`ensemble.Ensemble`, `swedg.rhs_p1_noalloc`).  The sizes and settings are
those of the repository's own workloads, tests and benchmark (512 to
2,097,152 triangles, orders 0..4, FP64, mixed and tensor-core modes,
SSP-RK2/3, tide, friction and Coriolis, ensembles, adaptivity, streaming).

`exact` evaluates the same scheme in 64 bits with plain torch: the weak form
by Gauss quadrature on every element and edge.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2311_11348_gb300 import ensemble, swedg

KMAX = 15
DEG = [0, 1, 1, 2, 2, 2, 3, 3, 3, 3, 4, 4, 4, 4, 4]
PREC = {"fp64": swedg.PREC_FP64, "mixed": swedg.PREC_MIXED_FP32, "tf32": swedg.PREC_MIXED_TF32}
G = 9.81


def _case(name, kind, setting, nx, ny, orders, prec, steps, rk=3, **more):
    """orders: percent of the elements at p = 0, 1, 2, 3, 4"""
    c = dict(name=name, kind=kind, setting=setting, nx=nx, ny=ny, orders=orders, prec=prec, steps=steps, rk=rk,
             source=False, shape="", members=1, every=0)
    c.update(more)
    return c


def listed():
    return [
        # the allocation-free right-hand side inside another application's time loop
        _case("noalloc_20k", "noalloc", "ocean", 100, 100, "0,100,0,0,0", "fp64", 0),
        # the smallest simulation: 512 triangles, p = 1, FP64, where latency and launches count
        _case("unit_p1_fp64", "run", "unit", 16, 16, "0,100,0,0,0", "fp64", 20, rk=2),
        # a small request of a serving loop, and the step sizes of an interactive run
        _case("request_5k_mixed", "run", "ocean", 51, 49, "0,40,30,20,10", "mixed", 20),
        # one right-hand side for a caller's own time integrator, every order and source term
        _case("rhs_sources_fp64", "rhs", "shelf", 181, 183, "10,30,30,20,10", "fp64", 0, source=True),
        # the ocean workload as the benchmark runs it (its tuned launch shape)
        _case("ocean_mixed", "run", "ocean", 256, 256, "0,70,20,10,0", "mixed", 5, shape="0,128,128,64,1,2"),
        # the same in FP64, default launch shape
        _case("ocean_fp64", "run", "ocean", 256, 256, "0,70,20,10,0", "fp64", 2),
        # states streamed through one context from pinned host memory
        _case("ocean_stream", "stream", "ocean", 256, 256, "0,70,20,10,0", "mixed", 1, members=4),
        # dynamic adaptivity: the indicator and the regrouping between runs (FP64: every decision well defined)
        _case("ocean_adaptive", "adapt", "ocean", 256, 256, "0,70,20,10,0", "fp64", 10, every=5),
        # the statically adaptive p1-2 dam break in the sparse regime (1/32 of the elements at p = 2)
        _case("dam_break_mixed", "run", "dam", 512, 512, "0,96.875,3.125,0,0", "mixed", 2),
        # many independent meshes of uneven sizes in one context
        _case("ensemble_mixed", "ensemble", "ocean", 160, 160, "0,40,30,20,10", "mixed", 2, members=12),
        # tide-driven shelf, odd size, FP64 correction of every order
        _case("shelf_fp64", "run", "shelf", 301, 307, "0,40,30,20,10", "fp64", 1),
        # the largest single mesh, tensor-core correction
        _case("shelf_tf32", "run", "shelf", 1024, 1024, "0,40,30,20,10", "tf32", 2),
    ]


def draw(rng: random.Random):
    """one more case: any kind, 100 triangles up to about a million, odd sizes, any order mix and mode"""
    kind = rng.choice(["noalloc", "run", "run", "run", "rhs", "stream", "adapt", "ensemble"])
    top = {"noalloc": 32e3, "run": 5e5, "rhs": 2e5, "stream": 1e5, "adapt": 1e5, "ensemble": 5e4}[kind]
    cells = math.exp(rng.uniform(math.log(50.0), math.log(top)))
    nx = max(3, int(math.sqrt(cells) * rng.uniform(0.8, 1.25)))
    ny = max(3, int(cells / nx))
    prec = rng.choice(["fp64", "mixed", "mixed", "tf32"])
    orders = rng.choice(["0,100,0,0,0", "0,70,20,10,0", "0,40,30,20,10", "0,97,3,0,0", "10,30,30,20,10", "0,0,100,0,0"])
    setting = rng.choice(["ocean", "shelf", "dam", "unit"])
    steps = rng.choice([1, 2, 5]) if cells < 6e4 else 1
    if kind == "noalloc":
        return _drawn(kind, setting, nx, ny, "0,100,0,0,0", "fp64", 0)
    if kind == "rhs":
        return _drawn(kind, setting, nx, ny, orders, prec, 0, source=rng.random() < 0.5)
    if kind == "stream":
        return _drawn(kind, setting, nx, ny, orders, prec, 1, members=rng.choice([2, 3, 4]))
    if kind == "adapt":
        return _drawn(kind, "ocean", nx, ny, "0,70,20,10,0", "fp64", 6, every=3)
    if kind == "ensemble":
        return _drawn(kind, "ocean", nx, ny, orders, prec, 2, members=rng.randint(3, 12))
    return _drawn(kind, setting, nx, ny, orders, prec, steps, rk=rng.choice([2, 3]), source=rng.random() < 0.3,
                  shape=rng.choice(["", "", "0,128,128,64,1,2"]))


def _drawn(*a, **kw):
    c = _case("", *a, **kw)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _params(case):
    """the scheme's parameters that go into the solver"""
    tide = (1.0, 44714.0, 0.3) if case["setting"] == "shelf" else (0.0, 0.0, 0.0)
    return dict(g=G, cfl=0.1, rk_order=case["rk"], tide=tide,
                friction=(1e-4, 0.009) if case["source"] else (0.0, 0.0), f_c=1e-4 if case["source"] else 0.0)


def _mesh(nx, ny, width, jitter, rng):
    """nx x ny squares, each cut into two counter-clockwise triangles, interior vertices jittered"""
    h = width / nx
    i, j = np.meshgrid(np.arange(nx + 1), np.arange(ny + 1), indexing="ij")
    xy = np.stack([i.ravel() * h, j.ravel() * h], axis=1).astype(np.float64)
    d = rng.uniform(-jitter * h, jitter * h, size=xy.shape)
    inner = (i.ravel() > 0) & (i.ravel() < nx) & (j.ravel() > 0) & (j.ravel() < ny)
    xy[inner] += d[inner]
    a, b = np.meshgrid(np.arange(nx), np.arange(ny), indexing="ij")
    a, b = a.ravel(), b.ravel()
    v00 = a * (ny + 1) + b
    v10 = v00 + ny + 1
    tri = np.empty((2 * nx * ny, 3), np.int32)
    tri[0::2] = np.stack([v00, v10, v10 + 1], axis=1)
    tri[1::2] = np.stack([v00, v10 + 1, v00 + 1], axis=1)
    return xy, tri


def _waves(rng, count, kmax):
    """seeded smooth field on [0,1]^2 (several cosines), scaled to about [-1, 1]"""
    k = rng.integers(-kmax, kmax + 1, size=(count, 2)) + np.array([0.5, 0.25])
    amp = np.linalg.norm(k, axis=1) ** -1.5
    return 2 * math.pi * k, amp / (1.5 * np.sqrt(np.sum(amp ** 2))), rng.uniform(0, 2 * math.pi, count)


def _field(w, x, y):
    s = torch.zeros_like(x)
    for k, a, ph in zip(*w):
        s += float(a) * torch.cos(float(k[0]) * x + float(k[1]) * y + float(ph))
    return s


def _one_mesh(case, nx, ny, rng):
    """mesh, boundary tags, depths at the vertices, orders and the smooth initial fields of one member"""
    setting = case["setting"]
    width = {"unit": 1.0, "ocean": 1e5, "shelf": 5e5, "dam": 1e4}[setting]
    xy, tri = _mesh(nx, ny, width, 0.0 if setting == "unit" else 0.2, rng)
    p = torch.from_numpy(xy).to(_dev()) / width
    x, y = p[:, 0], p[:, 1]
    top = ny / nx
    hw, vw, uw = _waves(rng, 12, 8), _waves(rng, 4, 3), _waves(rng, 4, 3)
    cx, cy = rng.uniform(0.3, 0.7), top * rng.uniform(0.3, 0.7)
    if setting == "unit":
        hv = 1.0 + 0.1 * torch.sin(2 * math.pi * x) * torch.cos(2 * math.pi * y)
        amp, sig, speed = 0.01, 0.07, 0.01
    elif setting == "ocean":
        hv = 2025.0 + 1975.0 * torch.tanh(_field(hw, x, y))
        amp, sig, speed = 1.0, 0.05, 0.02
    elif setting == "shelf":
        hv = (20.0 + 1990.0 * (1.0 - torch.tanh((x - 0.5) * 25.0))) * (1.0 + 0.02 * torch.tanh(_field(hw, x, y)))
        amp, sig, speed = 3.0, 0.06, 0.05
    else:
        hv = torch.full_like(x, 10.0)
        amp, sig, speed = 1.0, 0.125, 0.02

    def fields(px, py):
        """xi and the velocity at points of the member's domain"""
        px, py = px / width, py / width
        r2 = (px - cx) ** 2 + (py - cy) ** 2
        if setting == "dam":
            xi = 0.5 * amp * (1.0 - torch.tanh((torch.sqrt(r2 + 1e-12) - sig) / 0.002))
        else:
            xi = amp * torch.exp(-r2 / (2 * sig * sig)) + 0.05 * amp * _field(uw, px, py)
        return xi, speed * _field(uw, px, py), speed * _field(vw, px, py)

    frac = np.cumsum([float(f) for f in case["orders"].split(",")])  # these shares, at random places
    orders = np.searchsorted(frac / frac[-1], (rng.permutation(len(tri)) + 0.5) / len(tri)).clip(0, 4).astype(np.int8)
    tags = None
    if setting == "shelf":  # open sea on x = 0
        tags = np.zeros(tri.shape, np.int8)
        for k in range(3):
            on = (xy[tri[:, (k + 1) % 3], 0] == 0.0) & (xy[tri[:, (k + 2) % 3], 0] == 0.0)
            tags[on, k] = 2
    return dict(xy=xy, tri=tri, bc_tag=tags, hv=hv.cpu().numpy(), orders=orders, fields=fields)


def _k_of(orders):
    return (orders.long() + 1) * (orders.long() + 2) // 2


def _project(m, fields, zero_rest=True):
    """L2 projection of (xi, H u, H v) onto every element's modes: c[3][15][ne] on the device"""
    dev = _dev()
    xy, tri = torch.from_numpy(m["xy"]).to(dev), torch.from_numpy(m["tri"]).long().to(dev)
    hv, orders = torch.from_numpy(m["hv"]).to(dev), torch.from_numpy(m["orders"]).to(dev)
    X, Y, W = _tri_rule(6)
    phi = torch.from_numpy(_basis(X, Y)[0] * W).to(dev)  # [15, nq]
    lam = torch.from_numpy(np.stack([1 - X - Y, X, Y])).to(dev)
    ne = len(tri)
    c = torch.empty((3, KMAX, ne), dtype=torch.float64, device=dev)
    for a in range(0, ne, 1 << 18):
        b = min(ne, a + (1 << 18))
        v = xy[tri[a:b]]  # [n, 3, 2]
        s = torch.sqrt((v[:, 1, 0] - v[:, 0, 0]) * (v[:, 2, 1] - v[:, 0, 1]) -
                       (v[:, 2, 0] - v[:, 0, 0]) * (v[:, 1, 1] - v[:, 0, 1]))
        px, py, hb = v[:, :, 0] @ lam, v[:, :, 1] @ lam, hv[tri[a:b]] @ lam
        xi, u, w = fields(px, py)
        for f, val in enumerate((xi, (xi + hb) * u, (xi + hb) * w)):
            c[f, :, a:b] = s * (phi @ val.T)
    c *= (torch.arange(KMAX, device=dev)[:, None] < _k_of(orders)[None, :])
    return c


def _inputs(case, seed):
    """the members' meshes and their initial states (several states of one mesh for the stream)"""
    rng = np.random.default_rng([int(seed), case["nx"], case["ny"]])
    if case["kind"] == "ensemble":  # member sizes spread evenly in their logarithm over a factor of 16
        f = [0.25 ** (i / case["members"]) for i in range(case["members"])]
        ms = [_one_mesh(case, max(3, int(case["nx"] * q)), max(3, int(case["ny"] * q)), rng) for q in f]
        return ms, [_project(m, m["fields"]) for m in ms]
    m = _one_mesh(case, case["nx"], case["ny"], rng)
    c = _project(m, m["fields"])
    if case["kind"] == "stream":
        return [m], [c * (1.0 - 0.1 * i) for i in range(case["members"])]
    return [m], [c]


def _pack(c, orders):
    """packed state: element by element, 3 K(p) values (xi, U, V modes)"""
    k = _k_of(torch.from_numpy(orders).to(c.device))
    mask = (torch.arange(KMAX, device=c.device)[None, :] < k[:, None])[:, None, :].expand(-1, 3, -1)
    return c.permute(2, 0, 1)[mask].contiguous()


# ------------------------------------------------------------------ the calls
def prepare(case, seed):
    meshes, states = _inputs(case, seed)
    kind = case["kind"]
    if kind == "noalloc":
        m, dev = meshes[0], _dev()
        ne = len(m["tri"])
        nbr, _ = swedg.mesh_adjacency(m["xy"], m["tri"])
        return dict(kind=kind, xy=torch.from_numpy(m["xy"]).to(dev), tri=torch.from_numpy(m["tri"]).to(dev),
                    hv=torch.from_numpy(m["hv"]).to(dev), nbr=torch.from_numpy(nbr).to(dev),
                    c=states[0][:, :3].contiguous(), out=torch.empty((3, 3, ne), dtype=torch.float64, device=dev),
                    stream=torch.cuda.current_stream().cuda_stream)
    kw = dict(_params(case), precision=PREC[case["prec"]])
    if kind == "ensemble":
        return dict(kind=kind, steps=case["steps"], states=states, ens=ensemble.Ensemble(meshes, **kw))
    m = meshes[0]
    s = swedg.Solver(**kw)
    s.set_mesh(m["xy"], m["tri"], m["bc_tag"])
    s.set_bathymetry(m["hv"])
    s.set_orders(m["orders"])
    if case["shape"]:
        s.set_launch_shape([int(v) for v in case["shape"].split(",")])
    if kind == "stream":
        ins = [_pack(c, m["orders"]).cpu().pin_memory() for c in states]
        return dict(kind=kind, steps=case["steps"], solver=s, ins=ins, outs=[torch.empty_like(c).pin_memory() for c in ins])
    return dict(kind=kind, steps=case["steps"], every=case["every"], solver=s, c=states[0], orders=m["orders"],
                out=torch.empty_like(states[0]))


def run(st):
    kind = st["kind"]
    if kind == "noalloc":
        swedg.rhs_p1_noalloc(st["xy"], st["hv"], st["tri"], st["nbr"], st["c"], G, st["out"], st["stream"])
        return {"xi": st["out"][0], "U": st["out"][1], "V": st["out"][2]}
    if kind == "ensemble":
        e = st["ens"]
        e.set_states(st["states"])
        e.run(st["steps"])
        return {"states": e.states(device=True), "times": e.times()[0]}
    s = st["solver"]
    if kind == "stream":
        for a, b in zip(st["ins"], st["outs"]):
            s.set_state_packed_async(a, 0.0)
            s.run_async(st["steps"])
            s.get_state_packed_async(b)
        s.sync()
        return st["outs"]
    if kind == "rhs":
        s.rhs(st["c"], st["out"])
        return {"xi": st["out"][0], "U": st["out"][1], "V": st["out"][2]}
    if kind == "adapt":
        s.set_orders(st["orders"])
        s.set_state(st["c"], 0.0)
        s.run_adaptive(st["steps"], st["every"], 0.05, 1e-3, 1, 3)
        orders, _ = s.adapt(float("inf"), 0.0, 1, 3)  # thresholds that change nothing: the current orders
        _, t = s.get_state(st["out"])
        return {"xi": st["out"][0], "U": st["out"][1], "V": st["out"][2], "t": t, "orders": orders}
    s.set_state(st["c"], 0.0)
    s.run(st["steps"])
    _, t = s.get_state(st["out"])
    return {"xi": st["out"][0], "U": st["out"][1], "V": st["out"][2], "t": t}


def work(case):
    """bytes: the states that go in and come out and the mesh, once; flops: the contractions of every stage"""
    pc = np.array([float(f) for f in case["orders"].split(",")])
    ks = np.array([1, 3, 6, 10, 15])
    ne = 2.0 * case["nx"] * case["ny"]
    if case["kind"] == "ensemble":
        ne *= sum(0.0625 ** (i / case["members"]) for i in range(case["members"]))
    k = float(pc @ ks) / pc.sum()
    # auxiliary solve (K^3/3 + 4 K^2), volume terms (two velocity components and the pressure against K test
    # modes over K coefficients: 6 K^2 with the orthonormal basis at the least), edge traces and projections
    fl = float(pc @ (ks ** 3 / 3 + 10 * ks ** 2 + 60 * ks)) / pc.sum()
    stages = {"noalloc": 1, "rhs": 1}.get(case["kind"], case["steps"] * case["rk"])
    copies = case["members"] if case["kind"] == "stream" else 1
    return {"bytes": ne * copies * (2 * 3 * k * 8) + ne * (12 + 0.5 * 24 + 1), "flops": ne * copies * stages * fl}


def tolerance(case):
    """About four times the largest difference from `exact` seen over the listed and 60 drawn cases.  FP64: rounding
    of the sums (a right-hand side is the small difference of its edge and volume terms, a state is not).  Mixed
    modes: the terms of degree >= 2 in 32 bits, in a right-hand side directly, in a state times the step."""
    if case["kind"] == "noalloc" or (case["kind"] == "rhs" and case["prec"] == "fp64"):
        return {"rel": 1.5e-13, "max": 2e-12}
    if case["kind"] == "rhs":
        return {"rel": 6e-6, "max": 1e-4}
    if case["prec"] == "fp64":
        return {"rel": 2e-15, "max": 5e-14, "differ": 1e-4}
    return {"rel": 1.5e-7, "max": 3e-6}


# ------------------------------------------------------------------ exact: the weak form by quadrature, 64 bits
def _gauss01(n):
    z, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (z + 1.0), 0.5 * w


def _tri_rule(n):
    """collapsed n x n Gauss rule on the reference triangle, exact to degree 2 n - 2"""
    s, w = _gauss01(n)
    u, v = np.meshgrid(s, s, indexing="ij")
    return (u * (1.0 - v)).ravel(), v.ravel(), (np.outer(w, w) * (1.0 - v)).ravel()


def _jacobi(n, al, t):
    """P_n^(al,0)(t) and its derivative"""
    p = [np.ones_like(t), 0.5 * ((al + 2.0) * t + al)]
    d = [np.zeros_like(t), np.full_like(t, 0.5 * (al + 2.0))]
    for m in range(1, n):
        s = 2.0 * m + al
        a1, a2 = 2.0 * (m + 1) * (m + al + 1) * s, (s + 1) * al * al
        a3, a4 = s * (s + 1) * (s + 2), 2.0 * (m + al) * m * (s + 2)
        p.append(((a2 + a3 * t) * p[m] - a4 * p[m - 1]) / a1)
        d.append((a3 * p[m] + (a2 + a3 * t) * d[m] - a4 * d[m - 1]) / a1)
    return p[n], d[n]


def _basis(x, y):
    """orthonormal Dubiner basis (by degree, then by the Jacobi index): values and both derivatives, [15, points]"""
    v, vx, vy = (np.zeros((KMAX,) + x.shape) for _ in range(3))
    l, m = 2.0 * x + y - 1.0, 1.0 - y
    r = [(np.ones_like(x), np.zeros_like(x), np.zeros_like(x)), (l, np.full_like(x, 2.0), np.ones_like(x))]
    for a in range(1, 4):  # R_a = P_a((2x+y-1)/(1-y)) (1-y)^a
        (f, fx, fy), (g, gx, gy) = r[a], r[a - 1]
        c1, c2 = (2.0 * a + 1) / (a + 1), a / (a + 1.0)
        r.append((c1 * l * f - c2 * m * m * g, c1 * (2 * f + l * fx) - c2 * m * m * gx,
                  c1 * (f + l * fy) - c2 * (m * m * gy - 2 * m * g)))
    i = 0
    for d in range(5):
        for b in range(d + 1):
            a = d - b
            p, dp = _jacobi(b, 2.0 * a + 1.0, 2.0 * y - 1.0)
            n = math.sqrt(2.0 * (2 * a + 1) * (a + b + 1))
            v[i], vx[i], vy[i] = n * r[a][0] * p, n * r[a][1] * p, n * (r[a][2] * p + r[a][0] * 2 * dp)
            i += 1
    return v, vx, vy


_EDGE = [((1.0, 0.0), (-1.0, 1.0)), ((0.0, 1.0), (0.0, -1.0)), ((0.0, 0.0), (1.0, 0.0))]


class _Reference:
    """the semi-discrete scheme on one union mesh; state c[3][15][ne]"""

    def __init__(self, m, member, nmem, prm):
        dev = _dev()
        put = lambda a: torch.as_tensor(a, dtype=torch.float64, device=dev)  # noqa: E731
        self.dev, self.put, self.prm, self.nmem = dev, put, prm, nmem
        tri = torch.from_numpy(m["tri"]).long().to(dev)
        v = put(m["xy"])[tri]
        self.ne = len(tri)
        self.member = torch.from_numpy(member).long().to(dev)
        self.hvt = put(m["hv"])[tri].T.contiguous()  # [3, ne]
        a, b = v[:, 1] - v[:, 0], v[:, 2] - v[:, 0]
        det = a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0]
        self.det, self.s = det, torch.sqrt(det)
        self.ji = torch.stack([b[:, 1], -b[:, 0], -a[:, 1], a[:, 0]]) / det
        h = self.hvt
        self.dh = torch.stack([(h[1] - h[0]) * self.ji[0] + (h[2] - h[0]) * self.ji[2],
                               (h[1] - h[0]) * self.ji[1] + (h[2] - h[0]) * self.ji[3]])
        x, y, w = _tri_rule(8)
        phi = _basis(x, y)[0]
        self.hb = self.s * (put((phi[:3] * w) @ np.stack([1 - x - y, x, y]).T) @ h)
        self.T = put(np.einsum("ng,ig,jg->nij", phi * w, phi, phi))
        # edges: outward normal, length, depths at both ends, neighbour and its local edge
        ends = [(1, 2), (2, 0), (0, 1)]
        d = torch.stack([v[:, q] - v[:, p] for p, q in ends])  # [3, ne, 2]
        self.len = torch.linalg.norm(d, dim=2)
        self.nx, self.ny = d[:, :, 1] / self.len, -d[:, :, 0] / self.len
        self.diam = 2.0 * det / self.len.sum(0)
        self.hA, self.hB = torch.stack([h[p] for p, _ in ends]), torch.stack([h[q] for _, q in ends])
        pq = torch.stack([torch.stack([tri[:, p], tri[:, q]]) for p, q in ends])  # [3, 2, ne]
        key = (pq.amin(1) * len(m["xy"]) + pq.amax(1)).reshape(-1)
        order = torch.argsort(key)
        same = torch.nonzero(key[order][1:] == key[order][:-1])[:, 0]
        nb = torch.full((3 * self.ne,), -1, dtype=torch.long, device=dev)
        nb[order[same]], nb[order[same + 1]] = order[same + 1], order[same]
        self.nb = nb.reshape(3, self.ne)  # edge id k ne + e across the edge, -1 on the boundary
        tag = m["bc_tag"] if m["bc_tag"] is not None else np.zeros(m["tri"].shape, np.int8)
        self.sea = (torch.from_numpy(tag).to(dev).T == 2) & (self.nb < 0)
        s7, self.w7 = _gauss01(7)
        self.s7 = put(s7)
        self.eb = put(np.stack([_basis(p[0] + q[0] * s7, p[1] + q[1] * s7)[0] for p, q in map(np.array, _EDGE)]))
        self.set_orders(torch.from_numpy(m["orders"]).to(dev))

    def set_orders(self, p):
        self.p = p.long()
        self.mask = torch.arange(KMAX, device=self.dev)[:, None] < _k_of(p)[None, :]
        self.groups = [(q, torch.nonzero(self.p == q)[:, 0]) for q in range(5)]

    def chunks(self):
        for p, idx in self.groups:
            for a in range(0, len(idx), 1 << 17):
                yield p, (p + 1) * (p + 2) // 2, idx[a:a + (1 << 17)]

    def velocity(self, c):
        u = torch.zeros((2, KMAX, self.ne), dtype=torch.float64, device=self.dev)
        H = c[0].clone()
        H[:3] += self.hb
        kt = torch.tensor([[(max(DEG[i], DEG[j]) + 1) * (max(DEG[i], DEG[j]) + 2) // 2 for j in range(KMAX)] for i in range(KMAX)])
        tt = self.T * (torch.arange(KMAX)[:, None, None] < kt[None]).to(self.dev)
        for p, K, e in self.chunks():
            M = torch.einsum("nij,ne->eij", tt[:K, :K, :K], H[:K][:, e]) / self.s[e][:, None, None]
            u[:, :K, e] = torch.linalg.solve(M, c[1:, :K][:, :, e].permute(2, 1, 0)).permute(2, 1, 0)
        return u, H

    def tide(self, t):
        a, period, ph = self.prm["tide"]
        return torch.full_like(t, a) if period <= 0 else a * torch.sin(2 * math.pi * t / period + ph)

    def rhs(self, c, t):
        """t: [members]"""
        g, s2 = G, math.sqrt(2.0)
        u, H = self.velocity(c)
        r = torch.zeros_like(c)
        for p, K, e in self.chunks():
            if K > 1:
                x, y, w = _tri_rule((3 * p + 4) // 2)
                phi, px, py = (self.put(z[:K]) for z in _basis(x, y))
                s, ji = self.s[e], self.ji[:, e]
                ev = lambda z: (phi.T @ z[:K][:, e]) / s  # noqa: E731
                xi, U, V, uu, vv = ev(c[0]), ev(c[1]), ev(c[2]), ev(u[0]), ev(u[1])
                hb = self.put(np.stack([1 - x - y, x, y]).T) @ self.hvt[:, e]
                P = g * xi * (0.5 * xi + hb)
                ws = self.put(w)[:, None] * s
                for f, (ax, ay) in enumerate(((U, V), (U * uu + P, U * vv), (V * uu, V * vv + P))):
                    r[f, :K, e] = px @ (ws * (ax * ji[0] + ay * ji[1])) + py @ (ws * (ax * ji[2] + ay * ji[3]))
        r[1] += g * self.dh[0] * c[0]
        r[2] += g * self.dh[1] * c[0]
        lin, quad = self.prm["friction"]
        m0 = s2 / self.s
        tau = lin * H[0] * m0 + quad * torch.sqrt((u[0, 0] * m0) ** 2 + (u[1, 0] * m0) ** 2)
        r[1] += self.prm["f_c"] * c[2] - tau * u[0]
        r[2] -= self.prm["f_c"] * c[1] + tau * u[1]
        # traces of every element on its three edges [5, 3, 7, ne], then both sides' flux
        w = torch.cat([c, u])  # [5, 15, ne]
        tr = torch.empty((5, 3, 7, self.ne), dtype=torch.float64, device=self.dev)
        for k in range(3):
            for f in range(5):
                tr[f, k] = (self.eb[k].T @ w[f]) / self.s
        xt = self.tide(t)[self.member]
        w7 = self.put(self.w7)[:, None]
        for k in range(3):
            nx, ny, nb = self.nx[k], self.ny[k], self.nb[k]
            inner = nb >= 0
            ke, ee = nb.clamp(min=0) // self.ne, nb.clamp(min=0) % self.ne
            a = tr[:, k]
            b = torch.empty_like(a)
            for j in range(3):  # the neighbour runs the edge the other way
                on = inner & (ke == j)
                b[:, :, on] = tr[:, j][:, :, ee[on]].flip(1)
            wall = ~inner & ~self.sea[k]
            for i in (1, 3):
                qn = a[i] * nx + a[i + 1] * ny
                b[i] = torch.where(inner, b[i], torch.where(wall, a[i] - 2 * qn * nx, a[i]))
                b[i + 1] = torch.where(inner, b[i + 1], torch.where(wall, a[i + 1] - 2 * qn * ny, a[i + 1]))
            b[0] = torch.where(inner, b[0], torch.where(wall, a[0], xt.expand_as(a[0])))
            hmid = 0.5 * (self.hA[k] + self.hB[k])
            un = (u[0, 0] * nx + u[1, 0] * ny) * m0
            un2 = torch.where(inner, ((u[0, 0] * m0)[ee] * nx + (u[1, 0] * m0)[ee] * ny), un)
            HL = c[0, 0] * m0 + hmid
            HR = torch.where(inner, (c[0, 0] * m0)[ee] + hmid, torch.where(wall, HL, xt + hmid))
            lam = torch.maximum(un.abs(), un2.abs()) + torch.sqrt(g * torch.maximum(HL, HR))
            hb = self.hA[k] + self.s7[:, None] * (self.hB[k] - self.hA[k])
            F = torch.zeros_like(a[:3])
            for z, sg in ((a, 1.0), (b, -1.0)):
                wn = z[3] * nx + z[4] * ny
                P = g * z[0] * (0.5 * z[0] + hb)
                F[0] += z[1] * nx + z[2] * ny + sg * lam * z[0]
                F[1] += z[1] * wn + P * nx + sg * lam * z[1]
                F[2] += z[2] * wn + P * ny + sg * lam * z[2]
            for f in range(3):
                r[f] -= self.eb[k] @ (0.5 * w7 * F[f] * (self.len[k] / self.s))
        return r * self.mask

    def step(self, c, t):
        u, H = self.velocity(c)
        m0 = math.sqrt(2.0) / self.s
        sp = torch.sqrt((u[0, 0] * m0) ** 2 + (u[1, 0] * m0) ** 2) + torch.sqrt(G * H[0] * m0)
        bound = self.diam / (sp * (2.0 * self.p + 1.0))
        dt = self.prm["cfl"] * torch.full((self.nmem,), math.inf, dtype=torch.float64, device=self.dev).scatter_reduce(
            0, self.member, bound, "amin")
        d = dt[self.member]
        c1 = c + d * self.rhs(c, t)
        if self.prm["rk_order"] == 2:
            return 0.5 * c + 0.5 * (c1 + d * self.rhs(c1, t + dt)), t + dt
        c2 = 0.75 * c + 0.25 * (c1 + d * self.rhs(c1, t + dt))
        return c / 3.0 + 2.0 / 3.0 * (c2 + d * self.rhs(c2, t + 0.5 * dt)), t + dt

    def adapt(self, c, up, down, pmin, pmax):
        deg = torch.tensor(DEG, device=self.dev)[:, None]
        x2 = c[0] ** 2
        den = (x2 * (deg >= 1)).sum(0)
        s = torch.where((den > 0) & (self.p > 0), (x2 * (deg == self.p)).sum(0) / den, torch.zeros_like(den))
        p = torch.where((s > up) & (self.p < pmax), self.p + 1, torch.where((s < down) & (self.p > pmin), self.p - 1, self.p))
        self.set_orders(p)
        return c * self.mask


def exact(case, seed):
    meshes, states = _inputs(case, seed)
    kind, prm = case["kind"], _params(case)
    v0 = np.cumsum([0] + [len(m["xy"]) for m in meshes])
    join = dict(xy=np.concatenate([m["xy"] for m in meshes]), hv=np.concatenate([m["hv"] for m in meshes]),
                tri=np.concatenate([m["tri"] + int(v) for m, v in zip(meshes, v0)]),
                orders=np.concatenate([m["orders"] for m in meshes]), bc_tag=meshes[0]["bc_tag"])
    if kind == "noalloc":
        join["bc_tag"] = None
        prm["tide"] = (0.0, 0.0, 0.0)
    member = np.repeat(np.arange(len(meshes)), [len(m["tri"]) for m in meshes])
    ref = _Reference(join, member, len(meshes), prm)
    t = torch.zeros(len(meshes), dtype=torch.float64, device=ref.dev)
    if kind in ("noalloc", "rhs"):
        r = ref.rhs(states[0], t)
        r = r[:, :3] if kind == "noalloc" else r
        return {"xi": r[0], "U": r[1], "V": r[2]}
    if kind == "stream":
        outs = []
        for c in states:
            tt = t
            for _ in range(case["steps"]):
                c, tt = ref.step(c, tt)
            outs.append(_pack(c, join["orders"]))
        return outs
    c = torch.cat(states, dim=2)
    for i in range(case["steps"]):
        c, t = ref.step(c, t)
        if kind == "adapt" and (i + 1) % case["every"] == 0:
            c = ref.adapt(c, 0.05, 1e-3, 1, 3)
    if kind == "ensemble":
        ends = np.cumsum([0] + [len(m["tri"]) for m in meshes])
        return {"states": [c[:, :, a:b].contiguous() for a, b in zip(ends[:-1], ends[1:])], "times": t}
    out = {"xi": c[0], "U": c[1], "V": c[2], "t": float(t[0])}
    if kind == "adapt":
        out["orders"] = None  # whole numbers
    return out
