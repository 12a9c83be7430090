"""The work that users of this library have it do, as measurable cases.

The sizes are those of the library's own workloads (inputs.workload, the
benchmark and the tests): products and solves on the sphere and the head-like
surface, the duct, the admittance gradient and the fields at points, from the
smallest mesh a call is made with to the 158,420-element surface.

A case is a dict of plain values:
  kind      what a pass calls: "product", "solve", "gradient", "field"
  surface   "sphere" (radius 0.1 m), "head" (the bumpy ellipsoid) or "duct"
  nu        geodesic frequency of the surface (20 nu^2 triangles); for the
            duct, squares per 0.2 m edge
  freq      Hz
  factor    factor of the expansion length (1.8: the paper's; 8: truncation
            below the FP32 rounding)
and, by kind, the number of right-hand sides, the options and the points.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2312_00005_gb300 import bemfmm, inputs

C, RHO = 343.0, 1.21
_DEV = "cuda" if torch.cuda.is_available() else "cpu"


def _case(kind, surface, nu, freq, factor, **kw):
    return dict(kind=kind, surface=surface, nu=nu, freq=freq, factor=factor, **kw)


def listed():
    return [
        # one product on the smallest sphere that the tests solve on: a caller's own iteration over a
        # coarse mesh, where launches and the work on the host count
        dict(_case("product", "sphere", 8, 1000.0, 1.8, rhs=1, direct=False, split=False), name="product_sphere1280"),
        # the product of the benchmark's default workload, in a caller's own iteration
        dict(_case("product", "sphere", 32, 4000.0, 8.0, rhs=1, direct=False, split=False), name="product_sphere20480"),
        # four right-hand sides at once with the aggregation on the tensor cores (split BF16)
        dict(_case("product", "head", 45, 10000.0, 8.0, rhs=4, direct=False, split=True),
             name="product_head40500_split"),
        # the largest workload: four right-hand sides on 158,420 elements at 20 kHz
        dict(_case("product", "head", 89, 20000.0, 8.0, rhs=4, direct=False, split=False),
             name="product_head158420"),
        # the conventional BEM product, every entry by quadrature in the product (no stored matrix)
        dict(_case("product", "sphere", 16, 2000.0, 8.0, rhs=1, direct=True, split=False),
             name="product_direct5120"),
        # a frequency sweep with the field at 100 points: the benchmark's default workload
        dict(_case("solve", "sphere", 32, 4000.0, 8.0, rhs=1, freqs=2, points=100, jacobi=False),
             name="sweep_sphere20480"),
        # the paper's duct (Sec. 5.3): interior problem, driven end, absorbing end, solves one by one
        dict(_case("solve", "duct", 4, 240.0, 1.8, rhs=1, freqs=2, points=0, jacobi=False), name="solve_duct2240"),
        # one band of the batched frequencies: head-like surface, point source at the surface, block-Jacobi
        dict(_case("solve", "head", 26, 7000.0, 8.0, rhs=1, freqs=2, points=100, jacobi=True),
             name="sweep_head13520"),
        # four plane waves solved together
        dict(_case("solve", "head", 23, 5000.0, 8.0, rhs=4, freqs=2, points=0, jacobi=True),
             name="solve4_head10580"),
        # a step of fitting eight region admittances: loss and gradient through the autograd function
        dict(_case("gradient", "head", 22, 2000.0, 8.0, points=100), name="gradient_head9680"),
        # the field on a grid of the paper's size, through the expansions
        dict(_case("field", "sphere", 32, 4000.0, 8.0, points=24874, velocity=False), name="field_sphere20480"),
        # field and particle velocity at a measurement grid, summed directly
        dict(_case("field", "sphere", 16, 2000.0, 8.0, points=1000, velocity=True), name="velocity_sphere5120"),
    ]


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def draw(rng):
    kind = rng.choice(["product", "product", "product", "solve", "solve", "gradient", "field", "field"])
    surface = rng.choice(["sphere", "head"])
    factor = rng.choice([5.0, 6.0, 8.0])

    def at(nu, lo, hi):
        # elements per wavelength between those of the workloads: the mean edge is about 0.115 m / nu
        return round(min(20000.0, max(200.0, C * nu / 0.115 / _log(rng, lo, hi))), 2)

    if kind == "product":
        direct = rng.random() < 0.2
        nu = round(_log(rng, 3, 20)) if direct else round(_log(rng, 5, 80))
        split = not direct and rng.random() < 0.2
        return _case(kind, surface, nu, at(nu, 10, 30), factor, rhs=rng.choice([1, 1, 2, 3, 4, 5]), direct=direct,
                     split=split)
    if kind == "solve":
        if rng.random() < 0.25:
            return _case(kind, "duct", rng.choice([2, 3, 4, 5]), round(rng.uniform(120.0, 300.0), 2), 1.8, rhs=1,
                         freqs=rng.choice([2, 3]), points=0, jacobi=False)
        nu = round(_log(rng, 6, 26))
        rhs = rng.choice([1, 1, 1, 2, 3])
        return _case(kind, surface, nu, at(nu, 13, 30), factor, rhs=rhs, freqs=2,
                     points=rng.choice([0, 37, 100]) if rhs == 1 else 0,
                     jacobi=surface == "head" or rng.random() < 0.5)
    if kind == "gradient":
        nu = round(_log(rng, 6, 22))
        return _case(kind, surface, nu, at(nu, 15, 30), factor, points=round(_log(rng, 10, 200)))
    nu = round(_log(rng, 8, 36))
    return _case(kind, surface, nu, at(nu, 12, 30), factor, points=round(_log(rng, 50, 25000)),
                 velocity=rng.random() < 0.3 and nu <= 16)


# ---------------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=6)
def _surface(surface, nu):
    if surface == "duct":
        return inputs.duct(3.4, 0.2, 0.2 / nu)
    if surface == "head":
        return inputs.bumpy_ellipsoid(nu)
    if nu & (nu - 1) == 0:
        return inputs.icosphere(nu.bit_length() - 1, 0.1)
    nodes, tris = inputs.geodesic_sphere(nu)
    return 0.1 * nodes, tris


def _params(case):
    kw = dict(trunc_factor=case["factor"])
    if case.get("direct"):
        kw["mode"] = bemfmm.MODE_DIRECT
    if case.get("split"):
        kw["far_precision"] = 1
    if case.get("jacobi"):
        kw.update(block_jacobi=1, restart=600)
    if case["surface"] == "duct":
        kw["tau"] = -1.0
    if case["kind"] == "field" and case["points"] > 10000 and case["nu"] >= 24:
        kw["field_mode"] = 2
    return kw


def _points(case, rng):
    """Field points off the surface: a sphere of 0.3 to 1 m around it and, for the larger sets, half of
    them on a plane grid through the middle of the scatterer, outside of it."""
    m = case["points"]
    if m <= 1000:
        return inputs.fibonacci_sphere(m, rng.uniform(0.8, 1.0))
    a = m // 2
    s = int(math.ceil(math.sqrt(2.0 * (m - a))))
    g = np.linspace(-0.4, 0.4, s) + rng.uniform(-1e-4, 1e-4)
    grid = np.stack([np.repeat(g, s), np.tile(g, s), np.zeros(s * s)], axis=1)
    grid = grid[np.linalg.norm(grid, axis=1) > 0.13]
    return np.concatenate([inputs.fibonacci_sphere(m - min(m - a, len(grid)), rng.uniform(0.8, 1.0)),
                           grid[rng.permutation(len(grid))[:m - a]]])


def _inputs(case, seed):
    """Everything that a pass takes, from the seed alone (host arrays)."""
    rng = np.random.default_rng(seed)
    nodes, tris = _surface(case["surface"], case["nu"])
    n = tris.shape[0]
    d = {"nodes": nodes, "tris": tris, "n": n, "bc_type": None, "bc_value": None, "region": None, "adm": None}
    cen = nodes[tris].mean(axis=1)
    if case["kind"] == "product":
        shape = (n,) if case["rhs"] == 1 else (case["rhs"], n)
        d["x"] = (rng.normal(size=shape) + 1j * rng.normal(size=shape)).astype(np.complex64)
    elif case["kind"] == "solve" and case["surface"] == "duct":
        # driven at x = 0, absorbing at x = 3.4 m, hard walls
        d["bc_type"] = np.where(cen[:, 0] > 3.4 - 1e-9, bemfmm.ADMI, bemfmm.VELO).astype(np.int32)
        d["bc_value"] = np.where(cen[:, 0] < 1e-9, -np.exp(1j * rng.uniform(0, 6.28)), 0.0)
        d["region"] = np.zeros(n, np.int32)
        d["adm"] = np.array([rng.uniform(0.8, 1.2) / (RHO * C)], np.complex128)
        d["freqs"] = [case["freq"] * (1.0 + 0.01 * i) for i in range(case["freqs"])]
        d["sources"] = []
    elif case["kind"] == "solve":
        d["freqs"] = [case["freq"] * (1.0 + 0.002 * i) for i in range(case["freqs"])]
        if case["surface"] == "head" and case["rhs"] == 1:
            d["sources"] = [("point", inputs.head_point_source(rng.uniform(0.001, 0.003)),
                             np.exp(1j * rng.uniform(0, 6.28)))]
        else:
            v = rng.normal(size=(case["rhs"], 3))
            v /= np.linalg.norm(v, axis=1, keepdims=True)
            d["sources"] = [("plane", u, np.exp(1j * rng.uniform(0, 6.28))) for u in v]
        d["points"] = _points(case, rng) if case["points"] else None
    elif case["kind"] == "gradient":
        c0 = cen - cen.mean(axis=0)
        d["bc_type"] = np.full(n, bemfmm.ADMI, np.int32)
        d["region"] = ((c0[:, 0] > 0) + 2 * (c0[:, 1] > 0) + 4 * (c0[:, 2] > 0)).astype(np.int32)
        adm = rng.uniform(0.05, 0.5, 8) * np.exp(1j * rng.uniform(-np.pi / 2, np.pi / 2, 8)) / (RHO * C)
        d["adm"] = adm.astype(np.complex64)
        v = rng.normal(size=3)
        d["sources"] = [("point", 0.4 * v / np.linalg.norm(v), 1.0)]
        d["points"] = _points(case, rng)
    else:
        # the surface data of a radiated field (monopoles inside), and the plane wave it was scattered from
        k = 2 * math.pi * case["freq"] / C
        a, b, c = (nodes[tris[:, i]] for i in range(3))
        nrm = np.cross(b - a, c - a)
        nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
        p, q = np.zeros(n, np.complex128), np.zeros(n, np.complex128)
        for _ in range(5):
            r = cen - 0.03 * rng.uniform(-1, 1, 3)
            R = np.linalg.norm(r, axis=1)
            g = (rng.normal() + 1j * rng.normal()) * np.exp(1j * k * R) / (4 * np.pi * R)
            p += g
            q += g * (1j * k - 1 / R) * np.einsum("ij,ij->i", r, nrm) / R
        d["p"], d["q"] = p.astype(np.complex64), q.astype(np.complex64)
        d["sources"] = [("plane", np.array([0.0, 0.0, 1.0]), 1.0)]
        d["points"] = _points(case, rng)
    return d


def _source(s):
    return bemfmm.plane_wave(s[1], s[2]) if s[0] == "plane" else bemfmm.point_source(s[1], s[2])


def prepare(case, seed):
    """The mesh handle that a user's program keeps, and the pass's inputs on the GPU."""
    d = _inputs(case, seed)
    st = {"case": case, "mesh": bemfmm.Mesh(d["nodes"], d["tris"], bc_type=d["bc_type"], bc_value=d["bc_value"],
                                            region=d["region"], **_params(case))}
    for name in ("x", "p", "q"):
        if name in d:
            st[name] = torch.from_numpy(d[name]).cuda()
    if case["kind"] == "product":
        st["y"] = torch.empty_like(st["x"])
    if case["kind"] == "gradient":
        st["Y"] = torch.from_numpy(d["adm"]).cuda().requires_grad_()
    else:
        st["adm"] = d["adm"]
    if "sources" in d:
        st["sources"] = [_source(s) for s in d["sources"]]
    st["points"] = d.get("points")
    st["freqs"] = d.get("freqs")
    return st


def run(state):
    case, mesh, f = state["case"], state["mesh"], state["case"]["freq"]
    if case["kind"] == "product":
        return mesh.matvec(f, state["x"], state["y"])
    if case["kind"] == "solve":
        if case["rhs"] > 1:
            return [mesh.solve_multi(g, state["sources"])[:2] for g in state["freqs"]]
        if case["surface"] == "duct":
            return [mesh.solve(g, state["sources"], admittance=state["adm"])[:2] for g in state["freqs"]]
        return mesh.solve_sweep(state["freqs"], state["sources"], points=state["points"])[:3]
    if case["kind"] == "gradient":
        Y = state["Y"]
        Y.grad = None
        loss = bemfmm.admittance_loss(mesh, Y, f, state["sources"], state["points"], tol=1e-6)
        loss.backward()
        return loss.detach(), Y.grad
    out = [mesh.evaluate(f, state["p"], state["q"], state["points"], state["sources"])]
    if case["velocity"]:
        out.append(mesh.evaluate_velocity(f, state["p"], state["q"], state["points"], state["sources"]))
    return out


# ---------------------------------------------------------------------- work
@functools.lru_cache(maxsize=None)
def _stats(surface, nu, freq, factor, direct):
    nodes, tris = _surface(surface, nu)
    kw = dict(mode=bemfmm.MODE_DIRECT) if direct else {}
    return bemfmm.plan_stats_host(nodes, tris, freq, params=bemfmm.default_params(trunc_factor=factor, **kw))


def work(case):
    """The lists at the automatic leaf size; 60 operations per kernel evaluation, 8 per complex
    multiply-add; the stored near field (which belongs to the handle) read once per product.  A solve
    takes at least 20 products per frequency; the near field of each frequency is computed and written."""
    n = _surface(case["surface"], case["nu"])[1].shape[0]
    if case["kind"] == "field":
        m = case["points"]
        return {"bytes": 80.0 * n + 32.0 * m, "flops": 60.0 * n * m * (2 if case["velocity"] else 1)
                if case["points"] <= 10000 else 60.0 * 50 * m}
    s = _stats(case["surface"], case["nu"], case["freq"], case["factor"], bool(case.get("direct")))
    rhs = case.get("rhs", 1)
    if case.get("direct"):
        return {"bytes": 80.0 * n, "flops": 60.0 * s["near_quad_points"] * rhs}
    far = sum(8.0 * L * L * (a + t) * 2 + 16.0 * L * L * i for L, a, t, i in
              zip(s["L"], s["n_src_elements"], s["n_tgt_elements"], s["n_interactions"]))
    prod = {"bytes": 8.0 * s["near_nnz"] + 16.0 * n * rhs, "flops": rhs * (8.0 * s["near_nnz"] + far)}
    if case["kind"] == "product":
        return prod
    nf, np_ = (case["freqs"], 20) if case["kind"] == "solve" else (1, 40)
    return {"bytes": nf * (8.0 * s["near_nnz"] + np_ * prod["bytes"]),
            "flops": nf * (60.0 * s["near_quad_points"] + np_ * prod["flops"])}


# ---------------------------------------------------------------------- in 64 bits
def _gauss01(m):
    x, w = np.polynomial.legendre.leggauss(m)
    return 0.5 * (x + 1), 0.5 * w


def _conical(m):
    """m x m conical rule on the unit triangle (Gauss-Jacobi (1,0) by Gauss-Legendre); the one-point
    rule is the centroid."""
    j = np.arange(m)
    a = -1.0 / ((2 * j + 1) * (2 * j + 3))                # recurrence of the Jacobi weight 1 - x
    b = np.arange(1, m) * (np.arange(1, m) + 1.0) / (2 * np.arange(1, m) + 1.0) ** 2
    T = np.diag(a) + np.diag(np.sqrt(b), 1) + np.diag(np.sqrt(b), -1)
    x, v = np.linalg.eigh(T)
    xj, wj = 0.5 * (x + 1), 0.25 * 2.0 * v[0] ** 2
    xl, wl = _gauss01(m)
    xi = np.repeat(xj, m)
    eta = ((1 - xj)[:, None] * xl[None, :]).ravel()
    return xi, eta, (wj[:, None] * wl[None, :]).ravel()


def _thresholds():
    """Distance ratios above which the regular rule of order m = 1..5 meets 1e-3 (the three estimates)."""
    out = []
    for m in range(1, 6):
        q = [(1e-3 / 32) ** (1 / (2 * m + 1)), (1e-3 / (64 * (2 * m + 1))) ** (1 / (2 * m + 2)),
             (1e-3 / (128 * (m + 1) * (2 * m + 1))) ** (1 / (2 * m + 3))]
        out.append(0.5 / min(q))
    return out


class _Dense:
    """The Burton-Miller collocation operator and the field formula with the method's quadrature rules,
    in 64 bits, as blocks of rows."""

    def __init__(self, nodes, tris, k):
        t = lambda v: torch.as_tensor(v, dtype=torch.float64, device=_DEV)  # noqa: E731
        P = t(nodes)[torch.as_tensor(tris, dtype=torch.int64, device=_DEV)]
        self.k, self.n = k, tris.shape[0]
        self.a, self.b, self.c = P[:, 0], P[:, 1], P[:, 2]
        self.cen = P.mean(dim=1)
        cr = torch.linalg.cross(self.b - self.a, self.c - self.a)
        len2 = cr.norm(dim=1)
        self.area, self.nrm = 0.5 * len2, cr / len2[:, None]
        self.R = _thresholds()
        self.rules = {m: [t(v) for v in _conical(m)] for m in range(1, 7)}

    # kernels at y = x + d, weight w: the two column kernels of the operator, G and H, or their gradients
    def _bm(self, d, nx, ny, w):
        k = self.k
        ir = d.square().sum(-1).rsqrt()
        G = torch.polar(w * ir / (4 * math.pi), k / ir)
        rx, ry, nn = (d * nx).sum(-1) * ir, (d * ny).sum(-1) * ir, (nx * ny).sum(-1)
        i2 = ir * ir / k
        return (G * torch.complex(ir * (ry - 3 * rx * ry + nn), -k * ry + (k - 3 * i2) * rx * ry + i2 * nn),
                G * torch.complex(1 - rx, -(ir / k) * rx))

    def _gh(self, d, nx, ny, w):
        ir = d.square().sum(-1).rsqrt()
        G = torch.polar(w * ir / (4 * math.pi), self.k / ir)
        ry = (d * ny).sum(-1) * ir
        return G * torch.complex(-ir * ry, self.k * ry), G

    def _grad(self, axis):
        def kernel(d, nx, ny, w):
            k = self.k
            ir = d.square().sum(-1).rsqrt()
            G = torch.polar(w * ir / (4 * math.pi), k / ir)
            f = G * torch.complex(-ir, torch.full_like(ir, k)) * ir
            fp = G * torch.complex(-k * k * ir + 3 * ir ** 3, -3 * k * ir * ir)
            return -fp * ((d * ny).sum(-1) * ir) * d[..., axis] - f * ny[..., axis], -f * d[..., axis]
        return kernel

    def block(self, x, nx, kernel, first=None):
        """[rows, n] integrals of a kernel pair over every element from the points x (rows `first`.. of
        the operator where `first` is given: their own elements are left zero)."""
        d0 = self.cen[None] - x[:, None]
        rt = d0.norm(dim=-1) / self.area.sqrt()[None]
        nxe = None if nx is None else nx[:, None]
        P, Q = kernel(d0, nxe, self.nrm[None], self.area[None].expand(rt.shape))
        near = rt <= self.R[0]
        if first is not None:
            rows = torch.arange(x.shape[0], device=_DEV)
            near[rows, first + rows] = False
            P[rows, first + rows] = 0
            Q[rows, first + rows] = 0
        i, j = near.nonzero(as_tuple=True)
        P[i, j] = 0
        Q[i, j] = 0
        flat = i * self.n + j
        a, b, c, area = self.a[j], self.b[j], self.c[j], self.area[j]
        Pf, Qf = P.view(-1), Q.view(-1)
        while flat.numel():
            # (sub)elements: subdivided while the ratio is below 1.3, else one rule
            ratio = ((a + b + c) / 3 - x[flat // self.n]).norm(dim=-1) / area.sqrt()
            left = ratio < 1.3
            order = 1 + sum((ratio <= r).to(torch.int64) for r in self.R)
            for m in range(1, 7):
                s = ((order == m) & ~left).nonzero()[:, 0]
                for part in s.split(2_000_000):
                    fl = flat[part]
                    xi, eta, w = self.rules[m]
                    row, col = fl // self.n, fl % self.n
                    p, q = 0, 0
                    base, e1, e2 = a[part] - x[row], b[part] - a[part], c[part] - a[part]
                    for u in range(m * m):
                        dp, dq = kernel(base + xi[u] * e1 + eta[u] * e2, None if nx is None else nx[row],
                                        self.nrm[col], 2 * area[part] * w[u])
                        p, q = p + dp, q + dq
                    Pf.index_add_(0, fl, p)
                    Qf.index_add_(0, fl, q)
            s = left.nonzero()[:, 0]
            a, b, c, fl, ar = a[s], b[s], c[s], flat[s], area[s] / 4
            ab, bc, ca = (a + b) / 2, (b + c) / 2, (c + a) / 2
            a, b, c = torch.cat([a, ab, ca, ab]), torch.cat([ab, b, bc, bc]), torch.cat([ca, bc, c, ca])
            flat, area = fl.repeat(4), ar.repeat(4)
        return P, Q

    def self_terms(self):
        """Own-element entries: the Duffy rule on six sub-triangles for G, the edge rule for E; returns
        (gamma E, G), gamma = i / k."""
        k = self.k
        x, w = (torch.as_tensor(v, device=_DEV) for v in _gauss01(4))
        a, b, c = self.a - self.cen, self.b - self.cen, self.c - self.cen
        ring = [a, (a + b) / 2, b, (b + c) / 2, c, (c + a) / 2]
        G = 0
        for e in range(6):
            p, dp = ring[e], ring[(e + 1) % 6] - ring[e]
            jac = torch.linalg.cross(p, dp).norm(dim=1)
            for i in range(4):
                for j in range(4):
                    r = (x[i] * (p + x[j] * dp)).norm(dim=1)
                    G = G + torch.polar(w[i] * w[j] * jac * x[i] / r / (4 * math.pi), k * r)
        x, w = (torch.as_tensor(v, device=_DEV) for v in _gauss01(3))
        E = k * k * G
        for p, p2 in ((a, b), (b, c), (c, a)):
            pq = p2 - p
            length = pq.norm(dim=1)
            hm = (p * torch.linalg.cross(pq / length[:, None], self.nrm)).sum(-1)
            for part in range(4):
                for i in range(3):
                    d = p + (part + x[i]) / 4 * pq
                    ir = 1 / d.norm(dim=1)
                    E = E + torch.polar(w[i] * length / 4 * ir * hm * ir / (4 * math.pi), k / ir) * \
                        torch.complex(-ir, torch.full_like(ir, k))
        return E * (1j / k), G

    def rows(self, cp, cq, tau=1.0):
        """The operator for column coefficients that carry tau, block of rows by block."""
        sE, sG = self.self_terms()
        diag = cp * sE + cq * sG + 0.5 * tau * (cp - (1j / self.k) * cq)
        step = max(1, 12_000_000 // self.n)
        for r0 in range(0, self.n, step):
            r = torch.arange(r0, min(self.n, r0 + step), device=_DEV)
            P, Q = self.block(self.cen[r], self.nrm[r], self._bm, r0)
            A = P.mul_(cp[None]) if not bool(cq.any()) else P * cp[None] + Q * cq[None]
            A[r - r0, r] = diag[r]
            yield r0, A

    def product(self, cp, cq, x, tau=1.0):
        return torch.cat([A @ x for _, A in self.rows(cp, cq, tau)])

    def matrix(self, cp, cq, tau=1.0):
        return torch.cat([A for _, A in self.rows(cp, cq, tau)])

    def incident(self, x, nx, sources):
        """p_inc and dp_inc / dn along the vectors nx at the points x."""
        p, dp = 0, 0
        for kind, v, amp in sources:
            v = torch.as_tensor(np.asarray(v, np.float64), device=_DEV)
            if kind == "plane":
                v = v / v.norm()
                g = complex(amp) * torch.polar(torch.ones_like(x[:, 0]), self.k * (x @ v))
                p, dp = p + g, dp + 1j * self.k * (nx @ v) * g
            else:
                r = x - v
                R = r.norm(dim=1)
                g = complex(amp) * torch.polar(1 / (4 * math.pi * R), self.k * R)
                p, dp = p + g, dp + g * (1j * self.k - 1 / R) * (r * nx).sum(-1) / R
        return p, dp

    def field(self, x, p, q, sources, tau=1.0):
        out = []
        for xs in x.split(max(1, 12_000_000 // self.n)):
            H, G = self.block(xs, None, self._gh)
            out.append(tau * (H @ p - G @ q))
        return torch.cat(out) + self.incident(x, x, sources)[0]

    def velocity(self, x, p, q, sources, omega):
        out = []
        for ax in range(3):
            v = []
            for xs in x.split(max(1, 12_000_000 // self.n)):
                H, G = self.block(xs, None, self._grad(ax))
                v.append(H @ p - G @ q)
            e = torch.zeros_like(x)
            e[:, ax] = 1
            out.append((torch.cat(v) + self.incident(x, e, sources)[1]) / (1j * omega * RHO))
        return torch.stack(out, dim=1)


def _gmres(A, b, tol=1e-11, steps=300):
    """Plain GMRES with a dense matrix (modified by a second orthogonalisation)."""
    beta = b.norm()
    V, H = [b / beta], torch.zeros(steps + 1, steps, dtype=b.dtype)
    for j in range(steps):
        w = A @ V[j]
        B = torch.stack(V)
        h = B.conj() @ w
        w = w - h @ B
        h2 = B.conj() @ w
        w = w - h2 @ B
        H[:j + 1, j] = (h + h2).cpu()
        H[j + 1, j] = w.norm().cpu()
        V.append(w / w.norm())
        e = torch.zeros(j + 2, dtype=b.dtype)
        e[0] = beta.cpu()
        y = torch.linalg.lstsq(H[:j + 2, :j + 1], e[:, None]).solution[:, 0]
        if float((H[:j + 2, :j + 1] @ y - e).norm()) < tol * float(beta):
            break
    return y.to(b.device) @ torch.stack(V[:-1])


def exact(case, seed):
    d = _inputs(case, seed)
    n, tau = d["n"], -1.0 if case["surface"] == "duct" else 1.0
    if n > 45000:
        return None          # the dense rows take minutes
    t = lambda v, f=torch.complex128: torch.as_tensor(v, device=_DEV).to(f)  # noqa: E731
    one, zero = torch.ones(n, dtype=torch.complex128, device=_DEV), torch.zeros(n, dtype=torch.complex128, device=_DEV)
    if case["kind"] == "product":
        D = _Dense(d["nodes"], d["tris"], 2 * math.pi * case["freq"] / C)
        x = t(d["x"])
        return D.product(one, zero, x.reshape(-1, n).T).T.reshape(x.shape).contiguous()
    if case["kind"] == "field":
        D = _Dense(d["nodes"], d["tris"], 2 * math.pi * case["freq"] / C)
        x, p, q = t(d["points"], torch.float64), t(d["p"]), t(d["q"])
        out = [D.field(x, p, q, d["sources"])]
        if case["velocity"]:
            out.append(D.velocity(x, p, q, d["sources"], 2 * math.pi * case["freq"]))
        return out
    if case["kind"] == "gradient":
        k = 2 * math.pi * case["freq"] / C
        D = _Dense(d["nodes"], d["tris"], k)
        cq = -1j * k * RHO * C * t(d["adm"])[t(d["region"], torch.int64)]
        Ap, Aq = D.matrix(one, zero), D.matrix(zero, one)
        A = Ap.add_(Aq * cq[None])
        pi, dpi = D.incident(D.cen, D.nrm, d["sources"])
        u = torch.linalg.solve(A, (pi - (1j / k) * dpi)[:, None])[:, 0]
        x = t(d["points"], torch.float64)
        H, G = D.block(x, None, D._gh)
        f = H @ u - G @ (cq * u) + D.incident(x, x, d["sources"])[0]
        g = f.conj() @ G
        lam = torch.linalg.solve(A.T, (f.conj() @ H - cq * g)[:, None])
        s = -1j * k * RHO * C * u * (-g - lam[:, 0] @ Aq)
        grad = torch.zeros(8, dtype=torch.complex128, device=_DEV).index_add_(0, t(d["region"], torch.int64), s)
        return f.abs().square().sum(), (2 * grad).conj().resolve_conj()
    ps, qs, fs = [], [], []
    for f in d["freqs"]:
        k, omega = 2 * math.pi * f / C, 2 * math.pi * f
        D = _Dense(d["nodes"], d["tris"], k)
        b = torch.stack([p - (1j / k) * dp for p, dp in
                         (D.incident(D.cen, D.nrm, [s]) for s in d["sources"])] or [zero], dim=1)
        cq, z = zero, zero
        if d["bc_type"] is not None:
            adm = t(d["bc_type"], torch.int64) == bemfmm.ADMI
            cq = torch.where(adm, -1j * k * RHO * C * tau * t(d["adm"])[t(d["region"], torch.int64)], zero)
            z = 1j * omega * RHO * t(d["bc_value"])
            b = b - D.product(zero, tau * one, z[:, None], tau)
        A = D.matrix(tau * one, tau * cq, tau)
        u = torch.stack([_gmres(A, b[:, i]) for i in range(b.shape[1])], dim=1) if n > 16000 else torch.linalg.solve(A, b)
        del A
        ps.append(u.T.contiguous())
        qs.append((cq[:, None] * u + z[:, None]).T.contiguous())
        if d.get("points") is not None:
            fs.append(D.field(t(d["points"], torch.float64), ps[-1][0], qs[-1][0], d["sources"]))
    if case["rhs"] > 1:
        return [list(v) for v in zip(ps, qs)]
    if case["surface"] == "duct":
        return [[p[0], q[0]] for p, q in zip(ps, qs)]
    return [torch.cat(ps), torch.cat(qs), torch.stack(fs) if fs else None]
