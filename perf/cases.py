"""The work a user of this framework has it do, as cases whose time is measured.

    listed()            the cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) what the user's program holds before the call
    run(state)          one pass through the public entry points, and its outputs
    work(case)          bytes and operations the pass cannot do without
    exact(case, seed)   the outputs in 64 bits, without this repository's kernels

A case's "kind" names the call:

    apply    one application of the remainder or the parametrix to a density
    solve    div(a grad u) = f, one or several right-hand sides on one operator
    multi    several coefficient fields in one lockstep batch
    build    a new geometry: near-field quadrature and coefficient, then its corrections
    wave     div(a grad u) + c u = f with c != 0, real of either sign or complex
    edge     a Dirichlet or Neumann problem on an open surface

Surfaces, coefficients and right-hand sides are those of the workloads, with the
surface's position in space and its size, the coefficient and the data drawn from the seed.  Solves take
manufactured data: u = -1/|x - x0| less its mean (c = 0), or u itself.
"""

from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2401_12501_gb300 as pm
from workloads import cubed_sphere, torus, wavy_torus
from workloads import bvp as bands
from workloads.coefficients import smooth_random_coefficient
from workloads.rhs import newtonian_problem
from workloads.trisurfaces import tri_ellipsoid


def listed():
    return [
        # The smallest call: one float32 remainder apply on the validation sphere's
        # 1,536 nodes, as a caller's own Krylov loop issues it.  Launches and latency.
        dict(name="apply_fp32_1536", kind="apply", shape="ellipsoid", m=2, n=0, p=8, op="R",
             prec="fp32"),
        # The float64 apply that checks and open-surface solves stand on; 10 x 10 nodes.
        dict(name="apply_fp64_2400", kind="apply", shape="ellipsoid", m=2, n=0, p=10, op="R",
             prec="fp64"),
        # The N-body use of a fast apply, on a torus large enough for the FMM.
        dict(name="apply_fmm_24576", kind="apply", shape="torus", m=32, n=12, p=8, op="R",
             prec="fmm"),
        # A small served request on a resident operator.
        dict(name="solve_1536", kind="solve", shape="ellipsoid", m=2, n=0, p=8, prec="fp32",
             rhs=1, store=False),
        # An ordinary solve: the 9,600-node ellipsoid with a variable coefficient.
        dict(name="solve_9600", kind="solve", shape="ellipsoid", m=4, n=0, p=10, prec="fp32",
             rhs=1, store=False),
        # The large solve, on the paper's wavy torus at the paper's 58,752 nodes: FMM applies
        # and the operator's stored float-float matrices, the configuration the benchmark uses.
        dict(name="solve_fmm_58752", kind="solve", shape="wavy", m=51, n=18, p=8, prec="fmm",
             rhs=1, store=True),
        # Parameter studies: 8 coefficient fields with 8 right-hand sides each, one batch.
        dict(name="multi_8x8_24576", kind="multi", shape="ellipsoid", m=8, n=0, p=8, fields=8,
             rhs=8),
        # A geometry the program has not seen (a served request that describes its own):
        # quadrilateral patches of the largest usual order, and triangles of order 8.
        dict(name="build_quads_2400", kind="build", shape="ellipsoid", m=2, n=0, p=10),
        dict(name="build_triangles_2880", kind="build", shape="triangles", m=1, n=0, p=8),
        # c != 0: a variable Helmholtz coefficient, and the paper's complex one.
        dict(name="helmholtz_3456", kind="wave", shape="ellipsoid", m=3, n=0, p=8,
             c=4.0,
             sign="positive"),
        dict(name="complex_864", kind="wave", shape="ellipsoid", m=2, n=0, p=6, c=4.0,
             sign="complex"),
        # An open surface: the Dirichlet system on a torus band with 64 nodes an edge.
        dict(name="dirichlet_2048", kind="edge", m=4, n=8, p=8, edge=64, over=32,
             which="dirichlet"),
    ]


# Patch grids (m, n) by shape: 6 m^2 patches of an ellipsoid, m x n of a torus, 20 4^m triangles.
def _shape_of(rng, lo, hi):
    """A surface of about lo to hi nodes (uniform over the logarithm) at a drawn order."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    shape = rng.choice(["ellipsoid", "ellipsoid", "torus", "wavy"])
    p = rng.choice([5, 6, 7, 8, 8, 9, 10])
    if shape == "ellipsoid":
        m = max(1, round(math.sqrt(want / (6 * p * p))))
        return dict(shape=shape, m=m, n=0, p=p)
    ratio = 2.5 if shape == "torus" else 3.0
    n = max(3, round(math.sqrt(want / (ratio * p * p))))
    return dict(shape=shape, m=max(6, round(want / (n * p * p))), n=n, p=p)


def draw(rng):
    kind = rng.choice(["apply", "solve", "solve", "multi", "build", "wave", "edge"])
    if kind == "apply":
        prec = rng.choice(["fp32", "fp32", "fp64", "ff", "fmm"])
        lo, hi = {"fmm": (8000, 24000), "fp64": (400, 5000)}.get(prec, (400, 16000))
        return dict(kind=kind, **_shape_of(rng, lo, hi), op=rng.choice("RK"), prec=prec)
    if kind == "solve":
        prec = rng.choice(["fp32", "fp32", "fmm"])
        lo, hi = (8000, 24000) if prec == "fmm" else (1000, 16000)
        return dict(kind=kind, **_shape_of(rng, lo, hi), prec=prec,
                    rhs=rng.choice([1, 1, 1, 2, 5, 8, 16, 33]), store=rng.random() < 0.3)
    if kind == "multi":
        return dict(kind=kind, **_shape_of(rng, 1000, 16000), fields=rng.randint(2, 8),
                    rhs=rng.randint(1, 8))
    if kind == "build":
        if rng.random() < 0.4:
            return dict(kind=kind, shape="triangles", m=rng.choice([0, 1]), n=0,
                        p=rng.randint(4, 8))
        return dict(kind=kind, **_shape_of(rng, 400, 5000))
    if kind == "wave":
        sign = rng.choice(["positive", "negative", "complex"])
        m, p = (2, rng.randint(5, 6)) if sign == "complex" else (rng.randint(2, 3), rng.randint(6, 8))
        return dict(kind=kind, shape="ellipsoid", m=m, n=0, p=p,
                    c=round(rng.uniform(1.0, 8.0), 2), sign=sign)
    which = rng.choice(["dirichlet", "neumann"])
    m, n = rng.choice([(2, 4), (2, 5), (3, 5), (3, 6), (4, 8)])
    return dict(kind=kind, m=m, n=n, p=rng.randint(6, 9), edge=n * rng.choice([6, 7, 8, 9]),
                over=32 if which == "dirichlet" else 16, which=which)


# ---------------------------------------------------------------- inputs

def _surface(case, rng):
    """The case's surface, turned and scaled: other coordinates, the same near patches."""
    shape, m, n, p = case["shape"], case["m"], case["n"], case["p"]
    if shape == "ellipsoid":
        s = cubed_sphere(m, p, axes=(1.0, 1.5, 2.0))
    elif shape == "torus":
        s = torus(m, n, p)
    elif shape == "wavy":
        s = wavy_torus(m, n, p)
    else:
        s = tri_ellipsoid(m, p, axes=(1.0, 1.5, 2.0))
    Q, _ = np.linalg.qr(rng.standard_normal((3, 3)))
    Q = Q * np.sign(np.linalg.det(Q))
    size = rng.uniform(0.8, 1.25)
    s.nodes, s.normals = size * s.nodes @ Q, s.normals @ Q
    s.tangents = size * np.hstack([s.tangents[:, :3] @ Q, s.tangents[:, 3:] @ Q])
    s.curvature, s.weights = s.curvature / size, s.weights * size ** 2
    return s


def _field(surface, rng):
    return smooth_random_coefficient(surface, int(rng.integers(1 << 31)), amp=0.3)


def _pole(surface, rng):
    """Where the manufactured solution has its pole: well outside the surface."""
    d = rng.standard_normal(3)
    reach = np.linalg.norm(surface.nodes, axis=1).max()
    return d / np.linalg.norm(d) * reach * rng.uniform(2.0, 3.0)


def _wave(case, surface, rng):
    """(a, grad_a, c, f, u) of the paper's variable-coefficient c != 0 examples."""
    x, n = surface.nodes, surface.normals
    s = 1.0 + 0.1 * rng.uniform(-1.0, 1.0, 2)
    flat = lambda g: g - n * np.sum(g * n, 1, keepdims=True)     # noqa: E731
    if case["sign"] == "negative":
        a = 2.0 + 0.5 * s[0] * x[:, 2]
        ga = flat(np.tile([0.0, 0.0, 0.5 * s[0]], (len(x), 1)))
        c = -case["c"] - s[1] * np.exp(x[:, 0] / 2)
    else:
        ez = s[0] * np.exp(x[:, 2])
        a, ga = 1.0 + ez, flat(np.stack([0 * ez, 0 * ez, ez], 1))
        c = case["c"] * s[1] * (1.0 + 0.2 * x[:, 1])
        if case["sign"] == "complex":
            c = c + 0.2j * case["c"] * s[1] * np.sin(x[:, 0])
    d = x - _pole(surface, rng)
    rho = np.linalg.norm(d, axis=1)
    v, grad = -1.0 / rho, d / rho[:, None] ** 3
    dn = np.sum(grad * n, 1)
    dnn = 1.0 / rho ** 3 - 3.0 * np.sum(d * n, 1) ** 2 / rho ** 5
    f = np.sum(ga * (grad - n * dn[:, None]), 1) + a * (-2.0 * surface.curvature * dn - dnn) + c * v
    return a, ga, c, f, v


def _edge(case, rng):
    """The open surface, its coefficient, (f, f_gamma) and the exact u."""
    band = bands.torus_band(case["m"], case["n"], case["p"], case["edge"], case["over"],
                            theta0=rng.uniform(0.0, 2.0 * np.pi))
    x0 = _pole(band.surface, rng)
    if case["which"] == "neumann":
        co = bands.band_coefficient(band)
        data = bands.newtonian_neumann(band, co, x0=x0)
    else:
        co = bands.constant_band_coefficient(band)
        data = bands.newtonian_dirichlet(band, x0=x0)
    return band, co, data


def _inputs(case, seed):
    """Everything of a case that the seed decides, as numpy arrays."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "edge":
        return _edge(case, rng)
    surface = _surface(case, rng)
    if kind == "wave":
        return surface, _wave(case, surface, rng)
    fields = [_field(surface, rng) for _ in range(case.get("fields", 1))]
    if kind == "build":
        return surface, fields[0]
    if kind == "apply":
        return surface, fields[0], surface.nodes[:, 0] + rng.standard_normal(surface.N)
    data = [[newtonian_problem(surface, c, x0=_pole(surface, rng)) for _ in range(case["rhs"])]
            for c in fields]
    F = [np.stack([f for f, _ in d]) for d in data]
    U = [np.stack([u for _, u in d]) for d in data]
    return surface, fields, F, U


# ---------------------------------------------------------------- the calls

@functools.lru_cache(maxsize=None)
def _context():
    return pm.Context(torch.cuda.current_device())


def _operator(surface, coeff, ctx=None):
    s = pm.Surface.from_fixture(ctx or _context(), surface)
    s.set_coeff(coeff.a, coeff.grad_a)
    return s


def prepare(case, seed):
    kind = case["kind"]
    state = dict(case=dict(case))
    if kind == "edge":
        band, co, (f, fg, _) = _inputs(case, seed)
        s = _operator(band.surface, co)
        patch, uv = bands.edge_patches(band)
        if case["which"] == "neumann":
            ae, ao = bands.edge_a(band), bands.edge_a(band, True)
        else:
            ae, ao = np.ones(band.M), np.ones(case["over"] * band.M)
        state.update(surface=s, f=f, fg=fg, bvp=_Problem(
            s, band.curves, ae, ao, patch, uv, kind=case["which"]))
    elif kind == "wave":
        surface, (a, ga, c, f, _) = _inputs(case, seed)
        s = pm.Surface.from_fixture(_context(), surface)
        s.set_coeff_c(a, ga, c)
        state.update(surface=s, f=f.astype(np.complex128))
    elif kind == "build":
        fixture, coeff = _inputs(case, seed)
        _context()
        state.update(fixture=fixture, coeff=coeff)
    elif kind == "apply":
        surface, coeff, sigma = _inputs(case, seed)
        state.update(surface=_operator(surface, coeff), sigma=torch.from_numpy(sigma).cuda())
    else:
        surface, fields, F, _ = _inputs(case, seed)
        # a batch keeps its workspace in the context: each state stands for a program of its own
        ctx = pm.Context(torch.cuda.current_device()) if kind == "multi" else None
        ops = [_operator(surface, fields[0], ctx)]
        for c in fields[1:]:
            ops.append(ops[0].clone())
            ops[-1].set_coeff(c.a, c.grad_a)
        if case.get("store"):
            ops[0].store_ff()
        state.update(ops=ops, F=[torch.from_numpy(f).cuda() for f in F])
    return state


class _Problem(pm.BoundaryValueProblem):
    """Gives its handle back with the state it belongs to, before the surface's."""

    def __del__(self):
        self.close()


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "apply":
        s = state["surface"]
        apply = s.apply_R if case["op"] == "R" else s.apply_K
        out = apply(state["sigma"], prec=case["prec"])
        # a caller who asked for float32 or FMM sums keeps what they are good for
        return out.float() if case["prec"] in ("fp32", "fmm") else out
    if kind == "solve":
        return state["ops"][0].solve(state["F"][0], prec=case["prec"])[0]
    if kind == "multi":
        return pm.solve_multi(state["ops"], state["F"])[0]
    if kind == "build":
        s = _operator(state["fixture"], state["coeff"])
        out = s.get_near()
        s.close()
        return out
    if kind == "wave":
        u, _, sigma = state["surface"].solve_c(state["f"], tol=1e-12, return_sigma=True)
        return u, sigma
    u, _, sigma, mu = state["bvp"].solve(state["f"], state["fg"])
    return u, sigma, mu


# ---------------------------------------------------------------- work

def _nodes(case):
    m, n, p = case["m"], case["n"], case["p"]
    if case["kind"] == "edge" or case["shape"] in ("torus", "wavy"):
        return m * n * p * p
    return 6 * m * m * p * p if case["shape"] == "ellipsoid" else 20 * 4 ** m * p * (p + 1) // 2


def work(case):
    """Geometry and data read once and results written once; the operations of the pass's
    sums over all ordered node pairs with the fewest applies a solve can do (each density
    once through the remainder and once through the parametrix), 26 a pair for the
    remainder and 10 for the parametrix, 100 where the kernel is a Bessel function; for the
    FMM a few hundred neighbours and a few thousand expansion operations a node.  A build's
    are those of its weight sets: about 4 blocks a node, each weight a sum over at least
    256 points of five kernels."""
    N, kind = _nodes(case), case["kind"]
    rhs = case.get("rhs", 1) * case.get("fields", 1)
    per_patch = case["p"] ** 2
    if kind == "build":
        return dict(bytes=N * (14 * 8 + 4 * per_patch * 16), flops=N * 4.0 * per_patch * 256 * 10)
    pair = {"apply": 26 if case.get("op") == "R" else 10, "wave": 2 * 100.0}.get(kind, 36)
    if kind == "edge":
        pairs = float(N) * (N + 2 * case["edge"] * case["over"])
    elif case.get("prec") == "fmm":
        pairs = N * 400.0
    else:
        pairs = float(N) * N * (1 if kind != "multi" else case["fields"])
    flops = pairs * (pair + 2 * (rhs - 1)) + (N * 6000.0 if case.get("prec") == "fmm" else 0.0)
    width = 8 if kind == "wave" else 4
    nbytes = N * (10 * 8 + 4 * per_patch * width + 16 * rhs)
    if case.get("store"):
        nbytes += 9 * N * N
    return dict(bytes=float(nbytes), flops=flops)


# ---------------------------------------------------------------- 64-bit references

def exact(case, seed):
    kind = case["kind"]
    if kind == "edge":
        # the Neumann problem's constant is the method's own choice; the densities have no
        # closed form
        u = None if case["which"] == "neumann" else _inputs(case, seed)[2][2]
        return None if u is None else (u, None, None)
    if kind == "wave":
        # the solution of the equation itself; complex Bessel functions over the quadrature
        # points of a density's reference take minutes
        return _inputs(case, seed)[1][4].astype(np.complex128), None
    if kind == "solve":
        return _inputs(case, seed)[3][0]
    if kind == "multi":
        return _inputs(case, seed)[3]
    if _nodes(case) > 30000:
        return None
    if kind == "build":
        surface, coeff = _inputs(case, seed)
        ref = _Reference(surface, coeff)
        R, K = ref.corrections("RK")
        return None, None, R.cpu().numpy(), K.cpu().numpy()
    surface, coeff, sigma = _inputs(case, seed)
    ref = _Reference(surface, coeff)
    return ref.apply(case["op"], torch.from_numpy(sigma).to(ref.dev))


def _legendre(n, x):
    """P_0 .. P_{n-1} and their derivatives at x, stacked in a last dimension."""
    P, D = [torch.ones_like(x), x], [torch.zeros_like(x), torch.ones_like(x)]
    for k in range(1, n):
        P.append(((2 * k + 1) * x * P[k] - k * P[k - 1]) / (k + 1))
        D.append(D[k - 1] + (2 * k + 1) * P[k])
    return torch.stack(P[:n], -1), torch.stack(D[:n], -1)


class _Reference:
    """The discretised remainder and parametrix of a closed surface in plain 64-bit torch.

    Density and geometry on a patch are the polynomial interpolants of the node data.
    Corrections: a target's own patch by polar quadrature about its node (along each edge
    the variable that keeps the angle's density smooth next to the edge; radial panels
    graded to the node), near patches by subdivision until a cell is smaller than its
    distance, 16 x 16 Gauss points a cell; less the smooth rule's terms."""

    def __init__(self, surface, coeff):
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        put = lambda v: torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64,     # noqa: E731
                                        device=self.dev)
        self.npatch, self.p = surface.npatch, surface.p
        self.N = surface.N
        self.n = self.N // self.npatch
        self.x, self.nrm, self.H = put(surface.nodes), put(surface.normals), put(surface.curvature)
        self.w, self.a, self.g = put(surface.weights), put(coeff.a), put(coeff.grad_a)
        tan = put(surface.tangents)
        self.J = torch.linalg.cross(tan[:, :3], tan[:, 3:]).norm(dim=1)
        self.tri = hasattr(surface, "ref_u")
        p = self.p
        if self.tri:
            self.corners = put([[0, 0], [1, 0], [0, 1]])
            uv = torch.stack([put(surface.ref_u), put(surface.ref_v)], 1)
            pick = [(i, j) for i in range(p) for j in range(p - i)]
        else:
            t = put(np.polynomial.legendre.leggauss(p)[0])
            self.corners = put([[-1, -1], [1, -1], [1, 1], [-1, 1]])
            uv = torch.stack([t.repeat_interleave(p), t.repeat(p)], 1)
            pick = [(i, j) for i in range(p) for j in range(p)]
        self.pick = torch.tensor(pick, device=self.dev).T
        self.uv, self.inv = uv, None
        self.inv = torch.linalg.inv(self._poly(uv)[0])
        self.gt, self.gw = (put(v) for v in np.polynomial.legendre.leggauss(16))

    def _poly(self, uv):
        z = 2.0 * uv - 1.0 if self.tri else uv
        (Pu, Du), (Pv, Dv) = _legendre(self.p, z[..., 0]), _legendre(self.p, z[..., 1])
        i, j = self.pick
        return Pu[..., i] * Pv[..., j], Du[..., i] * Pv[..., j], Pu[..., i] * Dv[..., j]

    def basis(self, uv):
        return self._poly(uv)[0] @ self.inv

    # R and K at r = x - y times a(y), for targets' data broadcast against r
    def _kernels(self, which, r, n, H, a, g):
        r2 = (r * r).sum(-1)
        out = []
        if "R" in which:
            q = (r * n).sum(-1) / r2
            out.append(a * (q * q - H * q) / math.pi + (r * g).sum(-1) / (2 * math.pi * r2))
        if "K" in which:
            out.append(r2.log() / (4 * math.pi))
        return out

    def _radial(self, which):
        """Nodes and weights (times rho) on [0, 1], panels graded to 0: far for the logarithm;
        the remainder is smooth there and loses digits in n . r / r^2 the closer it goes."""
        levels = 16 if "K" in which else 4
        br = [0.0] + [2.0 ** -k for k in range(levels, -1, -1)]
        h = [0.5 * (b - a) for a, b in zip(br, br[1:])]
        t = torch.cat([a + s * (self.gt + 1.0) for a, s in zip(br, h)])
        w = torch.cat([s * self.gw for s in h])
        return t, w * t

    def _polar(self, x0, which):
        """Points and weights of the polar rule about x0, a point inside the reference cell."""
        rho, wr = self._radial(which)
        pts, wts = [], []
        for va, vb in zip(self.corners, self.corners.roll(-1, 0)):
            e = (vb - va) / (vb - va).norm()
            s0 = ((x0 - va) * e).sum()
            foot = va + s0 * e
            d = (foot - x0).norm()
            lo, hi = (float(torch.asinh(v / d)) for v in (-s0, (vb - va).norm() - s0))
            k = max(1, math.ceil((hi - lo) / 0.5))
            mid = torch.tensor([lo + (hi - lo) * (q + 0.5) / k for q in range(k)], device=self.dev,
                               dtype=torch.float64)
            half = 0.5 * (hi - lo) / k
            eta = (mid[:, None] + half * self.gt).reshape(-1)
            weta = (half * self.gw).repeat(k)
            ray = foot + d * torch.sinh(eta)[:, None] * e - x0
            L2 = (ray * ray).sum(1)
            pts.append((x0 + rho[None, :, None] * ray[:, None, :]).reshape(-1, 2))
            wts.append(((weta / torch.cosh(eta) * L2)[:, None] * wr).reshape(-1))
        return torch.cat(pts), torch.cat(wts)

    def _self_weights(self, which):
        X = self.x.view(self.npatch, self.n, 3)
        J = self.J.view(self.npatch, self.n)
        _, Du, Dv = self._poly(self.uv)
        normal = torch.linalg.cross(torch.einsum("ij,pjc->pic", Du @ self.inv, X),
                                    torch.einsum("ij,pjc->pic", Dv @ self.inv, X))
        normal = normal / normal.norm(dim=2, keepdim=True)
        out = [torch.empty(self.npatch, self.n, self.n, device=self.dev, dtype=torch.float64)
               for _ in which]
        rows = lambda v: v.view(self.npatch, self.n, *v.shape[1:])       # noqa: E731
        H, a, g = rows(self.H), rows(self.a), rows(self.g)
        for loc in range(self.n):
            pts, wts = self._polar(self.uv[loc], which)
            B = self.basis(pts)
            step = max(1, 24_000_000 // len(pts))
            for s in range(0, self.npatch, step):
                P = slice(s, min(s + step, self.npatch))
                fields = torch.cat([X[P] - X[P, loc:loc + 1], J[P, :, None]], 2)
                y = torch.einsum("qn,pnc->pqc", B, fields)
                at = lambda v: v[P, loc][:, None]                        # noqa: E731
                ks = self._kernels(which, -y[..., :3], at(normal), at(H), at(a), at(g))
                for o, k in zip(out, ks):
                    o[P, loc] = (k * y[..., 3] * wts) @ B
        return [o.view(self.N, self.n) for o in out]

    def _near_pairs(self):
        """(target, patch) of all near pairs but the own patch, by target, then patch."""
        img = torch.einsum("cn,pnd->pcd", self.basis(self.corners), self.x.view(self.npatch, self.n, 3))
        cen = img.mean(1)
        rad = (img - cen[:, None]).norm(dim=2).amax(1)
        found = []
        for s in range(0, self.N, 4096):
            d = (self.x[s:s + 4096, None] - cen).norm(dim=2) < 1.5 * rad
            t, P = d.nonzero(as_tuple=True)
            keep = P != (t + s) // self.n
            found.append(torch.stack([t[keep] + s, P[keep]]))
        return torch.cat(found, 1)

    def _near_weights(self, which, tgt, patch):
        X, J = self.x.view(self.npatch, self.n, 3), self.J.view(self.npatch, self.n)
        out = [torch.zeros(len(tgt), self.n, device=self.dev, dtype=torch.float64) for _ in which]
        o, e1, e2 = (self.corners[0], self.corners[1] - self.corners[0],
                     self.corners[-1] - self.corners[0])
        cells = torch.cat([o, e1, e2]).repeat(len(tgt), 1)
        pair = torch.arange(len(tgt), device=self.dev)
        s, t = (0.5 * (self.gt + 1.0)).repeat_interleave(16), (0.5 * (self.gt + 1.0)).repeat(16)
        wq = (0.25 * self.gw[:, None] * self.gw).reshape(-1)
        if self.tri:
            wq, s = wq * (1.0 - t), s * (1.0 - t)
        st = torch.stack([s, t], 1)
        tests = torch.tensor([[0, 0], [1, 0], [0, 1], [1 / 3, 1 / 3]] if self.tri else
                             [[0, 0], [1, 0], [1, 1], [0, 1], [0.5, 0.5]], device=self.dev,
                             dtype=torch.float64)

        def points(c, st):
            return c[:, None, :2] + st[:, :1] * c[:, None, 2:4] + st[:, 1:] * c[:, None, 4:]

        for depth in range(13):
            split = torch.zeros(len(pair), dtype=torch.bool, device=self.dev)
            for b in range(0, len(pair), 1024):
                c, pr = cells[b:b + 1024], pair[b:b + 1024]
                # which cells are too close for their size
                y = self.basis(points(c, tests)) @ X[patch[pr]]
                size = (y[:, :-1] - y[:, -1:]).norm(dim=2).amax(1)
                dist = (self.x[tgt[pr]] - y[:, -1]).norm(dim=1)
                sp = (dist < 2.2 * size) if depth < 12 else torch.zeros_like(dist, dtype=torch.bool)
                split[b:b + 1024] = sp
                c, pr = c[~sp], pr[~sp]
                if not len(pr):
                    continue
                B = self.basis(points(c, st))
                i = tgt[pr]
                y = torch.bmm(B, torch.cat([X[patch[pr]] - self.x[i, None], J[patch[pr], :, None]], 2))
                area = (c[:, 2] * c[:, 5] - c[:, 3] * c[:, 4]).abs()[:, None]
                ks = self._kernels(which, -y[..., :3], self.nrm[i, None], self.H[i, None],
                                   self.a[i, None], self.g[i, None])
                for w, k in zip(out, ks):
                    w.index_add_(0, pr, torch.bmm((k * y[..., 3] * wq * area)[:, None], B)[:, 0])
            c, pair = cells[split], pair[split]
            if not len(pair):
                break
            o, e1, e2 = c[:, :2], 0.5 * c[:, 2:4], 0.5 * c[:, 4:]
            last = torch.cat([o + e1 + e2, -e1, -e2] if self.tri else [o + e1 + e2, e1, e2], 1)
            cells = torch.cat([torch.cat([o, e1, e2], 1), torch.cat([o + e1, e1, e2], 1),
                               torch.cat([o + e2, e1, e2], 1), last])
            pair = pair.repeat(4)
        return out

    def _blocks(self, which):
        """Targets and patches of all blocks (each target's own patch first) and the
        corrections of every kernel in `which`."""
        own = torch.arange(self.N, device=self.dev)
        near = self._near_pairs()
        i = torch.cat([own, near[0]])
        P = torch.cat([own // self.n, near[1]])
        order = torch.argsort(i, stable=True)
        own = [self._self_weights(k)[0] for k in which]
        W = [torch.cat([s, q])[order] for s, q in zip(own, self._near_weights(which, *near))]
        i, P = i[order], P[order]
        k = P[:, None] * self.n + torch.arange(self.n, device=self.dev)
        same = k == i[:, None]
        r = self.x[i, None] - self.x[k]
        r[same] = 1.0
        G = self._kernels(which, r, self.nrm[i, None], self.H[i, None], self.a[i, None],
                          self.g[i, None])
        return i, k, [(w - torch.where(same, 0.0, self.w[k] * g)) / self.a[k] for w, g in zip(W, G)]

    def corrections(self, which):
        return self._blocks(which)[2]

    def apply(self, op, sigma):
        i, k, (C,) = self._blocks(op)
        out = torch.zeros_like(sigma).index_add_(0, i, (C * sigma[k]).sum(1))
        s = self.w * sigma / self.a
        step = max(1, 30_000_000 // self.N)
        for b in range(0, self.N, step):
            t = slice(b, min(b + step, self.N))
            r = self.x[t, None] - self.x
            diag = (torch.arange(t.stop - b, device=self.dev), torch.arange(b, t.stop, device=self.dev))
            r[diag] = 1.0
            (G,) = self._kernels(op, r, self.nrm[t, None], self.H[t, None], self.a[t, None],
                                 self.g[t, None])
            G[diag] = 0.0
            out[t] += G @ s
        return out
