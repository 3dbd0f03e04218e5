"""The work that a user of this library has it do, as cases that can be timed.

Each case is one call (or one short sequence of calls) of the Python front end
on a scene whose meshes, media and vectors are made here from the case's plain
values and a seed.  The scenes have the shapes, media and sizes of the
library's own scenes: a penetrable sphere, five ribs between a fat slab and a
liver in front of a 256-piston bowl, and a kidney inside a hollow fat shell.

Result types: operators at FP64, native or assembled, return complex128.  What
is computed in single precision (the FP32 and split-BF16 operators, the field)
or to a solver's tolerance comes from the library in complex128 containers and
is kept here as complex64, the precision that it has.

`exact` evaluates the same discretisation in 64 bits with torch: P1 Galerkin,
6-point rule, Sauter-Schwab rules for touching triangles, a collapsed
Gauss-Legendre rule for near ones.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1910_01011_gb300 import api

DEV = "cuda"
PRECISION = {"fp32": api.FP32, "fp64": api.FP64, "bf16x3": api.BF16X3, "fp64_assembled": api.FP64_ASSEMBLED}

# (sound speed m/s, density kg/m^3, attenuation at 1 MHz in Np/m, its power of the frequency)
WATER, FAT = (1500.0, 1000.0, 0.0, 2.0), (1478.0, 950.0, 0.0, 1.0)
LIVER, BONE, KIDNEY = (1570.0, 1060.0, 0.0, 1.3), (2800.0, 1900.0, 47.0, 1.0), (1560.0, 1050.0, 0.0, 1.0)


# ---------------------------------------------------------------- the cases


def listed():
    return [
        # one vector on a very small surface: launches and host work are all there is
        dict(name="fp32_smallest", run="apply", scene="sphere", h=0.38, precision="fp32", rhs=1),
        # an ordinary matrix-free product on a scene of three domains, resolved by its mesh (k h = 1)
        dict(name="fp32_ribs", run="apply", scene="ribs", h=6.1e-3, precision="fp32", rhs=1),
        # the headline product: 41k triangles at 0.5 MHz
        dict(name="fp32_ribs_full", run="apply", scene="ribs", h=2.65e-3, mhz=0.5, precision="fp32", rhs=1),
        # one block GMRES step's product where the operator is too large to be assembled
        dict(name="fp32_kidney_16rhs", run="apply", scene="kidney", h=4.1e-3, precision="fp32", rhs=16),
        # the residual of a matrix-free mixed-precision solve, one excitation
        dict(name="fp64_sphere", run="apply", scene="sphere", h=0.151, precision="fp64", rhs=1),
        # the same for a block of excitations, attenuating domain, odd count
        dict(name="fp64_ribs_5rhs", run="apply", scene="ribs", h=10.1e-3, precision="fp64", rhs=5),
        # one block GMRES step's product with the assembled operator
        dict(name="bf16x3_ribs_16rhs", run="apply", scene="ribs", h=3.75e-3, precision="bf16x3", rhs=16),
        # the residual of a block of excitations with the assembled operator
        dict(name="fp64_assembled_ribs_16rhs", run="apply", scene="ribs", h=5.3e-3, precision="fp64_assembled", rhs=16),
        # a new exterior medium: near field and both assembled operators anew, and their first products
        dict(name="new_medium_ribs", run="medium", scene="ribs", h=8.3e-3, rhs=3),
        # the single-sphere problem with a plane wave: mixed precision, matrix-free, one excitation
        dict(name="solve_sphere", run="solve_wave", scene="sphere", h=0.151),
        # a planning request: 16 excitations of the bowl, block GMRES on assembled operators
        dict(name="solve_ribs_16exc", run="solve_block", scene="ribs", h=6.1e-3, exc=16),
        # the total field of a solved excitation on the paper's 200 x 200 grid
        dict(name="field_sphere_grid", run="field", scene="sphere", h=0.151, n=200),
    ]


def draw(rng):
    def size(lo, hi):
        return float("%.3g" % math.exp(rng.uniform(math.log(lo), math.log(hi))))

    def count(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["fp32", "fp32", "fp32_multi", "fp64", "fp64_multi", "bf16x3", "fp64_assembled", "medium", "solve_wave",
                       "solve_block", "field"])
    scene = rng.choice(["sphere", "ribs", "kidney"])
    if kind == "fp32":
        h = {"sphere": size(0.05, 0.5), "ribs": size(2.7e-3, 15e-3), "kidney": size(1.9e-3, 9e-3)}[scene]
        return dict(run="apply", scene=scene, h=h, precision="fp32", rhs=1)
    if kind == "fp32_multi":
        h = {"sphere": size(0.06, 0.5), "ribs": size(5.5e-3, 15e-3), "kidney": size(4.1e-3, 9e-3)}[scene]
        return dict(run="apply", scene=scene, h=h, precision="fp32", rhs=count(2, 16))
    if kind in ("fp64", "fp64_multi"):
        h = {"sphere": size(0.1, 0.5), "ribs": size(9e-3, 18e-3), "kidney": size(6e-3, 12e-3)}[scene]
        return dict(run="apply", scene=scene, h=h, precision="fp64", rhs=1 if kind == "fp64" else count(2, 8))
    if kind in ("bf16x3", "fp64_assembled"):
        h = {"sphere": size(0.06, 0.4), "ribs": size(5e-3, 15e-3), "kidney": size(3.9e-3, 9e-3)}[scene]
        return dict(run="apply", scene=scene, h=h, precision=kind, rhs=count(1, 64 if kind == "bf16x3" else 16))
    if kind == "medium":
        h = {"sphere": size(0.11, 0.4), "ribs": size(8e-3, 15e-3), "kidney": size(6.5e-3, 9e-3)}[scene]
        return dict(run="medium", scene=scene, h=h, rhs=count(1, 8))
    if kind == "solve_wave":
        return dict(run="solve_wave", scene="sphere", h=size(0.13, 0.4))
    if kind == "solve_block":
        h = {"sphere": size(0.1, 0.3), "ribs": size(6.5e-3, 12e-3), "kidney": size(5e-3, 9e-3)}[scene]
        return dict(run="solve_block", scene=scene, h=h, exc=count(2, 16))
    return dict(run="field", scene="sphere", h=size(0.12, 0.4), n=count(20, 400))


# ---------------------------------------------------------------- meshes, media, vectors


def _surface(semi, p, h, centre=(0.0, 0.0, 0.0), inward=False):
    """Closed surface |x/a|^p + |y/b|^p + |z/c|^p = 1: a lattice of spacing about h on the
    box around it, projected radially (equiangular for p = 2)."""
    semi = np.asarray(semi, dtype=np.float64)
    m = np.maximum(1, np.ceil(2.0 * semi / h - 1e-9).astype(np.int64))
    quads = []
    for ax in range(3):
        u, w = (ax + 1) % 3, (ax + 2) % 3
        i, j = (a.ravel() for a in np.meshgrid(np.arange(m[u]), np.arange(m[w]), indexing="ij"))
        for side in (0, 1):
            q = np.zeros((i.size, 4, 3), dtype=np.int64)
            q[:, :, ax] = side * m[ax]
            q[:, :, u] = i[:, None] + np.array([0, 1, 1, 0])
            q[:, :, w] = j[:, None] + np.array([0, 0, 1, 1])
            quads.append(q if side else q[:, ::-1])
    quads = np.concatenate(quads)
    key = (quads[..., 0] * (m[1] + 1) + quads[..., 1]) * (m[2] + 1) + quads[..., 2]
    _, first, idx = np.unique(key.ravel(), return_index=True, return_inverse=True)
    idx = idx.reshape(-1, 4)
    tris = np.concatenate([idx[:, [0, 1, 2]], idx[:, [0, 2, 3]]], axis=1).reshape(-1, 3).astype(np.int32)
    q = -1.0 + 2.0 * quads.reshape(-1, 3)[first] / m
    x = (np.tan(q * (math.pi / 4.0)) if p == 2.0 else q) * semi
    v = x / (np.abs(x / semi) ** p).sum(axis=1, keepdims=True) ** (1.0 / p) + np.asarray(centre)
    return v, (tris[:, [0, 2, 1]].copy() if inward else tris)


def _joined(parts):
    off = np.cumsum([0] + [v.shape[0] for v, _ in parts])
    return np.concatenate([v for v, _ in parts]), np.concatenate([t + o for (_, t), o in zip(parts, off)]).astype(np.int32)


@functools.lru_cache(maxsize=32)
def _meshes(scene, h):
    if scene == "sphere":
        return (_surface((1.0, 1.0, 1.0), 2.0, h * 4.0 / math.pi),)
    if scene == "ribs":
        ribs = [_surface((50e-3, 6e-3, 4e-3), 4.0, h, (0.0, (i - 2) * 18e-3, 40e-3)) for i in range(5)]
        return (_joined(ribs), _surface((75e-3, 75e-3, 10e-3), 6.0, h, (0.0, 0.0, 62e-3)),
                _surface((60e-3, 50e-3, 40e-3), 2.0, h, (0.0, 0.0, -12e-3)))
    a = np.array([55e-3, 30e-3, 20e-3])
    return (_surface(a, 2.0, h), _joined([_surface(a + 8e-3, 2.0, h), _surface(a + 1e-3, 2.0, h, inward=True)]))


class _Scene:
    """Meshes with their media: k0, rho0, and per domain k and rho."""

    def __init__(self, case):
        self.kind, self.h = case["scene"], case["h"]
        self.meshes = _meshes(self.kind, self.h)
        if self.kind == "sphere":
            # nondimensional: k h = 0.75, as 1,280 triangles at k = 5
            self.k0 = complex(0.75 / self.h)
            self.rho0, self.k, self.rho, self.omega_rho0 = 1.0, [1.05 * self.k0], [1.1], 2.6
            self.r_eps = 0.1
        else:
            f = case["mhz"] * 1e6 if "mhz" in case else 1500.0 / (2.0 * math.pi * self.h)
            self.k0, self.rho0 = _k(WATER, f), WATER[1]
            media = (BONE, FAT, LIVER) if self.kind == "ribs" else (KIDNEY, FAT)
            self.k, self.rho = [_k(m, f) for m in media], [m[1] for m in media]
            self.omega_rho0 = 2.0 * math.pi * f * self.rho0
            self.r_eps = (1e-4 if self.kind == "ribs" else 1e-3) * 1e6 / f
        self.n = sum(2 * v.shape[0] for v, _ in self.meshes)
        self.nt = [t.shape[0] for _, t in self.meshes]

    def context(self, **opts):
        c = api.Context(**opts)
        c.set_exterior(self.k0, self.rho0)
        for (v, t), k, rho in zip(self.meshes, self.k, self.rho):
            c.add_domain(v, t, k, rho)
        return c

    def interactions(self):
        """Point pairs and wavenumbers of one product: every pair at k0, pairs within a domain at its own k too."""
        return 36.0 * (sum(self.nt) ** 2 + sum(n * n for n in self.nt))


def _k(medium, f):
    c, _, alpha, power = medium
    return complex(2.0 * math.pi * f / c, alpha * (f / 1e6) ** power)


def _vectors(scene, rhs, seed):
    """Traces as the iterations meet them: a few plane waves of the exterior and a rough part, system order."""
    rng = np.random.default_rng([seed, 11])
    out = np.empty((rhs, scene.n), dtype=np.complex128)
    for r in range(rhs):
        d = rng.standard_normal((4, 3))
        d /= np.linalg.norm(d, axis=1, keepdims=True)
        at = 0
        for v, _ in scene.meshes:
            for block in range(2):
                a = rng.standard_normal(4) + 1j * rng.standard_normal(4)
                wave = np.exp(1j * scene.k0.real * (v @ d.T)) @ a
                rough = rng.standard_normal(v.shape[0]) + 1j * rng.standard_normal(v.shape[0])
                out[r, at:at + v.shape[0]] = (wave + 0.2 * rough) * (abs(scene.k0) if block == 0 else 1.0)
                at += v.shape[0]
    return torch.from_numpy(out if rhs > 1 else out[0]).to(DEV)


def _bowl(scene, seed):
    """Pistons on a spherical bowl that face its focus: a spiral of equal areas on the cap."""
    n, R, aperture, radius, focus = (32, 4.0, 4.0, 0.2, 0.0) if scene.kind == "sphere" else (256, 0.18, 0.2, 3e-3, 0.0)
    turn = np.random.default_rng([seed, 12]).uniform(0.0, 2.0 * math.pi)
    i = np.arange(n) + 0.5
    cz = 1.0 - (1.0 - math.cos(math.asin(aperture / 2.0 / R))) * i / n
    phi = turn + math.pi * (3.0 - math.sqrt(5.0)) * i
    sz = np.sqrt(1.0 - cz * cz)
    d = np.stack([sz * np.cos(phi), sz * np.sin(phi), cz], axis=1)
    return focus + R * d, -d, np.full(n, radius)


def _direction(seed):
    d = np.random.default_rng([seed, 13]).standard_normal(3)
    return d / np.linalg.norm(d)


def _grid(n):
    """n x n points over +-3 radii through the centre, those within 5 % of the surface left out."""
    g = np.linspace(-3.0, 3.0, n)
    x, z = np.meshgrid(g, g)
    pts = np.stack([x.ravel(), np.zeros(x.size), z.ravel()], axis=1)
    r = np.linalg.norm(pts, axis=1)
    pts = pts[np.abs(r - 1.0) > 0.05]
    return pts, np.where(np.linalg.norm(pts, axis=1) < 1.0, 0, -1).astype(np.int32)


def _medium(scene, seed):
    """The exterior medium of a step of a sweep: another sound speed of the couplant."""
    return scene.k0 * (1.0 + 0.02 * np.random.default_rng([seed, 14]).uniform(-1.0, 1.0))


# ---------------------------------------------------------------- prepare and run

WAVE = dict(precision=api.FP32, tol=1e-8, restart=100, operator_mode=0)
BLOCK = dict(precision=api.FP32, tol=1e-8, restart=100, operator_mode=1, batch_rhs=16, block_gmres=1)


def prepare(case, seed):
    s = _Scene(case)
    st = dict(case=case, scene=s)
    if case["run"] == "apply":
        c = s.context()
        st["x"] = _vectors(s, case["rhs"], seed)
        c.apply(st["x"], precision=PRECISION[case["precision"]])  # a program's first product sets the operator up
    elif case["run"] == "medium":
        c = s.context()
        st["x"], st["k0"] = _vectors(s, case["rhs"], seed), _medium(s, seed)
        c.apply(st["x"], precision=api.BF16X3)
        c.apply(st["x"], precision=api.FP64_ASSEMBLED)
    elif case["run"] in ("solve_wave", "field"):
        c = s.context(n_pade=4, r_eps=s.r_eps)
        c.set_plane_wave(_direction(seed))
        c.solve(**WAVE)
        if case["run"] == "field":
            st["points"], st["domain"] = _grid(case["n"])
    else:
        c = s.context(n_pade=8, r_eps=s.r_eps)
        c.set_transducer(*_bowl(s, seed), s.omega_rho0)
        n_elem = 32 if s.kind == "sphere" else 256
        st["w"] = np.exp(2j * math.pi * np.random.default_rng([seed, 15]).random((case["exc"], n_elem)))
        c.set_excitations(st["w"])
        c.solve(**BLOCK)
    st["ctx"] = c
    return st


def run(st):
    case, c = st["case"], st["ctx"]
    if case["run"] == "apply":
        y = c.apply(st["x"], precision=PRECISION[case["precision"]])
        return y if case["precision"].startswith("fp64") else y.to(torch.complex64)
    if case["run"] == "medium":
        c.set_exterior(st["k0"], st["scene"].rho0)
        y32 = c.apply(st["x"], precision=api.BF16X3)
        return [y32.to(torch.complex64), c.apply(st["x"], precision=api.FP64_ASSEMBLED)]
    if case["run"] == "field":
        return c.field(st["points"], st["domain"]).astype(np.complex64)
    if case["run"] == "solve_wave":
        c.solve(**WAVE)
        return c.solution().astype(np.complex64)
    c.set_excitations(st["w"])
    c.solve(**BLOCK)
    return np.stack([c.solution(i) for i in range(case["exc"])]).astype(np.complex64)


def work(case):
    """One evaluation of the kernels per interaction (73 operations for one vector, 29 more for each
    further one), or one pass over the assembled operator; vectors read and written once."""
    s = _Scene(case)
    inter, vec = s.interactions(), 16.0 * s.n
    geometry = 6.0 * 16.0 * sum(s.nt)
    if case["run"] == "apply" and not case["precision"].endswith(("x3", "assembled")):
        r = case["rhs"]
        return {"bytes": 2 * r * vec + geometry, "flops": inter * (73 + 29 * (r - 1))}
    if case["run"] == "apply":
        r, entry = case["rhs"], 8.0 if case["precision"] == "bf16x3" else 16.0
        return {"bytes": entry * s.n ** 2 + 2 * r * vec, "flops": 8.0 * s.n ** 2 * r}
    if case["run"] == "medium":
        return {"bytes": 24.0 * s.n ** 2 + 3 * case["rhs"] * vec, "flops": 2 * 73 * inter + 16.0 * s.n ** 2 * case["rhs"]}
    if case["run"] == "field":
        return {"bytes": geometry + 44.0 * case["n"] ** 2, "flops": 60.0 * case["n"] ** 2 * 6 * sum(s.nt)}
    if case["run"] == "solve_wave":  # ten iterations, one residual before and one after
        return {"bytes": 12 * (2 * vec + geometry), "flops": 12 * 73 * inter}
    return {"bytes": 30 * 8.0 * s.n ** 2, "flops": 30 * 8.0 * s.n ** 2 * case["exc"]}  # thirty block steps


# ---------------------------------------------------------------- the same in 64 bits


def _rule6():
    """The symmetric degree-4 rule of six points on a triangle: (lambda [6, 3], weights that sum to 1)."""
    s10, root = math.sqrt(10.0), math.sqrt(38.0 - 44.0 * math.sqrt(0.4))
    lam, wts = [], []
    for sign in (1.0, -1.0):
        a = (8.0 - s10 + sign * root) / 18.0
        w = (620.0 + sign * math.sqrt(213125.0 - 53320.0 * s10)) / 3720.0
        for p in ((a, a, 1 - 2 * a), (a, 1 - 2 * a, a), (1 - 2 * a, a, a)):
            lam.append(p)
            wts.append(w)
    return np.array(lam), np.array(wts)


def _pair_rules():
    """Rules of a pair by its number of common vertices: s [m, 2] and t [m, 2] on 0 <= s2 <= s1 <= 1, weights."""
    x, w = np.polynomial.legendre.leggauss(6)
    x, w = 0.5 * (x + 1.0), 0.5 * w
    g = [a.ravel() for a in np.meshgrid(x, x, x, x, indexing="ij")]
    wt = np.prod([a.ravel() for a in np.meshgrid(w, w, w, w, indexing="ij")], axis=0)
    o, a, b, c = g
    near = [((o, o * a), (b, b * c), o * b)]
    vertex = [((o, o * a), (o * b, o * b * c), o ** 3 * b), ((o * b, o * b * c), (o, o * a), o ** 3 * b)]
    j = o ** 3 * a ** 2
    edge = [((o, o * a * c), (o * (1 - a * b), o * a * (1 - b)), j)]
    for p, q in (((o, o * a), (o * (1 - a * b * c), o * a * b * (1 - c))),
                 ((o * (1 - a * b), o * a * (1 - b)), (o, o * a * b * c)),
                 ((o * (1 - a * b * c), o * a * b * (1 - c)), (o, o * a)),
                 ((o * (1 - a * b * c), o * a * (1 - b * c)), (o, o * a * b))):
        edge.append((p, q, j * b))
    same = []
    for p, q in (((o, o * (1 - a + a * b)), (o * (1 - a * b * c), o * (1 - a))),
                 ((o, o * a * (1 - b + b * c)), (o * (1 - a * b), o * a * (1 - b))),
                 ((o * (1 - a * b * c), o * a * (1 - b * c)), (o, o * a * (1 - b)))):
        same += [(p, q, j * b), (q, p, j * b)]
    out = []
    for maps in (near, vertex, edge, same):
        s = np.concatenate([np.stack(m[0], axis=1) for m in maps])
        t = np.concatenate([np.stack(m[1], axis=1) for m in maps])
        out.append((s, t, np.concatenate([wt * m[2] for m in maps])))
    return out


def _kernels(d, k):
    """G = e^{ikr} / (4 pi r) and its radial factor F = G (ik - 1/r) / r for differences d [..., 3]."""
    r = d.square().sum(-1).sqrt()
    g = torch.polar(torch.exp(-k.imag * r) / (4.0 * math.pi * r), k.real * r)
    return g, g * torch.complex(-k.imag - 1.0 / r, torch.full_like(r, k.real)) / r


class _Exact:
    """Products with the system matrix of a scene, in 64 bits on the GPU."""

    def __init__(self, scene, k0=None):
        self.s, self.k0 = scene, complex(scene.k0 if k0 is None else k0)
        vo, P, V, dom = 0, [], [], []
        for j, (v, t) in enumerate(scene.meshes):
            P.append(v[t])
            V.append(t.astype(np.int64) + vo)
            dom.append(np.full(t.shape[0], j))
            vo += v.shape[0]
        self.nv = vo
        self.P, self.V, self.dom = (torch.from_numpy(np.concatenate(a)).to(DEV) for a in (P, V, dom))
        # positions in system order: per domain [psi; phi]
        psi, phi, at = [], [], 0
        for v, _ in scene.meshes:
            psi.append(np.arange(v.shape[0]) + at)
            phi.append(np.arange(v.shape[0]) + at + v.shape[0])
            at += 2 * v.shape[0]
        self.psi, self.phi = (torch.from_numpy(np.concatenate(a)).to(DEV) for a in (psi, phi))
        e = torch.linalg.cross(self.P[:, 1] - self.P[:, 0], self.P[:, 2] - self.P[:, 0])
        ln = e.norm(dim=1)
        self.nrm, self.area = e / ln[:, None], 0.5 * ln
        self.curl = (self.P[:, [1, 2, 0]] - self.P[:, [2, 0, 1]]) / ln[:, None, None]  # [T, vertex, 3]
        lam, w = (torch.from_numpy(a).to(DEV) for a in _rule6())
        self.lam = lam
        self.pts = torch.einsum("qa,tac->tqc", lam, self.P)
        self.w = self.area[:, None] * w  # [T, 6]

    def densities(self, X):
        """Of X [R, N]: weighted psi and phi at the points [T, 6, R], weighted curls [T, 3, R]."""
        ps, ph = X[:, self.psi].T[self.V], X[:, self.phi].T[self.V]  # [T, 3, R]
        lam = self.lam.to(torch.complex128)
        d1 = torch.einsum("qa,tar->tqr", lam, ps) * self.w[:, :, None]
        d2 = torch.einsum("qa,tar->tqr", lam, ph) * self.w[:, :, None]
        return d1, d2, torch.einsum("tac,tar->tcr", self.curl.to(torch.complex128), ph), ps, ph

    def coefficients(self, j, slot):
        r = self.s.rho[j] / self.s.rho0
        return (r, 1.0 / r, complex(self.s.k[j])) if slot else (1.0, 1.0, self.k0)

    def times(self, X):
        R, T = X.shape[0], self.P.shape[0]
        d1, d2, curl, ps, ph = self.densities(X)
        loc = torch.zeros(2, T, 3, R, dtype=torch.complex128, device=DEV)  # tested rows per triangle
        lamw = (self.lam[None] * self.w[:, :, None]).to(torch.complex128)  # [T, 6, 3]
        self._near(loc, ps, ph)
        for j in range(len(self.s.meshes)):
            own = torch.nonzero(self.dom == j).ravel()
            for slot in (0, 1):
                cV, cW, k = self.coefficients(j, slot)
                src = own if slot else torch.arange(T, device=DEV)
                S = src.numel()
                y, ny = self.pts[src].reshape(-1, 3), self.nrm[src].repeat_interleave(6, 0)
                D1, D2 = d1[src].reshape(-1, R), d2[src].reshape(-1, R)
                Dc = (self.w[src, :, None, None] * curl[src, None]).reshape(S * 6, 3 * R)
                step = max(1, int(2.5e7 // (S * 36)))
                for b in range(0, own.numel(), step):
                    tt = own[b:b + step]
                    x, nx = self.pts[tt].reshape(-1, 3), self.nrm[tt].repeat_interleave(6, 0)
                    d = x[:, None] - y[None]
                    G, F = _kernels(d, k)
                    same = (tt[:, None] == src[None]).repeat_interleave(6, 0).repeat_interleave(6, 1)
                    G, F = G.masked_fill(same, 0.0), F.masked_fill(same, 0.0)
                    n = tt.numel()
                    row1 = cV * (G @ D1) + (F * (d * ny[None]).sum(-1)) @ D2  # -K: (y - x).n_y = -d.n_y
                    row2 = (F * (d * nx[:, None]).sum(-1)) @ D1 - cW * k * k * ((G * (nx @ ny.T)) @ D2)
                    loc[0, tt] += torch.einsum("tqa,tqr->tar", lamw[tt], row1.reshape(n, 6, R))
                    loc[1, tt] += torch.einsum("tqa,tqr->tar", lamw[tt], row2.reshape(n, 6, R))
                    wc = torch.einsum("tq,tqcr->tcr", self.w[tt].to(torch.complex128), (G @ Dc).reshape(n, 6, 3, R))
                    loc[1, tt] += cW * torch.einsum("tac,tcr->tar", self.curl[tt].to(torch.complex128), wc)
        return self._assembled(loc)

    def _assembled(self, loc):
        R = loc.shape[-1]
        rows = torch.zeros(2, self.nv, R, dtype=torch.complex128, device=DEV)
        for i in range(2):
            rows[i].index_add_(0, self.V.ravel(), loc[i].reshape(-1, R))
        Y = torch.empty(R, self.s.n, dtype=torch.complex128, device=DEV)
        Y[:, self.psi], Y[:, self.phi] = rows[0].T, rows[1].T
        return Y

    def _pairs(self):
        """Pairs with their own rule: (targets, sources, common vertices 0-3), near ones by the centroid rule."""
        c = (self.P[:, 0] + self.P[:, 1] + self.P[:, 2]) / 3.0
        h2 = (self.P[:, [1, 2, 0]] - self.P).square().sum(-1).amax(1)
        found = []
        for b in range(0, c.shape[0], 1024):
            common = torch.zeros(min(1024, c.shape[0] - b), c.shape[0], dtype=torch.int8, device=DEV)
            for i in range(3):
                for j in range(3):
                    common += self.V[b:b + 1024, i, None] == self.V[None, :, j]
            dist = (c[b:b + 1024, None] - c[None]).square()
            near = (dist[..., 0] + dist[..., 1] + dist[..., 2]) < 4.0 * torch.maximum(h2[b:b + 1024, None], h2[None])
            t, s = torch.nonzero((common > 0) | near, as_tuple=True)
            found.append((t + b, s, common[t, s].long()))
        return (torch.cat(a) for a in zip(*found))

    def _near(self, loc, ps, ph):
        tgt, src, rel = self._pairs()
        rules = _pair_rules()
        lam6, w6 = _rule6()
        for kind in range(4):
            pick = torch.nonzero(rel == kind).ravel()
            s, t, w = (torch.from_numpy(a).to(DEV) for a in rules[kind])
            ls = torch.stack([1 - s[:, 0], s[:, 0] - s[:, 1], s[:, 1]], 1)  # P1 values at vertices 0, 1, 2
            lt = torch.stack([1 - t[:, 0], t[:, 0] - t[:, 1], t[:, 1]], 1)
            regular = None
            if kind < 3:
                q = torch.from_numpy(lam6).to(DEV)
                w6t = torch.from_numpy(w6).to(DEV)
                regular = (q.repeat_interleave(6, 0), q.repeat(6, 1), -(w6t[:, None] * w6t[None]).ravel())
            step = max(1, int(2.5e7 // w.numel()))
            for b in range(0, pick.numel(), step):
                tt, ss = tgt[pick[b:b + step]], src[pick[b:b + step]]
                # common vertices first, in matching order, on both triangles
                eq = self.V[tt][:, :, None] == self.V[ss][:, None, :]
                on_t = eq.any(2)
                pa = torch.argsort((~on_t).to(torch.int8), dim=1, stable=True)
                match = torch.where(on_t, eq.to(torch.int8).argmax(2), torch.full_like(pa, 3)).gather(1, pa)
                order = torch.full_like(pa, 3)  # place of each source vertex: its match's, else after
                for i in range(3):
                    hit = match[:, i] < 3
                    order[hit, match[hit, i]] = i
                pb = torch.argsort(order, dim=1, stable=True)
                A, B = self.P[tt].gather(1, pa[..., None].expand(-1, -1, 3)), self.P[ss].gather(1, pb[..., None].expand(-1, -1, 3))
                scale = 4.0 * self.area[tt] * self.area[ss]
                parts = [(A, B, ls, lt, w, scale, pa, pb)]
                if regular is not None:
                    keep = torch.arange(3, device=DEV).expand_as(pa)
                    parts.append((self.P[tt], self.P[ss], *regular, 0.25 * scale, keep, keep))
                for A, B, la, lb, wt, sc, ia, ib in parts:
                    d = torch.einsum("ma,pac->pmc", la, A) - torch.einsum("mb,pbc->pmc", lb, B)
                    pp = (la[:, :, None] * lb[:, None, :] * wt[:, None, None]).reshape(-1, 9).to(torch.complex128)
                    nx, ny = self.nrm[tt][:, None], self.nrm[ss][:, None]
                    for slot in (0, 1):
                        for j in range(len(self.s.meshes)):
                            m = torch.nonzero((self.dom[tt] == j) & ((self.dom[ss] == j) | (slot == 0))).ravel()
                            if m.numel() == 0:
                                continue
                            cV, cW, k = self.coefficients(j, slot)
                            G, F = _kernels(d[m], k)
                            z = sc[m, None]
                            Vl = ((G @ pp) * z).reshape(-1, 3, 3)
                            Kl = ((-F * (d[m] * ny[m]).sum(-1)) @ pp * z).reshape(-1, 3, 3)
                            Pl = ((F * (d[m] * nx[m]).sum(-1)) @ pp * z).reshape(-1, 3, 3)
                            t_, s_ = tt[m], ss[m]
                            a_, b_ = ia[m][..., None], ib[m][..., None]
                            cc = torch.einsum("pac,pbc->pab", self.curl[t_], self.curl[s_])
                            cc = cc.gather(1, a_.expand(-1, -1, 3)).gather(2, ib[m][:, None].expand(-1, 3, -1))
                            nn = (self.nrm[t_] * self.nrm[s_]).sum(-1)[:, None, None]
                            Wl = cc * Vl.sum((1, 2))[:, None, None] - k * k * nn * Vl
                            xs, xf = (a[s_].gather(1, b_.expand(-1, -1, a.shape[2])) for a in (ps, ph))
                            y1 = cV * (Vl @ xs) - Kl @ xf
                            y2 = Pl @ xs + cW * (Wl @ xf)
                            back = t_[:, None] * 3 + ia[m]
                            for i, y in enumerate((y1, y2)):
                                loc[i].view(-1, y.shape[2]).index_add_(0, back.ravel(), y.reshape(-1, y.shape[2]))

    def wave_rhs(self, direction):
        """<p, phi_r> and <dp/dn, phi_r> of a unit plane wave, system order."""
        d = torch.from_numpy(direction).to(DEV)
        p = torch.exp(1j * self.k0 * (self.pts @ d))
        loc = torch.stack([p, 1j * self.k0 * (self.nrm @ d)[:, None] * p])
        lamw = (self.lam[None] * self.w[:, :, None]).to(torch.complex128)
        return self._assembled(torch.einsum("tqa,itq->ita", lamw, loc)[..., None])[0]

    def solution(self, direction):
        N = self.s.n
        A = self.times(torch.eye(N, dtype=torch.complex128, device=DEV)).T
        return torch.linalg.solve(A, self.wave_rhs(direction))

    def field(self, u, points, domain, direction):
        d1, d2, _, _, _ = self.densities(u[None])
        x, dom = torch.from_numpy(points).to(DEV), torch.from_numpy(domain).to(DEV)
        out = torch.empty(x.shape[0], dtype=torch.complex128, device=DEV)
        ny = self.nrm.repeat_interleave(6, 0)
        for j in [-1] + list(range(len(self.s.meshes))):
            k = self.k0 if j < 0 else complex(self.s.k[j])
            pick = torch.nonzero(dom == j).ravel()
            src = torch.ones_like(self.dom, dtype=torch.bool) if j < 0 else self.dom == j
            src = src.repeat_interleave(6)
            y, n = self.pts.reshape(-1, 3)[src], ny[src]
            D1, D2 = d1.reshape(-1)[src], d2.reshape(-1)[src]
            step = max(1, int(2.5e7 // y.shape[0]))
            for b in range(0, pick.numel(), step):
                at = pick[b:b + step]
                d = x[at][:, None] - y[None]
                G, F = _kernels(d, k)
                sl, dl = G @ D1, (F * -(d * n[None]).sum(-1)) @ D2
                if j < 0:
                    inc = torch.exp(1j * k * (x[at] @ torch.from_numpy(direction).to(DEV)))
                    out[at] = inc + dl - sl
                else:
                    out[at] = (self.s.rho[j] / self.s.rho0) * sl - dl
        return out


def _short(scene, rhs):
    """Whether a product in 64 bits takes under about 20 seconds (measured: 1.0 + 0.6 rhs ns per interaction)."""
    return scene.interactions() * (1.0 + 0.6 * rhs) < 1.8e10


def exact(case, seed):
    s = _Scene(case)
    if case["run"] == "apply":
        if not _short(s, case["rhs"]):
            return None
        X = _vectors(s, case["rhs"], seed)
        Y = _Exact(s).times(X.reshape(case["rhs"], -1))
        return Y.reshape(X.shape)
    if case["run"] == "medium":
        if not _short(s, case["rhs"]):
            return None
        X = _vectors(s, case["rhs"], seed)
        Y = _Exact(s, _medium(s, seed)).times(X.reshape(case["rhs"], -1)).reshape(X.shape)
        return [Y, Y]
    if case["run"] in ("solve_wave", "field") and s.n <= 1500:
        E, d = _Exact(s), _direction(seed)
        u = E.solution(d)
        return u.cpu().numpy() if case["run"] == "solve_wave" else E.field(u, *_grid(case["n"]), d).cpu().numpy()
    return None  # a dense solve of several thousand unknowns
