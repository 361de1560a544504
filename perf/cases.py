"""The work that a user of this library has it do, as measurable cases.

A case is one call pattern of a time-domain Maxwell program on a tetrahedral
mesh: advance a field by a few LSERK4 steps, evaluate the operator, watch the
energy, hand host buffers through, or advance a batch of packed solves.  Sizes
are those of the repository's workloads and order sweep (about 1.7e7 unknowns at
the large end, 384 tetrahedra at the small end) and odd sizes in between.

`exact` restates the discretisation in 64 bits without the library: Bernstein
polynomials (closed-form mass matrices and derivatives) on Warburton's Warp &
Blend nodes, faces matched by their vertex numbers.
"""
from __future__ import annotations

import functools
import itertools
import math
import random

import numpy as np
import torch

import paper_0901_1024_gb300 as dg

DEV = "cuda"


# --------------------------------------------------------------- the cases ---
def listed():
    base = dict(jitter=0.1, drop=0, shuffle=False, matter=False, absorb=False, alpha=1.0)

    def c(name, kind, n, N, steps, **kw):
        return dict(base, name=name, kind=kind, n=n, N=N, steps=steps, **kw)

    return [
        # the smallest solve anyone runs: the 384-tet order-3 verification run, its
        # energy read at the end (latency and launches are all of its time)
        c("golden_N3", "monitor", 4, 3, 10),
        # the benchmark workload: order 4, 82 944 tets, steps between two energy readings
        c("pulse_N4", "monitor", 24, 4, 4, jitter=0.15),
        # the split-precision workload: order 6, 24 576 tets
        c("cavity_N6", "step", 16, 6, 4),
        # the served stream's highest order, most of that stream's work
        c("pulse_N7", "step", 16, 7, 4, jitter=0.15),
        # order sweep, lowest orders: many elements with few nodes
        c("sweep_N1", "step", 49, 1, 4),
        c("sweep_N2", "step", 36, 2, 4),
        # a scattering set-up: dielectric regions and absorbing outer faces
        c("matter_N5", "step", 20, 5, 4, matter=True, absorb=True),
        # order sweep, highest orders
        c("sweep_N8", "step", 14, 8, 2),
        c("sweep_N9", "monitor", 13, 9, 2),
        # an external integrator's call on an unstructured generator's mesh: element
        # count of no particular divisibility, arbitrary numbering
        c("ragged_N4", "rhs", 17, 4, 1, drop=13, shuffle=True),
        # fields that live on the host between calls (e.g. an I/O or coupling loop)
        c("host_N3", "host", 29, 3, 1),
        # the batched solver: packs of small solves of several orders, one step of all
        dict(base, name="batch", kind="batch", seed_n=5, orders="23456", nmin=4, nmax=9, per=3,
             steps=1),
    ]


# Largest hexahedra count per side of each order: the order sweep's ~1.7e7 unknowns.
_NMAX = {1: 49, 2: 36, 3: 29, 4: 24, 5: 20, 6: 18, 7: 16, 8: 14, 9: 13}


def draw(rng: random.Random):
    if rng.random() < 0.12:
        first = rng.randint(1, 5)
        orders = "".join(str(o) for o in range(first, first + rng.randint(1, 3)))
        nmin = rng.randint(3, 6)
        return dict(kind="batch", seed_n=rng.randint(0, 99), orders=orders, nmin=nmin,
                    nmax=nmin + rng.randint(0, 5), per=rng.randint(1, 4), steps=rng.randint(1, 2),
                    jitter=0.1, drop=0, shuffle=False, matter=False, absorb=False, alpha=1.0)
    N = rng.randint(1, 9)
    n = max(2, round(math.exp(rng.uniform(math.log(2.0), math.log(_NMAX[N])))))
    kind = rng.choice(["step", "step", "step", "monitor", "rhs", "host"])
    return dict(kind=kind, n=n, N=N, steps=rng.randint(1, 2), jitter=rng.choice([0.05, 0.1, 0.15]),
                drop=rng.choice([0, 0, 1, 2, 3, 5, 7]), shuffle=rng.random() < 0.3,
                matter=rng.random() < 0.2, absorb=rng.random() < 0.25,
                alpha=rng.choice([1.0, 1.0, 1.0, 0.0, 0.5]))


# ------------------------------------------------------------------- meshes ---
def _box(n, jitter, seed, drop=0, shuffle=False):
    """[-1,1]^3 as n^3 hexahedra of 6 tetrahedra, inner vertices jittered; `drop`
    tetrahedra left out (their faces become walls), optionally renumbered."""
    rng = np.random.default_rng(seed)
    h = 2.0 / n
    g = np.arange(n + 1) * h - 1.0
    z, y, x = np.meshgrid(g, g, g, indexing="ij")
    v = np.stack([x.ravel(), y.ravel(), z.ravel()], axis=1)
    d = rng.uniform(-jitter * h, jitter * h, size=v.shape)
    d[np.abs(np.abs(v) - 1.0) < 1e-12] = 0.0
    v = v + d
    st = np.array([1, n + 1, (n + 1) ** 2])
    i = np.arange(n)
    v0 = (i[None, None, :] * st[0] + i[None, :, None] * st[1] + i[:, None, None] * st[2]).ravel()
    tets = []
    for a, b, c in itertools.permutations(range(3)):
        p = [v0, v0 + st[a], v0 + st[a] + st[b], v0 + st.sum()]
        if (a, b, c) in ((0, 2, 1), (1, 0, 2), (2, 1, 0)):      # odd: orient positively
            p[2], p[3] = p[3], p[2]
        tets.append(np.stack(p, axis=1))
    t = np.stack(tets, axis=1).reshape(-1, 4).astype(np.int32)
    if drop:
        t = np.delete(t, rng.choice(len(t), size=min(drop, len(t) - 1), replace=False), axis=0)
    if shuffle:
        t = t[rng.permutation(len(t))]
    return v, np.ascontiguousarray(t)


# --------------------------------------------------------- reference element ---
_WB_ALPHA = (0.0, 0.0, 0.0, 0.1002, 1.1332, 1.5608, 1.3413, 1.2577, 1.1603)
_FACES = ((0, 1, 2), (0, 1, 3), (1, 2, 3), (0, 2, 3))
_OPP = (3, 2, 0, 1)


def _multi(N, d):
    return [a for a in itertools.product(range(N + 1), repeat=d) if sum(a) == N]


@functools.lru_cache(None)
def _nodes(N):
    """Barycentric coordinates [Np, 4] (vertices 0..3) of the Warp & Blend nodes, the
    first reference coordinate running fastest (Warburton 2006)."""
    eq = np.array([(N - i - j - k, i, j, k) for k in range(N + 1) for j in range(N + 1 - k)
                   for i in range(N + 1 - j - k)]) / N
    if N < 3:
        return eq
    dl = np.polynomial.legendre.Legendre.basis(N).deriv().roots().real
    disp = np.concatenate([[-1.0], np.sort(dl), [1.0]]) - np.linspace(-1, 1, N + 1)
    xe = np.linspace(-1, 1, N + 1)
    alpha = _WB_ALPHA[N - 1]

    def warp(x):
        # displacement interpolated through the equidistant points, over 1 - x^2
        out = np.zeros_like(x)
        for p in range(N + 1):
            li = np.full_like(x, disp[p])
            for q in range(N + 1):
                if q != p:
                    li *= (x - xe[q]) / (xe[p] - xe[q])
            out += li
        ok = np.abs(x) < 1 - 1e-10
        return np.where(ok, out / np.where(ok, 1 - x * x, 1.0), 0.0)

    # equilateral vertices of local vertices 0..3
    P = np.array([[-1, -1 / 3 ** 0.5, -1 / 6 ** 0.5], [1, -1 / 3 ** 0.5, -1 / 6 ** 0.5],
                  [0, 2 / 3 ** 0.5, -1 / 6 ** 0.5], [0, 0, 3 / 6 ** 0.5]])
    X, shift = eq @ P, np.zeros((len(eq), 3))
    for a, b, c, d in ((3, 2, 0, 1), (2, 3, 0, 1), (0, 3, 1, 2), (1, 3, 0, 2)):
        # face without vertex a; edge c -> d is its first tangent, b its apex
        La, Lb, Lc, Ld = eq[:, a], eq[:, b], eq[:, c], eq[:, d]
        t1 = (P[d] - P[c]) / np.linalg.norm(P[d] - P[c])
        t2 = P[b] - 0.5 * (P[c] + P[d])
        t2 /= np.linalg.norm(t2)
        w1 = 4 * Lc * Ld * warp(Ld - Lc) * (1 + (alpha * Lb) ** 2)
        w2 = 4 * Lb * Ld * warp(Lb - Ld) * (1 + (alpha * Lc) ** 2)
        w3 = 4 * Lb * Lc * warp(Lc - Lb) * (1 + (alpha * Ld) ** 2)
        wx, wy = w1 - 0.5 * (w2 + w3), 0.75 ** 0.5 * (w2 - w3)
        den = (Lb + La / 2) * (Lc + La / 2) * (Ld + La / 2)
        ok = den > 1e-10
        bl = np.where(ok, (1 + (alpha * La) ** 2) * Lb * Lc * Ld / np.where(ok, den, 1.0), 0.0)
        add = np.outer(bl * wx, t1) + np.outer(bl * wy, t2)
        inner = (Lb > 1e-10).astype(int) + (Lc > 1e-10) + (Ld > 1e-10)
        edge = (La < 1e-10) & (inner < 3)
        flat = np.outer(wx, t1) + np.outer(wy, t2)
        shift += np.where(edge[:, None], 0.0, add)
        shift = np.where(edge[:, None], flat, shift)
    A = np.vstack([P.T, np.ones(4)])
    return np.linalg.solve(A, np.vstack([(X + shift).T, np.ones(len(X))])).T


def _bernstein(N, lam):
    """Bernstein polynomials of degree N at barycentric points and their multi-indices."""
    idx = _multi(N, lam.shape[1]) if N >= 0 else []
    cols = []
    for a in idx:
        f = math.factorial(N)
        v = np.ones(len(lam))
        for x, e in zip(lam.T, a):
            f //= math.factorial(e)
            v = v * x ** e
        cols.append(f * v)
    return np.stack(cols, axis=1), idx


def _bernstein_mass(N, d, vol):
    """Integral of products of Bernstein polynomials over a simplex with d + 1 vertices."""
    idx = _multi(N, d + 1)
    return vol / (math.comb(2 * N, N) * math.comb(2 * N + d, d)) * np.array(
        [[math.prod(math.comb(i + j, i) for i, j in zip(a, b)) for b in idx] for a in idx], float)


@functools.lru_cache(None)
def _ref(N):
    lam = _nodes(N)
    V, idx = _bernstein(N, lam)
    Vi = np.linalg.inv(V)
    low, lidx = _bernstein(N - 1, lam)
    pos = {a: q for q, a in enumerate(lidx)}
    Dl = []
    for v in range(4):                       # d/d lambda_v of a Bernstein polynomial
        G = np.zeros_like(V)
        for q, a in enumerate(idx):
            if a[v]:
                G[:, q] = N * low[:, pos[tuple(e - (w == v) for w, e in enumerate(a))]]
        Dl.append(G @ Vi)
    M = Vi.T @ _bernstein_mass(N, 3, 4 / 3) @ Vi
    fmask, E = [], np.zeros((len(lam), 0))
    for f, fv in enumerate(_FACES):
        on = np.nonzero(np.abs(lam[:, _OPP[f]]) < 1e-10)[0]
        Wi = np.linalg.inv(_bernstein(N, lam[on][:, fv])[0])
        Ef = np.zeros((len(lam), len(on)))
        Ef[on] = Wi.T @ _bernstein_mass(N, 2, 2.0) @ Wi
        fmask.append(on)
        E = np.hstack([E, Ef])
    # order[f][s]: face nodes of f sorted by their barycentric coordinates after
    # permuting the face's vertices by s, the same point order on both sides
    perms = list(itertools.permutations(range(3)))
    order = np.zeros((4, 6, len(fmask[0])), int)
    for f, fv in enumerate(_FACES):
        L = np.round(lam[fmask[f]][:, fv], 8)
        for s, p in enumerate(perms):
            order[f, s] = np.lexsort((L[:, p[1]], L[:, p[0]]))
    T = lambda a: torch.tensor(np.asarray(a), device=DEV)  # noqa: E731
    return dict(lam=lam, D=[T((Dl[v] - Dl[0]) / 2) for v in (1, 2, 3)], M=T(M),
                LIFT=T(np.linalg.solve(M, E)), fmask=T(np.stack(fmask)), order=order, perms=perms)


def _geometry(v, t):
    X = torch.tensor(v, device=DEV)[torch.tensor(t, dtype=torch.long, device=DEV)]
    Ed = X[:, 1:] - X[:, :1]                                   # [K, 3 edges, 3]
    G = torch.linalg.inv(Ed).transpose(1, 2)                   # gradients of lambda_1..3
    grad = torch.cat([-G.sum(1, keepdim=True), G], dim=1)      # [K, 4, 3]
    J = torch.linalg.det(Ed) / 8
    gf = grad[:, list(_OPP)]                                   # gradient opposite each face
    ln = gf.norm(dim=2)
    return J, 2 * grad[:, 1:], -gf / ln[..., None], 2 * ln     # J, dr/dx, normals, sJ / J


def _connect(t, N):
    """Global node numbers (inner, outer) of every face node [K, 4, Nfp] in matching
    order and the boundary mask [K, 4], plus the neighbour of every face."""
    R = _ref(N)
    K, Np = len(t), len(R["lam"])
    fv = t[:, np.array(_FACES)].astype(np.int64)               # [K, 4, 3] global vertices
    rank = np.argsort(fv, axis=2)
    key = np.take_along_axis(fv, rank, 2)
    nv = int(t.max()) + 1
    code = ((key[..., 0] * nv + key[..., 1]) * nv + key[..., 2]).ravel()
    srt = np.argsort(code, kind="stable")
    same = np.nonzero(code[srt][1:] == code[srt][:-1])[0]
    mate = np.arange(4 * K)
    mate[srt[same]], mate[srt[same + 1]] = srt[same + 1], srt[same]
    ptab = np.zeros((3, 3, 3), int)
    for s, p in enumerate(R["perms"]):
        ptab[p] = s
    sig = ptab[rank[..., 0], rank[..., 1], rank[..., 2]].ravel()
    face = np.tile(np.arange(4), K)
    loc = np.take_along_axis(R["fmask"].cpu().numpy()[face], R["order"][face, sig], 1)
    glob = torch.tensor(loc + (np.arange(4 * K) // 4 * Np)[:, None], device=DEV)
    m = torch.tensor(mate, device=DEV)
    pos = torch.tensor(R["order"][face, sig], device=DEV)      # position within the face
    return glob, glob[m], pos, (m == torch.arange(4 * K, device=DEV)).reshape(K, 4), \
        (m // 4).reshape(K, 4)


# --------------------------------------------------------------- exact answer ---
_A = (0.0, -567301805773 / 1357537059087, -2404267990393 / 2016746695238,
      -3550918686646 / 2091501179385, -1275806237668 / 842570457699)
_B = (1432997174477 / 9575080441755, 5161836677717 / 13612068292357,
      1720146321549 / 2090206949498, 3134564353537 / 4481467310338,
      2277821191437 / 14882151754819)


def _cross(a, b):
    return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]


class _Exact:
    """The semi-discrete operator in 64 bits."""

    def __init__(self, v, t, N, alpha=1.0, eps=None, mu=None, bc=None):
        self.R, self.N, self.alpha, self.K = _ref(N), N, alpha, len(t)
        self.J, self.drdx, self.nrm, self.Fs = _geometry(v, t)
        self.iM, self.iP, self.pos, self.bnd, nb = _connect(t, N)
        one = torch.ones(self.K, dtype=torch.float64, device=DEV)
        T = lambda a: one if a is None else torch.tensor(a, dtype=torch.float64, device=DEV)  # noqa: E731
        self.eps, self.mu = T(eps), T(mu)
        Z = (self.mu / self.eps).sqrt()
        self.Zm = Z[:, None].expand(-1, 4)
        self.Zp = torch.where(self.bnd, self.Zm, Z[nb])
        self.absorb = self.bnd & (torch.zeros_like(self.bnd) if bc is None
                                  else torch.tensor(bc, device=DEV) == 1)

    def rhs(self, u):
        K, R = self.K, self.R
        dr = [u @ D.T for D in R["D"]]                          # [6, K, Np] each
        dx = [sum(self.drdx[:, m, a, None] * dr[m] for m in range(3)) for a in range(3)]
        dE, dH = [d[:3] for d in dx], [d[3:] for d in dx]       # [axis][component]
        curl = lambda d: [d[1][2] - d[2][1], d[2][0] - d[0][2], d[0][1] - d[1][0]]  # noqa: E731
        vol = torch.stack(curl(dH) + [-x for x in curl(dE)])
        del dr, dx, dE, dH
        flat = u.reshape(6, -1)
        um = flat[:, self.iM].reshape(6, K, 4, -1)
        up = flat[:, self.iP].reshape(6, K, 4, -1)
        wall, ab = (self.bnd & ~self.absorb)[..., None], self.absorb[..., None]
        sign = torch.tensor([-1.0] * 3 + [1.0] * 3, dtype=u.dtype, device=DEV)[:, None, None, None]
        up = torch.where(wall, sign * um, torch.where(ab, torch.zeros_like(up), up))
        j = up - um
        n = [self.nrm[..., a, None] for a in range(3)]
        cE, cH = _cross(n, j[:3]), _cross(n, j[3:])
        ccE, ccH = _cross(n, cE), _cross(n, cH)
        Zm, Zp = self.Zm[..., None], self.Zp[..., None]
        fE = [(Zp * a - self.alpha * b) / (Zm + Zp) for a, b in zip(cH, ccE)]
        fH = [(-a / Zp - self.alpha * b) / (1 / Zm + 1 / Zp) for a, b in zip(cE, ccH)]
        fl = torch.stack(fE + fH) * self.Fs[None, ..., None]
        # back from matching order to the face's own node order
        out = torch.empty_like(fl).reshape(6, 4 * K, -1)
        out.scatter_(2, self.pos[None].expand(6, -1, -1), fl.reshape(6, 4 * K, -1))
        r = vol + out.reshape(6, K, -1) @ R["LIFT"].T
        w = torch.stack([1 / self.eps] * 3 + [1 / self.mu] * 3)
        return r * w[..., None]

    def steps(self, u, res, dt, n):
        for _ in range(n):
            for a, b in zip(_A, _B):
                res = a * res + dt * self.rhs(u)
                u = u + b * res
        return u, res

    def energy(self, u):
        w = torch.stack([self.eps] * 3 + [self.mu] * 3) * self.J
        return 0.5 * float((w * ((u @ self.R["M"]) * u).sum(2)).sum())


# -------------------------------------------------------------------- inputs ---
def _fields(v, t, N, seed):
    """Single-precision fields a solver meets: a few cavity-scale waves, pulses on
    two components, and a little noise."""
    rng = np.random.default_rng([seed, 7])
    lam = torch.tensor(_nodes(N), device=DEV)
    X = torch.tensor(v, device=DEV)[torch.tensor(t, dtype=torch.long, device=DEV)]
    x = torch.einsum("iv,kvd->dki", lam, X)
    u = torch.empty((6,) + tuple(x.shape[1:]), dtype=torch.float32, device=DEV)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    for c in range(6):
        k, ph = rng.integers(1, 3, 3) * math.pi / 2, rng.uniform(0, 2 * math.pi, 3)
        w = rng.normal() * torch.sin(k[0] * x[0] + ph[0]) * torch.sin(k[1] * x[1] + ph[1]) \
            * torch.sin(k[2] * x[2] + ph[2])
        if c in (2, 4):
            ctr = rng.uniform(-0.5, 0.5, 3)
            w = w + torch.exp(-sum((x[a] - ctr[a]) ** 2 for a in range(3)) / 0.2 ** 2)
        u[c] = w + 1e-3 * torch.randn(w.shape, generator=gen, device=DEV, dtype=torch.float64)
    return u


def _media(case, v, t, seed):
    """Permittivity and permeability of a dielectric ball and a slab, and the kind of
    every boundary face (absorbing outside)."""
    eps = mu = bc = None
    if case["matter"]:
        ctr = v[t].mean(1)
        r = np.random.default_rng([seed, 3]).uniform(0.4, 0.7)
        eps = np.where((ctr ** 2).sum(1) < r * r, 2.25, 1.0)
        mu = np.where(ctr[:, 2] > 0.5, 1.5, 1.0)
    if case["absorb"]:
        bc = np.ones((len(t), 4), np.int8)
    return eps, mu, bc


def _time_step(v, t, N, eps, mu):
    _, _, _, Fs = _geometry(v, t)
    slow = 1.0 if eps is None else torch.tensor(np.sqrt(eps * mu), device=DEV)[:, None]
    return float(np.float32(0.9 * float((slow / Fs).min()) * 2.0 / (N + 1) ** 2))


def _problem(case, seed):
    v, t = _box(case["n"], case["jitter"], seed, case["drop"], case["shuffle"])
    eps, mu, bc = _media(case, v, t, seed)
    u = _fields(v, t, case["N"], seed)
    return v, t, eps, mu, bc, u, _time_step(v, t, case["N"], eps, mu)


def _batch(case, seed):
    """Per order: the solves (mesh, fields, step) of one pack."""
    rng = random.Random(case["seed_n"])
    out = []
    for q, o in enumerate(case["orders"]):
        N = int(o)
        solves = []
        for s in range(case["per"]):
            v, t = _box(rng.randint(case["nmin"], case["nmax"]), case["jitter"],
                        [seed, q, s])
            solves.append((v, t, _fields(v, t, N, seed * 1000 + 10 * q + s),
                           _time_step(v, t, N, None, None)))
        out.append((N, solves))
    return out


# ---------------------------------------------------------------- the passes ---
def prepare(case, seed):
    if case["kind"] == "batch":
        packs = []
        for N, solves in _batch(case, seed):
            parts = [dg.Mesh(v, t, N) for v, t, _, _ in solves]
            u = torch.cat([f for _, _, f, _ in solves], dim=1).contiguous()
            dt = torch.cat([torch.full((f.shape[1],), d, dtype=torch.float32, device=DEV)
                            for _, _, f, d in solves])
            packs.append(dict(mesh=dg.Mesh.pack(parts), u=u, w=torch.empty_like(u),
                              res=torch.zeros_like(u), dt=dt))
        return dict(case=case, packs=packs)
    v, t, eps, mu, bc, u, dt = _problem(case, seed)
    mesh = dg.Mesh(v, t, case["N"])
    mesh.set_flux(case["alpha"])
    if eps is not None:
        mesh.set_materials(eps, mu)
    if bc is not None:
        mesh.set_boundary(bc)
    st = dict(case=case, mesh=mesh, dt=dt)
    if case["kind"] == "host":
        st["u"] = u.cpu().pin_memory()
    elif case["kind"] == "rhs":
        st["u"], st["out"] = u, torch.empty_like(u)
    else:
        st["u"], st["res"] = u, torch.zeros_like(u)
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        # one solve loop iteration: every pack through the stages, its two state
        # buffers taking turns
        for _ in range(case["steps"]):
            for stage in range(5):
                for p in state["packs"]:
                    p["mesh"].rk_stage_elem(p["u"], p["w"], p["res"], stage, p["dt"])
                    p["u"], p["w"] = p["w"], p["u"]
        return [x for p in state["packs"] for x in (p["u"], p["res"])]
    mesh, u = state["mesh"], state["u"]
    if kind == "rhs":
        return mesh.rhs(u, state["out"])
    if kind == "host":
        e = mesh.step_host(u, None, state["dt"], case["steps"])
        return u, e
    mesh.step(u, state["res"], state["dt"], case["steps"])
    if kind == "monitor":
        return u, state["res"], mesh.energy(u)
    return u, state["res"]


def exact(case, seed):
    if case["kind"] == "batch":
        out = []
        for N, solves in _batch(case, seed):
            us, rs = [], []
            for v, t, u, dt in solves:
                X = _Exact(v, t, N)
                a, b = X.steps(u.double(), torch.zeros_like(u, dtype=torch.float64), dt,
                               case["steps"])
                us.append(a)
                rs.append(b)
            out += [torch.cat(us, dim=1), torch.cat(rs, dim=1)]
        return out
    v, t, eps, mu, bc, u, dt = _problem(case, seed)
    X = _Exact(v, t, case["N"], case["alpha"], eps, mu, bc)
    u = u.double()
    if case["kind"] == "rhs":
        return X.rhs(u)
    u, res = X.steps(u, torch.zeros_like(u), dt, case["steps"])
    if case["kind"] == "host":
        return u.cpu(), X.energy(u)
    if case["kind"] == "monitor":
        return u, res, X.energy(u)
    return u, res


def _element_work(N):
    """(bytes, operations) per element and stage: u and the RK register read and
    written and the element's geometry read; derivative, flux and lifting as the
    library counts them (additions and multiplications)."""
    Np, Nfp = (N + 1) * (N + 2) * (N + 3) // 6, (N + 1) * (N + 2) // 2
    NF = 4 * Nfp
    return 96 * Np + 132, 36 * Np * Np + 66 * Np + 60 * NF + 12 * Np * NF + 36 * Np


def work(case):
    """One pass: every stage reads and writes whole fields (a stage needs its
    neighbours' values of the stage before)."""
    if case["kind"] == "batch":
        rng = random.Random(case["seed_n"])
        b = f = 0
        for o in case["orders"]:
            eb, ef = _element_work(int(o))
            K = sum(6 * rng.randint(case["nmin"], case["nmax"]) ** 3 for _ in range(case["per"]))
            b, f = b + 5 * case["steps"] * K * eb, f + 5 * case["steps"] * K * ef
        return dict(bytes=b, flops=f)
    N = case["N"]
    K = max(1, 6 * case["n"] ** 3 - case["drop"])
    Np = (N + 1) * (N + 2) * (N + 3) // 6
    eb, ef = _element_work(N)
    if case["kind"] == "rhs":
        return dict(bytes=K * (eb - 48 * Np), flops=K * (ef - 30 * Np))
    b, f = 5 * case["steps"] * K * eb, 5 * case["steps"] * K * ef
    if case["kind"] in ("monitor", "host"):       # the energy reads the fields once more
        b, f = b + 24 * K * Np, f + 12 * K * Np * Np
    return dict(bytes=b, flops=f)
