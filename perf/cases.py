"""What a user of this framework has it do, as cases that can be timed and checked.

A case is a dict of plain values.  ``listed()`` holds the standing ones, ``draw(rng)`` makes
another of the same ranges, ``prepare(case, seed)`` builds what a user's program holds
before the call (the context of its mesh, and inputs from the seed), ``run(state)`` is one
pass through the public entry points, ``work(case)`` counts what the path cannot do without
and ``exact(case, seed)`` gives the results in 64 bits from plain torch.

Kinds (field "kind"):
  apply    Hopu.apply_convection(w, u): the operator on a simplicial mesh, the wind in V_h;
           "orders" gives every facet its own HOPU order, "walls" a box that is not periodic
  substep  Hopu.rk_substep: SSP-RK3 substeps of a restarted state (wind "stage" or "frozen"),
           on a side stream ("side") or on the default stream
  batch    HopuBatch.rk_substep: many meshes of uneven size and order in one call
  grad     ConvectionApply forward and backward: y and the cotangents of w and u
  rollout  Rollout forward and backward: u_n and the cotangent of u_0
  hex      HopuHex.apply, with the wind equal to the field ("same") or separate
  hexsub   HopuHex.rk_substeps on a structured hexahedral box

Inputs: Taylor-Green fields of unit size with a phase of the seed, interpolated into V_h or
projected into L2, plus U[-1e-3, 1e-3] on every coefficient (the recipe of the benchmark and
the tests); the meshes are Kuhn-split boxes under a smooth periodic deformation, so that no
two elements are alike.  Hexahedral boxes have uneven grid lines and a shear.
"""
import itertools
import math
from functools import lru_cache

import numpy as np
import torch

TWO_PI = 2.0 * math.pi


def listed():
    return [
        # the smallest use: the 8 x 8 square of the 2D configuration, ten substeps as a
        # program makes them on the default stream; latency and launches count
        dict(name="square_k2_f64", kind="substep", dim=2, n=8, k=2, prec="f64", wind="stage", steps=10, side=False),
        # a small 3D mesh, one apply: what a coarse level or a test problem asks for
        dict(name="apply_k2_n7_f32", kind="apply", dim=3, n=7, k=2, prec="f32", orders=False, walls=False),
        # the 16^3 k = 3 configuration, with the adaptive method's per-facet orders
        dict(name="apply_k3_n16_f32", kind="apply", dim=3, n=16, k=3, prec="f32", orders=True, walls=False),
        # the operator at the headline's size: the wind and the field are different vectors,
        # as in an implicit-explicit splitting or a linearised solve
        dict(name="apply_k4_n32_f32", kind="apply", dim=3, n=32, k=4, prec="f32", orders=False, walls=False),
        # the highest order at an odd size, tensor-core mode
        dict(name="apply_k5_n13_f32tc", kind="apply", dim=3, n=13, k=5, prec="f32_tc", orders=False, walls=False),
        # double precision: the reference runs of a convergence study
        dict(name="apply_k3_n16_f64", kind="apply", dim=3, n=16, k=3, prec="f64", orders=False, walls=False),
        # the headline: one substep of the 32^3 k = 4 box, replayed from its graph
        dict(name="substep_k4_n32_f32tc", kind="substep", dim=3, n=32, k=4, prec="f32_tc", wind="stage", steps=1,
             side=True),
        # a batch of independent meshes of every size and order, one substep of all
        dict(name="batch_24_f32tc", kind="batch", meshes=24, mix=1, prec="f32_tc"),
        # differentiating through the operator (a training or sensitivity step)
        dict(name="grad_k3_n16_f32", kind="grad", dim=3, n=16, k=3, prec="f32"),
        # differentiating through time
        dict(name="rollout_k3_n12_f32tc", kind="rollout", dim=3, n=12, k=3, prec="f32_tc", steps=4, ckpt=2),
        # the paper's cell shape at the benchmark's size: one substep
        dict(name="hexsub_k4_32_f32", kind="hexsub", nx=32, ny=32, nz=32, k=4, prec="f32", steps=1),
        # a ragged hexahedral box in double precision, separate wind
        dict(name="hex_k3_odd_f64", kind="hex", nx=13, ny=9, nz=17, k=3, prec="f64", same=False),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _cost(c):
    """Time model (in FP32 operations) that keeps a drawn case below the largest listed one."""
    return work(c)["flops"] * (40.0 if c["prec"] == "f64" else 1.0)


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["apply", "apply", "apply", "substep", "substep", "batch", "grad", "rollout", "hex", "hexsub"])
        prec = rng.choice(["f32", "f32", "f32_tc", "f32_tc", "f64"])
        if kind in ("hex", "hexsub"):
            c = dict(kind=kind, nx=_log_int(rng, 3, 40), ny=_log_int(rng, 3, 40), nz=_log_int(rng, 3, 40),
                     k=rng.randint(2, 5), prec=rng.choice(["f32", "f32", "f64"]))
            if kind == "hex":
                c["same"] = rng.random() < 0.5
            else:
                c["steps"] = rng.choice([1, 2])
        elif kind == "batch":
            c = dict(kind=kind, meshes=_log_int(rng, 4, 32), mix=rng.randint(2, 10 ** 6), prec=rng.choice(["f32", "f32_tc"]))
        else:
            dim = 3 if rng.random() < 0.85 else 2
            n = _log_int(rng, 3, 32) if dim == 3 else _log_int(rng, 4, 160)
            c = dict(kind=kind, dim=dim, n=n, k=rng.randint(2, 5 if dim == 3 else 4), prec=prec)
            if kind == "apply":
                c.update(orders=rng.random() < 0.3, walls=rng.random() < 0.2)
            elif kind == "substep":
                c.update(wind=rng.choice(["stage", "stage", "stage", "frozen"]), steps=rng.choice([1, 2, 4]),
                         side=rng.random() < 0.5)
            elif kind == "rollout":
                steps = rng.choice([2, 3, 4])
                c.update(steps=steps, ckpt=rng.randint(1, steps))
        if _cost(c) <= most:
            return c


# ---------------------------------------------------------------------------- sizes
def _nb(d, k):
    return math.comb(k + d, d) if k >= 0 else 0


def _batch_meshes(c):
    """(n, k) of every mesh: the heterogeneous batch's draw, n in 4..12 and k in 2..5."""
    rng = np.random.Generator(np.random.PCG64(c["mix"]))
    n = rng.integers(4, 13, size=c["meshes"])
    k = rng.integers(2, 6, size=c["meshes"])
    return [(int(a), int(b)) for a, b in zip(n, k)]


_RULE = {(3, 3): 46, (3, 4): 100, (3, 5): 190}  # points of a compact rule exact to degree 3k - 1


def _simplex_flops(d, k, E, F):
    """(E v, one operator evaluation, R E^-1 y): the contractions of each."""
    nb, nf, nb1 = _nb(d, k), _nb(d - 1, k), _nb(d, k - 1)
    nq = _RULE.get((d, k)) or ((3 * k + 1) // 2) ** d
    nqf = ((3 * k + 2) // 2) ** (d - 1)
    vol = E * (2 * d * d * nb1 * nb + nq * (4 * nb * d + 2 * nb1 * d * d) + 2 * d * nb * (d + 1) * nf)
    fac = F * (4 * nf * nb * d + nqf * nf * (6 * d + 4 * d))
    proj = 2 * E * (d * nb) ** 2
    return proj, vol + fac, proj


def work(c):
    """Bytes: every input vector read and every output vector written once (the mesh and its
    tables belong to the context); flops: the contractions of the operator and the maps."""
    s = 8 if c["prec"] == "f64" else 4
    if c["kind"] in ("hex", "hexsub"):
        m, p = (3 * c["k"] + 2) // 2, c["k"] + 1
        E = c["nx"] * c["ny"] * c["nz"]
        fields = 3 if c["kind"] == "hexsub" or c["same"] else 6
        line = p * p * p * m + p * p * m * m + p * m * m * m          # one field to the points of a cell
        flops = E * (2 * line * (fields + 3 + 3) + 3 * (2 * 2 * 3 * p ** 3 + 2 * 3 * 3 * (p * p * m + p * m * m) * 2))
        n = E * 3 * p ** 3
        if c["kind"] == "hex":
            return {"bytes": s * n * (2 if c["same"] else 3), "flops": flops}
        return {"bytes": s * n * 2 * c["steps"], "flops": 3 * c["steps"] * flops}
    if c["kind"] == "batch":
        total = {"bytes": 0, "flops": 0}
        for n, k in _batch_meshes(c):
            w = work(dict(kind="substep", dim=3, n=n, k=k, prec=c["prec"], wind="stage", steps=1))
            total = {x: total[x] + w[x] for x in total}
        return total
    d, k, n = c["dim"], c["k"], c["n"]
    E = math.factorial(d) * n ** d
    F = E * (d + 1) // 2
    n_l2 = E * d * _nb(d, k)
    n_v = F * _nb(d - 1, k) + n_l2 - E * (d + 1) * _nb(d - 1, k)
    e, a, r = _simplex_flops(d, k, E, F)
    if c["kind"] == "apply":
        return {"bytes": s * (n_v + 2 * n_l2), "flops": e + a}
    if c["kind"] == "substep":
        if c["wind"] == "frozen":
            return {"bytes": s * c["steps"] * 2 * n_l2, "flops": 3 * c["steps"] * a + e}
        return {"bytes": s * c["steps"] * 2 * n_v, "flops": 3 * c["steps"] * (e + a + r)}
    if c["kind"] == "grad":
        return {"bytes": s * (2 * n_v + 4 * n_l2), "flops": 2 * e + 3 * a + r}
    forward = 3 * c["steps"] * (e + a + r)
    return {"bytes": s * 4 * n_v, "flops": forward + 3 * c["steps"] * (2 * e + 2 * a + r)}


# ---------------------------------------------------------------------------- meshes
@lru_cache(maxsize=64)
def _box(dim, n, walls=False):
    """(coords, elems, rep) of the Kuhn split of an n^dim grid on [0, 2 pi]^dim, vertices moved
    by a smooth periodic map; rep is None for a box with walls."""
    m = n + 1
    grid = np.indices((m,) * dim).reshape(dim, -1).T                        # last axis fastest
    x = grid * (TWO_PI / n)
    coords = x + 0.15 * np.sin(np.roll(x, 1, axis=1) + 0.3)
    weight = m ** np.arange(dim - 1, -1, -1)
    rep = None if walls else ((grid % n) @ (n ** np.arange(dim - 1, -1, -1))).astype(np.int64)
    cell = np.indices((n,) * dim).reshape(dim, -1).T
    elems = []
    for order in itertools.permutations(range(dim)):
        v = [cell]
        for axis in order:
            v.append(v[-1] + np.eye(dim, dtype=np.int64)[axis])
        elems.append(np.stack([c @ weight for c in v], axis=1))
    return coords, np.stack(elems, axis=1).reshape(-1, dim + 1).astype(np.int64), rep


@lru_cache(maxsize=8)
def _class_mesh(c_meshes, k):
    """The meshes of one order of a batch as one mesh: vertices and representatives offset."""
    co, el, re, at = [], [], [], 0
    for n, kk in c_meshes:
        if kk != k:
            continue
        x, e, r = _box(3, n)
        co.append(x)
        el.append(e + at)
        re.append(r + at)
        at += len(x)
    return np.concatenate(co), np.concatenate(el), np.concatenate(re)


def _hex_box(c):
    """Grid lines with uneven spacings and a shear, of the case alone."""
    rng = np.random.Generator(np.random.PCG64(7))
    lines = []
    for n in (c["nx"], c["ny"], c["nz"]):
        h = TWO_PI / n * (1.0 + rng.uniform(-0.2, 0.2, size=n))
        lines.append(np.concatenate([[0.0], np.cumsum(h)]))
    A = np.eye(3) + 0.2 * np.triu(rng.uniform(-1.0, 1.0, size=(3, 3)), 1)
    return lines, A


# ---------------------------------------------------------------------------- reference element, 64 bits
def _gauss_jacobi(m, alpha):
    """m nodes and weights on (0, 1) for the weight (1 - t)^alpha (Golub and Welsch)."""
    j = np.arange(m, dtype=np.float64)
    diag = np.where(2 * j + alpha > 0, -alpha ** 2 / np.maximum((2 * j + alpha) * (2 * j + alpha + 2), 1e-300), 0.0)
    if alpha == 0:
        diag[:] = 0.0
    j = np.arange(1, m, dtype=np.float64)
    s = 2 * j + alpha
    off = np.sqrt(4 * j * j * (j + alpha) ** 2 / (s * s * (s + 1) * (s - 1)))
    x, v = np.linalg.eigh(np.diag(diag) + np.diag(off, 1) + np.diag(off, -1))
    return (1 + x) / 2, v[0] ** 2 / (alpha + 1)


def _simplex_rule(d, m):
    t = [_gauss_jacobi(m, a) for a in range(d)]
    if d == 1:
        return t[0][0][:, None], t[0][1]
    g = np.meshgrid(*[p for p, _ in t], indexing="ij")
    w = np.einsum("i,j->ij", t[0][1], t[1][1]) if d == 2 else np.einsum("i,j,k->ijk", t[0][1], t[1][1], t[2][1])
    if d == 2:
        pts = [g[0] * (1 - g[1]), g[1]]
    else:
        pts = [g[0] * (1 - g[1]) * (1 - g[2]), g[1] * (1 - g[2]), g[2]]
    return np.stack([p.reshape(-1) for p in pts], axis=1), w.reshape(-1)


def _jacobi(n, a, x, t):
    """t^i P_i^(a,0)(x / t), i = 0..n, by the three-term recurrence (no division by t)."""
    out = [np.ones_like(x)]
    if n > 0:
        out.append((a * t + (a + 2) * x) / 2)
    for i in range(1, n):
        c1 = 2 * (i + 1) * (i + a + 1) * (2 * i + a)
        c2 = (2 * i + a + 1) * a * a
        c3 = (2 * i + a) * (2 * i + a + 1) * (2 * i + a + 2)
        c4 = 2 * (i + a) * i * (2 * i + a + 2)
        out.append(((c2 * t + c3 * x) * out[i] - c4 * t * t * out[i - 1]) / c1)
    return out


def _dubiner(d, k, x):
    """Orthonormal Dubiner basis of P^k of the unit simplex at x [N, d]: [N, nb]."""
    one = np.ones_like(x[:, 0])
    cols = []
    if d == 1:
        P = _jacobi(k, 0, 2 * x[:, 0] - 1, one)
        return np.stack([math.sqrt(2 * m + 1) * P[m] for m in range(k + 1)], axis=1)
    s = one - x[:, 1] - (x[:, 2] if d == 3 else 0)
    F1 = _jacobi(k, 0, 2 * x[:, 0] - s, s)
    if d == 2:
        F2 = [_jacobi(k, 2 * p + 1, 2 * x[:, 1] - 1, one) for p in range(k + 1)]
        for n in range(k + 1):
            for p in range(n + 1):
                cols.append(math.sqrt((2 * p + 1) * (2 * n + 2)) * F1[p] * F2[p][n - p])
        return np.stack(cols, axis=1)
    t = one - x[:, 2]
    F2 = [_jacobi(k, 2 * p + 1, 2 * x[:, 1] - t, t) for p in range(k + 1)]
    F3 = [_jacobi(k, 2 * i + 2, 2 * x[:, 2] - 1, one) for i in range(k + 1)]
    for n in range(k + 1):
        for p in range(n + 1):
            for q in range(n - p + 1):
                c = math.sqrt((2 * p + 1) * (2 * p + 2 * q + 2) * (2 * n + 3))
                cols.append(c * F1[p] * F2[p][q] * F3[p + q][n - p - q])
    return np.stack(cols, axis=1)


def _gradients(d, k, x):
    """Derivatives of the basis, [N, nb, d]: complex steps, exact to rounding for polynomials."""
    out = []
    for c in range(d):
        z = x.astype(np.complex128)
        z[:, c] += 1e-40j
        out.append(_dubiner(d, k, z).imag / 1e-40)
    return np.stack(out, axis=2)


def _moment_space(d, k, x):
    """Interior moment functions of the V_h element at x: [nint, N, d]."""
    phi, lo, out = _dubiner(d, k - 2, x), _nb(d, k - 3), []
    for m in range(d):
        for j in range(phi.shape[1]):
            out.append(np.eye(d)[m] * phi[:, j:j + 1])
    y = (d + 1) * x - 1.0
    if d == 2:
        out += [np.stack([-y[:, 1], y[:, 0]], axis=1) * phi[:, j:j + 1] for j in range(lo, phi.shape[1])]
        return np.stack(out)
    chi, lo2 = _dubiner(2, k - 2, x[:, :2]), _nb(2, k - 3)
    for m in range(3):
        q = phi[:, lo:] if m < 2 else chi[:, lo2:]
        out += [np.cross(y, np.eye(3)[m]) * q[:, j:j + 1] for j in range(q.shape[1])]
    return np.stack(out)


@lru_cache(maxsize=16)
def _tables(d, k, device):
    """Tables of one order (64 bits): rules, basis values, the matrix of the V_h functionals."""
    T = {}
    xq, wq = _simplex_rule(d, (3 * k + 2) // 2 + 1)
    sq, wf = _simplex_rule(d - 1, (3 * k + 2) // 2)
    corner = np.vstack([np.zeros(d), np.eye(d)])
    side = []
    for f in range(d + 1):
        P = np.delete(corner, f, axis=0)
        side.append(_dubiner(d, k, P[0] + sq @ (P[1:] - P[0])))
    phi, psi, z = _dubiner(d, k, xq), _dubiner(d - 1, k, sq), _moment_space(d, k, xq)
    nb, nf = phi.shape[1], psi.shape[1]
    normal = np.vstack([np.ones(d), -np.eye(d)])
    D = np.zeros((d * nb, d * nb))
    for b in range(d):
        cols = slice(b * nb, (b + 1) * nb)
        for f in range(d + 1):
            D[f * nf:(f + 1) * nf, cols] = normal[f, b] * np.einsum("q,qm,qi->mi", wf, psi, side[f])
        D[(d + 1) * nf:, cols] = np.einsum("q,jq,qi->ji", wq, z[:, :, b], phi)
    degree = np.concatenate([[n] * (n + 1) for n in range(k + 1)]) if d == 3 else np.arange(k + 1)
    for name, v in dict(xq=xq, wq=wq, sq=sq, wf=wf, side=np.stack(side), phi=phi, dphi=_gradients(d, k, xq), psi=psi, z=z,
                        D=D, Dinv=np.linalg.inv(D), normal=normal, degree=degree).items():
        T[name] = torch.as_tensor(np.ascontiguousarray(v), device=device)
    T.update(d=d, k=k, nb=nb, nf=nf, nint=d * nb - (d + 1) * nf)
    return T


class _Mesh:
    """Geometry, facets and the operators of a simplicial mesh in plain torch, 64 bits."""

    CHUNK = 1 << 14

    def __init__(self, box, k, device):
        coords, elems, rep = box
        self.T = T = _tables(coords.shape[1], k, device)
        d = T["d"]
        rep = np.arange(len(coords)) if rep is None else rep
        x, el, rp = (torch.as_tensor(a, device=device) for a in (coords, elems, rep))
        key = rp[el]
        el = torch.gather(el, 1, torch.argsort(key, dim=1))
        key = rp[el]
        X = x[el]                                                            # [E, d+1, d]
        self.X0, self.E = X[:, 0], X.shape[0]
        self.J = (X[:, 1:] - X[:, :1]).transpose(1, 2).contiguous()
        J = self.J.cpu()
        self.det, self.Jinv = torch.linalg.det(J).to(device), torch.linalg.inv(J).to(device)
        far, P, out = [], [], []
        for f in range(d + 1):
            own = [j for j in range(d + 1) if j != f]
            code = torch.zeros_like(key[:, 0])
            for j in own:
                code = code * len(coords) + key[:, j]
            far.append(code)
            P.append(X[:, own])
            out.append(torch.einsum("ecb,c->eb", self.Jinv, T["normal"][f]))
        code, P, out = torch.stack(far, 1), torch.stack(P, 1), torch.stack(out, 1)
        uniq, self.ef = torch.unique(code, return_inverse=True)              # sorted: lexicographic
        self.F = F = uniq.numel()
        if d == 3:
            n = torch.linalg.cross(P[:, :, 1] - P[:, :, 0], P[:, :, 2] - P[:, :, 0])
        else:
            t = P[:, :, 1] - P[:, :, 0]
            n = torch.stack([t[..., 1], -t[..., 0]], dim=-1)
        area = n.norm(dim=-1)
        n = n / area[..., None]
        s = torch.sign((n * out).sum(-1))                                    # +1: outward is n_F
        count = torch.zeros(F, dtype=torch.int64, device=device).index_add_(
            0, self.ef.reshape(-1), torch.ones(self.E * (d + 1), dtype=torch.int64, device=device))
        self.single = count == 1
        turn = torch.where(self.single[self.ef] & (s < 0), -1.0, 1.0)        # a boundary normal points out
        n, s = n * turn[..., None], s * turn
        self.sigma = s * torch.sign(self.det)[:, None]
        self.count = count.double()
        flat = self.ef.reshape(-1)
        self.n = torch.zeros(F, d, dtype=torch.float64, device=device)
        self.n[flat] = n.reshape(-1, d)
        self.area = torch.zeros(F, dtype=torch.float64, device=device)
        self.area[flat] = area.reshape(-1)
        slot = torch.arange(self.E * (d + 1), device=device)
        up = s.reshape(-1) > 0
        self.A = torch.zeros(F, dtype=torch.int64, device=device)            # element * (d+1) + local facet
        self.A[flat[up]] = slot[up]
        self.B = self.A.clone()
        self.B[flat[~up]] = slot[~up]
        PA = P.reshape(-1, d, d)[self.A]
        self.points_f = PA[:, None, 0] + torch.einsum("qj,Fjc->Fqc", T["sq"], PA[:, 1:] - PA[:, :1])
        self.n_l2 = self.E * d * T["nb"]
        self.n_v = F * T["nf"] + self.E * T["nint"]

    def parts(self):
        return [slice(a, min(self.E, a + self.CHUNK)) for a in range(0, self.E, self.CHUNK)]

    def points(self, p):
        return self.X0[p, None] + torch.einsum("ecj,qj->eqc", self.J[p], self.T["xq"])

    # inputs
    def interpolate(self, fun):
        """V_h coefficients of a field from its facet and interior moments."""
        T = self.T
        un = (fun(self.points_f) * self.n[:, None]).sum(-1)
        facet = self.area[:, None] * torch.einsum("Fq,q,qm->Fm", un, T["wf"], T["psi"])
        inner = [torch.einsum("eqb,jqb,q->ej", self.det[p, None, None] * torch.einsum("eba,eqa->eqb", self.Jinv[p], fun(self.points(p))),
                              T["z"], T["wq"]) for p in self.parts()]
        return torch.cat([facet.reshape(-1), torch.cat(inner).reshape(-1)])

    def project(self, fun):
        """L2 projection of a field, element by element."""
        T = self.T
        return torch.cat([torch.einsum("eqa,q,qi->eai", fun(self.points(p)), T["wq"], T["phi"]) for p in self.parts()]).reshape(-1)

    # the maps between V_h and L2
    def to_l2(self, v):
        T = self.T
        d, nf = T["d"], T["nf"]
        facet = v[: self.F * nf].reshape(self.F, nf)[self.ef] * self.sigma[:, :, None]
        local = torch.cat([facet.reshape(self.E, -1), v[self.F * nf:].reshape(self.E, -1)], dim=1)
        c = (local @ T["Dinv"].T).reshape(self.E, d, T["nb"])
        return torch.einsum("eab,ebi->eai", self.J / self.det[:, None, None], c)

    def to_v(self, u):
        T = self.T
        d, nf = T["d"], T["nf"]
        c = torch.einsum("eba,eai->ebi", self.det[:, None, None] * self.Jinv, u)
        local = c.reshape(self.E, -1) @ T["D"].T
        facet = (local[:, :(d + 1) * nf].reshape(self.E, d + 1, nf) * self.sigma[:, :, None]).reshape(-1, nf)
        facet = torch.zeros(self.F, nf, dtype=u.dtype, device=u.device).index_add(0, self.ef.reshape(-1), facet)
        return torch.cat([(facet / self.count[:, None]).reshape(-1), local[:, (d + 1) * nf:].reshape(-1)])

    # the operator, in its conservative form
    def apply(self, w, u, l):
        T = self.T
        d, nb, phi = T["d"], T["nb"], T["phi"]
        M = self.det.abs()[:, None, None] * self.Jinv
        r = torch.cat([-torch.einsum("eqa,eqc,qic->eai", torch.einsum("qi,eai->eqa", phi, u[p]) * T["wq"][:, None],
                                     torch.einsum("ecb,eqb->eqc", M[p], torch.einsum("qi,ebi->eqb", phi, w[p])), T["dphi"])
                       for p in self.parts()])

        def trace(v, at):
            out = torch.zeros(self.F, T["wf"].numel(), d, dtype=v.dtype, device=v.device)
            for f in range(d + 1):
                m = (at % (d + 1) == f).nonzero()[:, 0]
                out = out.index_copy(0, m, torch.einsum("qi,Fai->Fqa", T["side"][f], v[at[m] // (d + 1)]))
            return out

        uA, uB = trace(u, self.A), trace(u, self.B)
        wn = 0.5 * ((trace(w, self.A) + trace(w, self.B)) * self.n[:, None]).sum(-1)
        low = T["degree"][None] <= torch.as_tensor(l, device=u.device).reshape(-1, 1)      # [F or 1, nf]

        def rest(v):
            c = torch.einsum("Fqa,q,qm->Fma", v, T["wf"], T["psi"]) * low[..., None]
            t = torch.einsum("Fma,qm->Fqa", c, T["psi"])
            return v - t + (t * self.n[:, None]).sum(-1, keepdim=True) * self.n[:, None]

        g = wn[..., None] * 0.5 * (uA + uB) + rest(0.5 * wn.abs()[..., None] * rest(uA - uB))
        g = g * (self.area[:, None] * T["wf"])[..., None]
        for at, v, keep in ((self.A, g, slice(None)), (self.B, -g, ~self.single)):
            at, v = at[keep], v[keep]
            for f in range(d + 1):
                m = (at % (d + 1) == f).nonzero()[:, 0]
                r = r.index_add(0, at[m] // (d + 1), torch.einsum("Fqa,qi->Fai", v[m], T["side"][f]))
        return r / self.det.abs()[:, None, None]

    def l2(self, u):
        return u.reshape(self.E, self.T["d"], self.T["nb"])

    def substeps(self, u, dt, steps, l, w=None):
        """SSP-RK3; w None: the state is a V_h vector and its own wind."""
        def rhs(v):
            if w is not None:
                return self.apply(w, self.l2(v), l).reshape(-1)
            x = self.to_l2(v)
            return self.to_v(self.apply(x, x, l))
        for _ in range(steps):
            a = u - dt * rhs(u)
            b = 0.75 * u + 0.25 * (a - dt * rhs(a))
            u = u / 3.0 + 2.0 / 3.0 * (b - dt * rhs(b))
        return u


@lru_cache(maxsize=6)
def _mesh(dim, n, walls, k, device):
    return _Mesh(_box(dim, n, walls), k, device)


@lru_cache(maxsize=6)
def _class(c_meshes, k, device):
    return _Mesh(_class_mesh(c_meshes, k), k, device)


# ---------------------------------------------------------------------------- hexahedra, 64 bits
class _Hex:
    """The operator on a periodic box of parallelepipeds in plain torch."""

    def __init__(self, c, device):
        lines, A = _hex_box(c)
        self.n, self.k, k = (c["nx"], c["ny"], c["nz"]), c["k"], c["k"]
        x, w = _gauss_jacobi((3 * k + 2) // 2, 0)

        def legendre(t):
            P = _jacobi(k, 0, 2 * t - 1, np.ones_like(t))
            return np.stack([math.sqrt(2 * i + 1) * P[i] for i in range(k + 1)], axis=1)
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=device)  # noqa: E731
        self.L, self.dL = t(legendre(x)), t(legendre(x + 1e-40j).imag / 1e-40)
        self.end = t(legendre(np.array([0.0, 1.0])))
        self.x, self.w = t(x), t(w)
        h = [t(np.diff(a)) for a in lines]
        self.lo = [t(a[:-1]) for a in lines]
        self.A, self.Ainv, self.detA = t(A), t(np.linalg.inv(A)), float(np.linalg.det(A))
        one = [torch.ones_like(v) for v in h]
        grid = lambda a, b, c: torch.einsum("i,j,l->lji", a, b, c)             # noqa: E731  [nz, ny, nx]
        self.h = h
        self.H = torch.stack([grid(h[0], one[1], one[2]), grid(one[0], h[1], one[2]), grid(one[0], one[1], h[2])])
        self.vol = self.detA * self.H.prod(0)
        self.n_l2 = int(np.prod(self.n)) * 3 * (k + 1) ** 3

    def shape(self, u):
        """[nz, ny, nx, 3, i3, i2, i1]"""
        return u.reshape(self.n[2], self.n[1], self.n[0], 3, self.k + 1, self.k + 1, self.k + 1)

    def project(self, fun):
        k, m = self.k, self.x.numel()
        at = [self.lo[a][:, None] + self.h[a][:, None] * self.x for a in range(3)]     # [n_a, m]
        out = []
        for z in range(self.n[2]):
            g = torch.stack(torch.broadcast_tensors(at[0][None, :, None, None, :], at[1][:, None, None, :, None],
                                                    at[2][z][None, None, :, None, None]), dim=-1)
            f = fun(g @ self.A.T)
            v = torch.einsum("yxcbad,ai,bj,cl,a,b,c->yxdlji", f, self.L, self.L, self.L, self.w, self.w, self.w)
            out.append(v)
        return torch.stack(out).reshape(-1)

    def apply(self, w, u, l):
        slabs = [self._volume(self.shape(w)[z], self.shape(u)[z], z) for z in range(self.n[2])]
        return ((torch.stack(slabs) + self._facets(self.shape(w), self.shape(u), l)) / self.vol[..., None, None, None, None]).reshape(-1)

    def _volume(self, w, u, z):
        up = lambda v, a, b, c: torch.einsum("yxdlji,ai,bj,cl->yxdcba", v, a, b, c)    # noqa: E731
        L = self.L
        U, W = up(u, L, L, L), up(w, L, L, L)
        Wt = torch.einsum("cb,yxbrst->yxcrst", self.Ainv, W)                            # A^-1 w
        Wt = Wt * (self.vol[z][None] / self.H[:, z]).permute(1, 2, 0)[..., None, None, None]
        q = torch.einsum("a,b,c->cba", self.w, self.w, self.w)
        r = 0
        for c in range(3):
            t = [self.dL if a == c else L for a in range(3)]
            r = r - torch.einsum("yxdcba,ai,bj,cl->yxdlji", U * (Wt[:, :, c] * q)[:, :, None], t[0], t[1], t[2])
        return r

    def _facets(self, w, u, l):
        r = torch.zeros_like(u)
        L, wt = self.L, torch.einsum("a,b->ba", self.w, self.w)
        for a in range(3):
            ax, grid_ax = 6 - a, 2 - a                          # basis axis and cell axis of direction a
            v = self.detA * self.Ainv[a]
            n = v / v.norm()
            area = v.norm() * self.vol / self.detA / self.H[a]
            s, t = [b for b in range(3) if b != a]              # s the lower axis: first facet coordinate

            def trace(x, end):
                y = torch.tensordot(x, self.end[end], dims=([ax], [0]))                # [.., 3, (t), (s)]
                return torch.einsum("zyxdts,as,bt->zyxdba", y, L, L)

            uA, uB = trace(u, 1), torch.roll(trace(u, 0), -1, dims=grid_ax)
            wn = 0.5 * torch.einsum("zyxdba,d->zyxba", trace(w, 1) + torch.roll(trace(w, 0), -1, dims=grid_ax), n)

            def rest(y):
                if l < 0:
                    return y
                P = L[:, :l + 1]
                c = torch.einsum("zyxdba,ba,as,bt->zyxdts", y, wt, P, P)
                c = torch.einsum("zyxdts,as,bt->zyxdba", c, P, P)
                return y - c + torch.einsum("zyxdba,d,e->zyxeba", c, n, n)

            g = wn[:, :, :, None] * 0.5 * (uA + uB) + rest(0.5 * wn.abs()[:, :, :, None] * rest(uA - uB))
            g = g * wt * area[:, :, :, None, None, None]
            mom = torch.einsum("zyxdba,as,bt->zyxdts", g, L, L)
            hi = (mom.unsqueeze(ax) * self.end[1].reshape([-1 if i == ax else 1 for i in range(7)]))
            lo = torch.roll(mom, 1, dims=grid_ax).unsqueeze(ax) * self.end[0].reshape([-1 if i == ax else 1 for i in range(7)])
            r = r + hi - lo
        return r

    def substeps(self, u, dt, steps, l):
        for _ in range(steps):
            a = u - dt * self.apply(u, u, l)
            b = 0.75 * u + 0.25 * (a - dt * self.apply(a, a, l))
            u = u / 3.0 + 2.0 / 3.0 * (b - dt * self.apply(b, b, l))
        return u


@lru_cache(maxsize=4)
def _hex(nx, ny, nz, k, device):
    return _Hex(dict(nx=nx, ny=ny, nz=nz, k=k), device)


# ---------------------------------------------------------------------------- inputs
def _field(phase):
    """Taylor-Green with its origin moved by phase."""
    def f(x):
        y = x + phase
        if x.shape[-1] == 2:
            return torch.stack([y[..., 0].sin() * y[..., 1].cos(), -y[..., 0].cos() * y[..., 1].sin()], dim=-1)
        c = y[..., 2].cos()
        return torch.stack([y[..., 0].sin() * y[..., 1].cos() * c, -y[..., 0].cos() * y[..., 1].sin() * c,
                            torch.zeros_like(c)], dim=-1)
    return f


class _Make:
    """Input vectors of one seed: the first field, the second field, and so on."""

    def __init__(self, case, seed, device):
        self.g = torch.Generator(device=device).manual_seed(int(seed) * 2 + 1)
        self.dtype = torch.float64 if case["prec"] == "f64" else torch.float32
        self.device = device

    def field(self, d):
        return _field(torch.rand(d, generator=self.g, device=self.device, dtype=torch.float64) * TWO_PI)

    def noise(self, n):
        return (torch.rand(n, generator=self.g, device=self.device, dtype=torch.float64) * 2 - 1) * 1e-3

    def v(self, M):
        return (M.interpolate(self.field(M.T["d"])) + self.noise(M.n_v)).to(self.dtype)

    def l2(self, M, d):
        return (M.project(self.field(d)) + self.noise(M.n_l2)).to(self.dtype)

    def normal(self, n):
        return torch.randn(n, generator=self.g, device=self.device, dtype=torch.float64).to(self.dtype)


def _dt(case):
    return 1e-3 if case.get("dim") == 2 else 5e-4


def _inputs(case, seed, device):
    """The input vectors of a case, in the precision of the call."""
    make, kind = _Make(case, seed, device), case["kind"]
    if kind in ("hex", "hexsub"):
        H = _hex(case["nx"], case["ny"], case["nz"], case["k"], device)
        x = {"u": make.l2(H, 3)}
        if kind == "hex" and not case["same"]:
            x["w"] = make.l2(H, 3)
        return H, x
    if kind == "batch":
        pairs = tuple(_batch_meshes(case))
        M = [_class(pairs, k, device) for k in sorted({k for _, k in pairs})]
        return M, {"u": [make.v(m) for m in M]}
    d = case["dim"]
    M = _mesh(d, case["n"], bool(case.get("walls")), case["k"], device)
    x = {}
    if kind in ("apply", "grad") or (kind == "substep" and case["wind"] == "frozen"):
        x["w"] = make.v(M)
        x["u"] = make.l2(M, d)
    else:
        x["u"] = make.v(M)
    if case.get("orders"):
        x["l"] = torch.randint(-1, case["k"] + 1, (M.F,), generator=make.g, device=device).to(torch.int8)
    if kind == "grad":
        x["ybar"] = make.normal(M.n_l2)
    if kind == "rollout":
        x["ubar"] = make.normal(M.n_v)
    return M, x


# ---------------------------------------------------------------------------- the calls
def prepare(case, seed):
    from paper_2408_06698_gb300 import Hopu, HopuBatch, HopuHex

    _, x = _inputs(case, seed, "cuda")
    kind, k = case["kind"], case["k"] if "k" in case else None
    s = dict(case=case, dt=_dt(case), **x)
    if kind in ("hex", "hexsub"):
        lines, A = _hex_box(case)
        s["hopu"] = HopuHex(lines, A, k=k, prec=case["prec"])
        s["out"] = torch.empty_like(x["u"])
    elif kind == "batch":
        pairs = _batch_meshes(case)
        s["hopu"] = HopuBatch([_box(3, n) for n, _ in pairs], [kk for _, kk in pairs], l=-2, prec=case["prec"])
        s["state"] = [torch.empty_like(u) for u in x["u"]]
    else:
        coords, elems, rep = _box(case["dim"], case["n"], bool(case.get("walls")))
        s["hopu"] = Hopu(coords, elems, rep, k=k, l=k - 1, prec=case["prec"], wind=case.get("wind", "stage"))
        if kind == "substep":
            s["state"] = torch.empty_like(x["u"])
            if case["side"]:
                s["stream"] = torch.cuda.Stream()
            if case["wind"] == "frozen":
                s["hopu"].set_frozen_wind(x["w"])
    return s


def run(s):
    case, h = s["case"], s["hopu"]
    kind = case["kind"]
    if kind == "apply":
        return h.apply_convection(s["w"], s["u"], facet_l=s.get("l"))
    if kind == "substep":
        if not case["side"]:
            s["state"].copy_(s["u"])
            return h.rk_substep(s["state"], s["dt"], case["steps"])
        here = torch.cuda.current_stream()
        s["stream"].wait_stream(here)
        with torch.cuda.stream(s["stream"]):
            s["state"].copy_(s["u"])
            h.rk_substep(s["state"], s["dt"], case["steps"])
        here.wait_stream(s["stream"])
        return s["state"]
    if kind == "batch":
        for a, b in zip(s["state"], s["u"]):
            a.copy_(b)
        h.rk_substep(s["state"], s["dt"], 1)
        return s["state"]
    if kind == "grad":
        from paper_2408_06698_gb300 import ConvectionApply
        w, u = s["w"].detach().requires_grad_(), s["u"].detach().requires_grad_()
        y = ConvectionApply.apply(h, w, u)
        wbar, ubar = torch.autograd.grad(y, (w, u), s["ybar"])
        return {"y": y.detach(), "wbar": wbar, "ubar": ubar}
    if kind == "rollout":
        from paper_2408_06698_gb300 import Rollout
        u0 = s["u"].detach().requires_grad_()
        u = Rollout.apply(h, u0, s["dt"], case["steps"], case["ckpt"])
        (g,) = torch.autograd.grad(u, u0, s["ubar"])
        return {"u": u.detach(), "u0bar": g}
    if kind == "hex":
        return h.apply(s["u"] if case["same"] else s["w"], s["u"], case["k"] - 1, out=s["out"])
    s["out"].copy_(s["u"])
    return h.rk_substeps(s["out"], s["dt"], case["steps"], case["k"] - 1)


# ---------------------------------------------------------------------------- the results, 64 bits
def exact(case, seed, device="cuda"):
    M, x = _inputs(case, seed, device)
    kind, dt = case["kind"], _dt(case)
    if kind == "batch":
        return [m.substeps(u.double(), dt, 1, m.T["k"] - 1) for m, u in zip(M, x["u"])]
    l = case["k"] - 1
    if kind == "hex":
        return M.apply(x["u" if case["same"] else "w"].double(), x["u"].double(), l)
    if kind == "hexsub":
        return M.substeps(x["u"].double(), dt, case["steps"], l)
    if kind == "apply":
        return M.apply(M.to_l2(x["w"].double()), M.l2(x["u"].double()), x.get("l", l)).reshape(-1)
    if kind == "substep":
        w = M.to_l2(x["w"].double()) if case["wind"] == "frozen" else None
        return M.substeps(x["u"].double(), dt, case["steps"], l, w)
    if kind == "grad":
        w, u = x["w"].double().requires_grad_(), x["u"].double().requires_grad_()
        y = M.apply(M.to_l2(w), M.l2(u), l).reshape(-1)
        wbar, ubar = torch.autograd.grad(y, (w, u), x["ybar"].double())
        return {"y": y.detach(), "wbar": wbar, "ubar": ubar}
    u0 = x["u"].double().requires_grad_()
    u = u0
    with torch.autograd.graph.save_on_cpu() if M.E * case["steps"] > 40000 else torch.enable_grad():
        u = M.substeps(u0, dt, case["steps"], l)
    (g,) = torch.autograd.grad(u, u0, x["ubar"].double())
    return {"u": u.detach(), "u0bar": g}
