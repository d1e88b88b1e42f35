"""Performance cases of the slab library, through the entry points a user's program calls.

A case is one residual apply R(U) (``Slab.residual_apply``), one apply of the GMRES operator
A P^{-1} V (``Slab.operator_apply``) or one whole slab solve (``Slab.set_state``, ``slab_solve``,
``get_state``) on a synthetic mesh.  Keys of a case:

  kind    "residual" | "operator" | "solve"
  geom    "brick" | "affine" | "curved" | "octree" (2:1 faces, uneven p and q) |
          "timeref" (bricks, N_K in {1, 2, 4})
  prec    "fp64" | "fp32" (applies), "fp64" | "mixed" (solves)
  nx, ny, nz   grid (octree: nx is the base grid)
  p, q    degrees (octree: the largest, drawn per element from 1)
  order   "lex" | "morton" element numbering
  tol     relative residual of a solve

``exact`` restates the method in plain torch FP64 (quadrature tables, dense 1-D contractions,
one (p, q, N_K) class at a time) and shares no code with the library.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1307_5310_gb300 import meshgen, stm

SHEAR = ((1.0, 0.3, 0.1), (0.0, 0.9, -0.2), (0.15, 0.0, 1.1))


def listed():
    def c(name, kind, geom, prec, n, p, q, order="morton", **kw):
        nx, ny, nz = n if isinstance(n, tuple) else (n, n, n)
        return dict(name=name, kind=kind, geom=geom, prec=prec, nx=nx, ny=ny, nz=nz, p=p, q=q, order=order, **kw)

    return [
        # the smallest problem users run (the 4^3 cavity): one apply is launch latency
        c("residual-fp64-cavity4", "residual", "brick", "fp64", 4, 2, 1, "lex"),
        # the throughput workload: 64^3 bricks, p = 4, q = 3, both precisions
        c("residual-fp64-bricks64", "residual", "brick", "fp64", 64, 4, 3),
        c("residual-fp32-bricks64", "residual", "brick", "fp32", 64, 4, 3),
        # the operator a caller's own Krylov method applies: odd grid, plain numbering, low degree
        c("operator-fp32-bricks-odd", "operator", "brick", "fp32", (37, 41, 29), 3, 2, "lex"),
        # curved hexahedra: the O(p^5) mass, FP64 at the lowest and FP32 at the higher degrees
        c("residual-fp64-curved-p3", "residual", "curved", "fp64", 32, 3, 2),
        c("residual-fp32-curved-p5", "residual", "curved", "fp32", 32, 5, 4),
        c("operator-fp32-curved-p7", "operator", "curved", "fp32", (16, 15, 17), 7, 6, "lex"),
        # locally refined meshes: uneven degrees and 2:1 faces, then local time refinement
        c("residual-fp64-octree", "residual", "octree", "fp64", 30, 7, 4),
        c("operator-fp32-octree", "operator", "octree", "fp32", 30, 7, 4),
        c("residual-fp64-timeref", "residual", "timeref", "fp64", (25, 24, 23), 3, 2),
        # whole slab solves: the small cavity (latency of the Krylov loop) and a mixed-precision one
        c("solve-fp64-cavity4", "solve", "brick", "fp64", 4, 2, 1, "lex", tol=1e-12),
        c("solve-mixed-bricks32", "solve", "brick", "mixed", 32, 4, 3, tol=1e-10),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case: grids from a few cells to a few hundred thousand, every degree, geometry,
    precision and numbering of the listed ones, with at most about the largest listed work."""
    kind = rng.choice(("residual", "residual", "operator", "operator", "solve"))
    geom = rng.choice(("brick", "brick", "brick", "affine", "curved", "curved", "octree", "timeref"))
    if kind == "solve":
        geom = rng.choice(("brick", "brick", "affine", "timeref"))
    prec = rng.choice(("fp64", "mixed" if kind == "solve" else "fp32"))
    order = rng.choice(("lex", "morton"))
    if geom == "octree":
        nx = _log_int(rng, 4, 20)
        p, q = rng.randint(3, 7), rng.randint(2, 4)
        return dict(kind=kind, geom=geom, prec=prec, nx=nx, ny=nx, nz=nx, p=p, q=q, order=order)
    if geom == "curved":
        p = rng.randint(2, 7)
        q = max(1, p - rng.randint(1, 2))
    elif geom == "timeref":
        p, q = rng.randint(1, 4), rng.randint(1, 3)
    else:
        p, q = rng.randint(1, 7), rng.randint(1, 4)
    # trial coefficients: from a few thousand elements' worth of low degree up to a budget per kind
    budget = {"solve": 2e7, "residual": 1.5e8, "operator": 1.5e8}[kind]
    if geom in ("curved", "timeref"):
        budget = min(budget, 4e7)
    per = 6 * (q + 1) * (p + 1) ** 3 * (2 if geom == "timeref" else 1)
    n_max = max(4, int((budget / per) ** (1.0 / 3.0)))
    n = _log_int(rng, 4, min(n_max, 56))
    nx, ny, nz = (max(3, n + rng.randint(-n // 4, n // 4)) for _ in range(3))
    c = dict(kind=kind, geom=geom, prec=prec, nx=nx, ny=ny, nz=nz, p=p, q=q, order=order)
    if kind == "solve":
        c["tol"] = 1e-12 if prec == "fp64" else 1e-10
    return c


# ---- inputs ------------------------------------------------------------------------------------

@functools.lru_cache(maxsize=2)
def _grid(geom, nx, ny, nz, order):
    """Connectivity and vertices (the same for every seed)."""
    if geom == "octree":
        return meshgen.corner_octree_mesh(nx, [0.45, 0.2], order=order)
    if geom == "affine":
        return meshgen.box_mesh(nx, ny, nz, order=order, affine=SHEAR)
    return meshgen.box_mesh(nx, ny, nz, order=order, perturb=0.1 if geom == "curved" else 0.0)


def _mesh(case, seed):
    m = dict(_grid(case["geom"], case["nx"], case["ny"], case["nz"], case["order"]))
    ne = m["hex"].shape[0]
    m["p"], m["q"] = np.full(ne, case["p"], np.uint8), np.full(ne, case["q"], np.uint8)
    # the degrees and partitions belong to the case (they set the vectors' lengths), the materials
    # and coefficients to the seed
    if case["geom"] == "octree":
        meshgen.random_hp(m, 1307, p_range=(1, case["p"]), q_range=(1, case["q"]))
    if case["geom"] == "timeref":
        meshgen.random_nk(m, 1309)
    meshgen.random_materials(m, seed, seed + 1)
    return m


def _dt(case):
    n = max(case["nx"], case["ny"], case["nz"]) * (4 if case["geom"] == "octree" else 1)
    return 1.0 / n / (2 * case["p"] + 1)


def _dtype(case):
    return torch.float32 if case["prec"] == "fp32" else torch.float64


def _vector(case, seed, n):
    """Coefficients U[-1, 1]."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    return torch.empty(n, dtype=_dtype(case), device="cuda").uniform_(-1.0, 1.0, generator=g)


def _state(m, seed):
    """Slab-start coefficients of a field E_z = sum of three cavity modes sin(a pi x) sin(b pi y)
    with amplitudes from the seed, H = 0 (state layout), as an L2 projection on the boxes."""
    rng = np.random.Generator(np.random.PCG64(seed))
    amp = rng.uniform(0.5, 1.5, 3)
    x0 = m["vert"][m["hex"][:, 0]]
    h = m["vert"][m["hex"][:, 7]] - x0
    xg, wg = _gauss(14)
    p = int(m["p"][0])
    L = _legendre(p + 1, xg) * wg  # [n, g]
    ne, n = len(x0), p + 1
    Ez = torch.zeros(ne, n, n, dtype=torch.float64)
    for k, (a, b) in enumerate(((1, 1), (2, 1), (1, 3))):
        cx = np.sin(a * math.pi * (x0[:, :1] + h[:, :1] * xg)) @ L.T
        cy = np.sin(b * math.pi * (x0[:, 1:2] + h[:, 1:2] * xg)) @ L.T
        Ez += torch.from_numpy(amp[k] * h[:, 2][:, None, None] * cy[:, :, None] * cx[:, None, :])
    u = torch.zeros(ne, 2, 3, n, n, n, dtype=torch.float64)
    u[:, 0, 2, 0] = Ez
    return u.reshape(-1).cuda()


def prepare(case, seed):
    m = _mesh(case, seed)
    st = {"kind": case["kind"], "dt": _dt(case), "prec": stm.STM_FP32 if case["prec"] == "fp32" else stm.STM_FP64}
    if case["kind"] == "solve":
        st["slab"] = s = stm.Slab(m, precision=stm.STM_MIXED if case["prec"] == "mixed" else stm.STM_FP64,
                                  tol=case["tol"], max_it=2000)
        st["u0"] = _state(m, seed)
        st["out"] = torch.empty_like(st["u0"])
        return st
    st["slab"] = s = stm.Slab(m)
    st["x"] = _vector(case, seed, s.n_trial if case["kind"] == "residual" else s.n_test)
    st["y"] = torch.empty(s.n_test, dtype=_dtype(case), device="cuda")
    return st


def run(state):
    s = state["slab"]
    if state["kind"] == "residual":
        s.residual_apply(state["x"], state["y"], 0.0, state["dt"], prec=state["prec"])
        return state["y"]
    if state["kind"] == "operator":
        s.operator_apply(state["x"], state["y"], state["dt"], prec=state["prec"])
        return state["y"]
    s.set_state(state["u0"])
    _, report = s.slab_solve(state["dt"])
    s.get_state(state["out"])
    return {"state": state["out"], "energy": report["energy"]}


def work(case):
    """Inputs read once, outputs written once; the flops of the sum-factorised chain.  A solve
    counts one operator apply per iteration and reads of the growing basis (14 iterations, the
    count of the cavity at 1e-12)."""
    if case["geom"] == "octree":
        ne, pq = 1.63 * case["nx"] ** 3, [(p, q) for p in range(1, case["p"] + 1) for q in range(1, case["q"] + 1)]
    else:
        ne, pq = case["nx"] * case["ny"] * case["nz"], [(case["p"], case["q"])]
    es = {"fp32": 4, "mixed": 4, "fp64": 8}[case["prec"]]
    b = f = 0.0
    for p, q in pq:
        n, n2, n3, g = p + 1, (p + 1) ** 2, (p + 1) ** 3, p + 2
        nk = 7.0 / 3.0 if case["geom"] == "timeref" else 1.0
        qe = nk * q
        mass = 3 * qe * n3
        if case["geom"] == "curved":
            mass = qe * (6 * (n3 * g + n2 * g * g + n * g ** 3) + 9 * g ** 3)
        elif case["geom"] == "affine":
            mass = 9 * qe * n3
        fl = 2 * 2 * (3 * n3 * nk * (2 * q + 1 if q > 1 else 2) + 12 * qe * n3 + mass + 6 * qe * n2 * (n * n // 4))
        read = 6 * (qe + 1) * n3 if case["kind"] == "residual" else 6 * qe * n3
        by = es * (read + 6 * qe * n3) + 16 + (192 if case["geom"] in ("curved", "affine") else 0)
        b, f = b + ne * by / len(pq), f + ne * fl / len(pq)
    if case["kind"] == "solve":
        n_un = ne * 6 * qe * n3
        its = 14
        b, f = its * b + es * n_un * sum(2 * (j % 10 + 1) for j in range(its)), its * f
    return {"bytes": b, "flops": f}


# ---- the method in plain torch FP64 ------------------------------------------------------------

def _gauss(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (x + 1.0), 0.5 * w


def _legendre(n, x):
    """L_0..L_{n-1}, orthonormal on [0, 1], at the points x: [n, len(x)]."""
    return np.stack([np.polynomial.legendre.legval(2.0 * np.asarray(x) - 1.0, np.eye(n)[k]) * math.sqrt(2 * k + 1)
                     for k in range(n)])


def _dlegendre(n, x):
    return np.stack([2.0 * np.polynomial.legendre.legval(2.0 * np.asarray(x) - 1.0,
                                                         np.polynomial.legendre.legder(np.eye(n)[k]))
                     * math.sqrt(2 * k + 1) for k in range(n)])


def _time_tables(q):
    """A[i, m] = int L_i l_m', B[i, m] = int L_i l_m for the trial functions 1 - s, s and the
    integrated Legendre polynomials."""
    x, w = _gauss(q + 3)
    L = _legendre(q, x)
    l, dl = np.zeros((q + 1, x.size)), np.zeros((q + 1, x.size))
    l[0], l[1], dl[0], dl[1] = 1.0 - x, x, -1.0, 1.0
    for m in range(2, q + 1):
        dl[m] = L[m - 1]
        l[m] = [t * np.sum(w * _legendre(q, t * x)[m - 1]) for t in x]
    return (L * w) @ dl.T, (L * w) @ l.T


def _time_transfer(q, nk, q2, nk2):
    """M with <H', Pi phi_own> = M (moments of H' against the neighbour's test functions): Pi is
    the projection onto the common test space (the lower degree on the coarser partition)."""
    r, qc, nc = max(nk, nk2), min(q, q2), min(nk, nk2)
    x, w = _gauss(max(q, q2) + 1)
    t = ((np.arange(r)[:, None] + x) / r).ravel()
    wt = np.tile(w, r) / r

    def piecewise(qq, n):
        out = np.zeros((n * qq, t.size))
        for k in range(n):
            s = (t * n - k)
            inside = (s > 0) & (s < 1)
            out[k * qq:(k + 1) * qq, inside] = _legendre(qq, s[inside])
        return out

    own, nb, com = piecewise(q, nk), piecewise(q2, nk2), piecewise(qc, nc) * math.sqrt(nc)
    return (own * wt) @ com.T @ ((com * wt) @ nb.T * nk2)


class _Exact:
    """R(U) and A P^{-1} V of a mesh dict, FP64, on the device torch has."""

    def __init__(self, m, dt):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.m, self.dt = m, dt
        ne = m["hex"].shape[0]
        nk = np.asarray(m.get("nk", np.ones(ne)), np.int64)
        key = np.stack([m["p"].astype(np.int64), m["q"].astype(np.int64), nk], 1)
        self.classes, inv = np.unique(key, axis=0, return_inverse=True)
        inv = inv.reshape(-1)
        self.cls, self.pos = inv, np.zeros(ne, np.int64)
        self.elems = [np.nonzero(inv == k)[0] for k in range(len(self.classes))]
        for e in self.elems:
            self.pos[e] = np.arange(e.size)
        self.X = m["vert"][m["hex"]]  # [ne, 8, 3]
        self.mat = np.stack([m["eps"], m["mu"]], 1)

    def t(self, a):
        return torch.as_tensor(np.ascontiguousarray(a), device=self.dev)

    def offsets(self, trial):
        p, q, k = (self.classes[self.cls][:, j] for j in range(3))
        return np.concatenate([[0], np.cumsum(6 * (k * q + (1 if trial else 0)) * (p + 1) ** 3)])

    def gather(self, v, trial):
        """Per class [ne_c, 2, 3, T, n, n, n] of a global vector."""
        off, out = self.offsets(trial), []
        for (p, q, k), e in zip(self.classes, self.elems):
            T, n = k * q + (1 if trial else 0), p + 1
            size = 6 * T * n ** 3
            if len(self.classes) == 1:
                out.append(v.reshape(len(e), 2, 3, T, n, n, n))
            else:
                idx = self.t(off[e])[:, None] + torch.arange(int(size), device=self.dev)
                out.append(v[idx].reshape(len(e), 2, 3, T, n, n, n))
        return out

    def scatter(self, parts):
        off = self.offsets(False)
        if len(parts) == 1:
            return parts[0].reshape(-1)
        r = torch.empty(int(off[-1]), dtype=torch.float64, device=self.dev)
        for x, e in zip(parts, self.elems):
            x = x.reshape(len(e), -1)
            r[self.t(off[e])[:, None] + torch.arange(x.shape[1], device=self.dev)] = x
        return r

    def metric(self, e, p):
        """w_g |J| DF^{-1} DF^{-T} at (p+2)^3 Gauss points, [ne, 3, 3, gz, gy, gx]; the weights."""
        x, w = _gauss(p + 2)
        bit = np.array([[v & 1, (v >> 1) & 1, (v >> 2) & 1] for v in range(8)])
        f = np.where(bit[:, :, None] == 1, x, 1.0 - x)  # [8, 3, g]
        d = np.where(bit[:, :, None] == 1, np.ones_like(x), -np.ones_like(x))
        dN = np.stack([np.einsum("va,vb,vc->vcba", *(d[:, k] if k == a else f[:, k] for k in range(3)))
                       for a in range(3)], 1)  # [8, axis, gz, gy, gx]
        DF = torch.einsum("evi,vjabc->eabcij", self.t(self.X[e]), self.t(dN))
        J = torch.linalg.det(DF)
        F = torch.linalg.inv(DF)
        W = self.t(np.einsum("a,b,c->abc", w, w, w))
        return (J * W)[..., None, None] * (F @ F.transpose(-1, -2))

    def mass(self, k, v):
        """Metric mass of v [ne, 2, 3, T, n, n, n]."""
        p, e = int(self.classes[k][0]), self.elems[k]
        mat = self.t(self.mat[e])
        if self.m.get("geometry", "brick") == "trilinear":
            L = self.t(_legendre(p + 1, _gauss(p + 2)[0]))
            out = torch.empty_like(v)
            for s in range(0, len(e), 1024):
                G = self.metric(e[s:s + 1024], p)
                for f in range(2):
                    x = torch.einsum("emtlkj,la,kb,jc->emtabc", v[s:s + 1024, f], L, L, L)
                    x = torch.einsum("eabcdm,emtabc->edtabc", G, x)
                    x = torch.einsum("emtabc,la,kb,jc->emtlkj", x, L, L, L)
                    out[s:s + 1024, f] = mat[s:s + 1024, f, None, None, None, None, None] * x
            return out
        return torch.einsum("ef,ecd,efdtlkj->efctlkj", mat, self.mean_metric(k), v)

    def mean_metric(self, k):
        p, e = int(self.classes[k][0]), self.elems[k]
        if self.m.get("geometry", "brick") == "trilinear":
            return torch.cat([self.metric(e[s:s + 4096], p).sum((1, 2, 3)) for s in range(0, len(e), 4096)])
        X = self.X[e]
        DF = self.t(np.stack([X[:, 1] - X[:, 0], X[:, 2] - X[:, 0], X[:, 4] - X[:, 0]], 2))
        F = torch.linalg.inv(DF)
        return torch.linalg.det(DF)[:, None, None] * (F @ F.transpose(-1, -2))

    def precondition(self, v):
        """P^{-1}: the inverse of the cell-mean metric mass, per temporal and spatial index."""
        out = []
        for k, x in enumerate(self.gather(v, False)):
            inv = torch.linalg.inv(self.mean_metric(k))
            out.append(torch.einsum("ef,ecd,efdtlkj->efctlkj", 1.0 / self.t(self.mat[self.elems[k]]), inv, x))
        return self.scatter(out)

    def operator(self, v):
        """A v: the residual of v as the unknown modes, slab start 0."""
        return self.residual([torch.cat([torch.zeros_like(x[:, :, :, :1]), x], 3) for x in self.gather(v, False)])

    def residual(self, U):
        """R(U) from the per-class trial blocks U."""
        hang = np.asarray(self.m.get("hang", np.zeros((0, 6), np.int64))).reshape(-1, 6)
        Y, R = [], []
        for k, (p, q, nk) in enumerate(self.classes):
            A, B = (self.t(a) for a in _time_tables(int(q)))
            u = U[k]
            y, du = [], []
            for s in range(nk):
                idx = [0 if s == 0 else 1 + (s - 1) * q] + [1 + s * q + i for i in range(q)]
                sub = u[:, :, :, idx]
                y.append(torch.einsum("im,efcmlkj->efcilkj", B, sub) * (self.dt / nk))
                du.append(torch.einsum("im,efcmlkj->efcilkj", A, sub))
            Y.append(torch.cat(y, 3))
            R.append(self.mass(k, torch.cat(du, 3)))
            del y, du
        for k, (p, q, nk) in enumerate(self.classes):
            n = int(p) + 1
            x, w = _gauss(n + 1)
            D = self.t((_legendre(n, x) * w) @ _dlegendre(n, x).T)  # int L_a L_b'
            for a in range(3):  # derivative axis; tensor dim of x, y, z is 6, 5, 4
                b, c = (a + 1) % 3, (a + 2) % 3
                dY = torch.tensordot(Y[k], D, dims=([6 - a], [1])).movedim(-1, 6 - a)
                # (curl y)_c += d_a y_b, (curl y)_b -= d_a y_c
                R[k][:, 0, c] -= dY[:, 1, b]
                R[k][:, 0, b] += dY[:, 1, c]
                R[k][:, 1, c] += dY[:, 0, b]
                R[k][:, 1, b] -= dY[:, 0, c]
                del dY
                for side in (0, 1):
                    lift = self.t(_legendre(n, [float(side)])[:, 0])
                    own = self.trace(Y[k], a, side)  # [ne, 2, 3, T, s, f]
                    jump = own - self.other(Y, k, a, side, own, hang)
                    g = torch.einsum("efctuv,l->efctluv", jump, lift).movedim(4, 6 - a) * (0.5 if side else -0.5)
                    # n x (0.5 jump), n = +-e_a: component c gets +jump_b, component b gets -jump_c
                    R[k][:, 0, c] += g[:, 1, b]
                    R[k][:, 0, b] -= g[:, 1, c]
                    R[k][:, 1, c] -= g[:, 0, b]
                    R[k][:, 1, b] += g[:, 0, c]
                    del own, jump, g
        return self.scatter(R)

    def trace(self, y, a, side):
        L = self.t(_legendre(y.shape[-1], [float(side)])[:, 0])
        return torch.tensordot(y, L, dims=([6 - a], [0]))

    def other(self, Y, k, a, side, own, hang):
        """The other side's trace on face (a, side) of class k in its own test space: the
        neighbour's, or on the boundary the mirror value (E: -own, H: +own)."""
        e = self.elems[k]
        q, nk = int(self.classes[k][1]), int(self.classes[k][2])
        out = own.clone()
        out[:, 0] *= -1.0
        nb = self.m["nbr"][e, 2 * a + side]
        x, w = _gauss(10)
        T1 = [_legendre(8, 0.5 * (x + u)) * w @ _legendre(8, x).T for u in (0, 1)]  # [u][coarse mode, fine mode]
        inner = np.nonzero(nb == -2)[0]
        if inner.size:
            out[self.t(inner)] = 0.0
        for k2 in range(len(self.classes)):
            q2, nk2 = int(self.classes[k2][1]), int(self.classes[k2][2])
            M = self.t(_time_transfer(q, nk, q2, nk2))
            sel = np.nonzero((nb >= 0) & (self.cls[np.maximum(nb, 0)] == k2))[0]
            if sel.size:
                for s in range(0, sel.size, 65536):
                    part = sel[s:s + 65536]
                    tr = self.trace(Y[k2][self.t(self.pos[nb[part]])], a, 1 - side)
                    out[self.t(part)] = self.pad(torch.einsum("ij,efcjuv->efciuv", M, tr), own.shape[-1])
            if not hang.size or not inner.size:
                continue
            # rows where an element of class k is the fine side, then the coarse side
            for fine in (True, False):
                me, face, them = (2, 3, 0) if fine else (0, 1, 2)
                rows = hang[(self.cls[hang[:, me]] == k) & (hang[:, face] == 2 * a + side)
                            & (self.cls[hang[:, them]] == k2)]
                for u in (0, 1):
                    for v in (0, 1):
                        r = rows[(rows[:, 4] == u) & (rows[:, 5] == v)]
                        if not len(r):
                            continue
                        tr = self.trace(Y[k2][self.t(self.pos[r[:, them]])], a, 1 - side)
                        n2, n1 = tr.shape[-1], own.shape[-1]
                        # the last tensor index is the lower tangential axis
                        Tu, Tv = (self.t(T1[w][:n2, :n1] if fine else T1[w][:n1, :n2].T) for w in (u, v))
                        z = 0.5 * torch.einsum("ij,efcjab,am,bn->efcimn", M, tr, Tv, Tu)
                        out.index_add_(0, self.t(self.pos[r[:, me]]), z)
        return out

    @staticmethod
    def pad(x, n):
        m = min(n, x.shape[-1])
        y = x.new_zeros(x.shape[:-2] + (n, n))
        y[..., :m, :m] = x[..., :m, :m]
        return y

    def solve(self, u0):
        """End state of the slab from the state u0: GMRES without restarts to 1e-13."""
        st = u0.reshape(-1)
        n = [int(p) + 1 for p in self.classes[:, 0]]
        off = np.concatenate([[0], np.cumsum([6 * n[c] ** 3 for c in self.cls])])
        start = [st[self.t(off[e])[:, None] + torch.arange(6 * m ** 3, device=self.dev)].reshape(-1, 2, 3, 1, m, m, m)
                 for e, m in zip(self.elems, n)]
        guess = []
        for (p, q, nk), s in zip(self.classes, start):
            g = s.new_zeros(s.shape[:3] + (int(q * nk),) + s.shape[4:])
            g[:, :, :, ::int(q)] = s
            guess.append(g)
        x = self.scatter(guess)
        r = -self.residual([torch.cat([s, g], 3) for s, g in zip(start, guess)])
        ref = self.residual([torch.cat([s, torch.zeros_like(g)], 3) for s, g in zip(start, guess)]).norm()
        beta = r.norm()
        V, H = [r / beta], np.zeros((61, 60))
        for j in range(60):
            w = self.operator(self.precondition(V[j]))
            for _ in range(2):
                for i in range(j + 1):
                    h = torch.dot(V[i], w)
                    H[i, j] += float(h)
                    w -= h * V[i]
            H[j + 1, j] = float(w.norm())
            V.append(w / H[j + 1, j])
            b = np.zeros(j + 2)
            b[0] = float(beta)
            y, res = np.linalg.lstsq(H[:j + 2, :j + 1], b, rcond=None)[:2]
            if np.linalg.norm(H[:j + 2, :j + 1] @ y - b) <= 1e-13 * float(ref):
                break
        x = x + self.precondition(sum(float(c) * v for c, v in zip(y, V)))
        end = [g[:, :, :, int(q * (nk - 1))] for (p, q, nk), g in zip(self.classes, self.gather(x, False))]
        if len(end) == 1:
            return end[0].reshape(-1)
        out = torch.empty_like(st)
        for z, e in zip(end, self.elems):
            z = z.reshape(len(e), -1)
            out[self.t(off[e])[:, None] + torch.arange(z.shape[1], device=self.dev)] = z
        return out

    def energy(self, st):
        n = [int(p) + 1 for p in self.classes[:, 0]]
        off = np.concatenate([[0], np.cumsum([6 * n[c] ** 3 for c in self.cls])])
        tot = 0.0
        for k, e in enumerate(self.elems):
            idx = self.t(off[e])[:, None] + torch.arange(6 * n[k] ** 3, device=self.dev)
            v = st[idx].reshape(len(e), 2, 3, 1, n[k], n[k], n[k])
            tot += 0.5 * float((v * self.mass(k, v)).sum())
        return tot


def exact(case, seed):
    m = _mesh(case, seed)
    x = _Exact(m, _dt(case))
    n_trial, n_test = int(x.offsets(True)[-1]), int(x.offsets(False)[-1])
    if case["kind"] == "solve":
        if n_test > 1e8:
            return None
        st = x.solve(_state(m, seed))
        return {"state": st, "energy": x.energy(st)}
    if case["kind"] == "residual":
        return x.residual(x.gather(_vector(case, seed, n_trial).double(), True))
    return x.operator(x.precondition(_vector(case, seed, n_test).double()))
