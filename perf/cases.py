"""Performance cases of the modal DG library, through its public Python API.

Every case is a piece of work that a flow solver has the library do: one
residual, LSERK steps, an adjoint.  prepare() makes what the
program holds beforehand (the mesh handle, the state in the caller's layout,
output buffers), run() is one call sequence of such a program and returns the
whole result in the caller's layout, exact() evaluates the same discretisation
with dense operators in plain torch.

Meshes are periodic boxes [-pi, pi]^3 of m^3 cubes, each cube kept as a
hexahedron or split into prisms, pyramids or tetrahedra; the flow is the
Taylor-Green vortex at Mach 0.1 with a smooth random perturbation.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2511_08020_gb300 as dg

GAMMA, MACH, PRANDTL, MU = 1.4, 0.1, 0.72, 1.0 / 1600.0
HEX, PRISM, PYR, TET = 0, 1, 2, 3


# --------------------------------------------------------------------------- the cases

def listed():
    """What each case stands for is said beside it."""
    return [
        # one residual of a small mesh of all four types: unit runs, outer solvers; launches and latency
        dict(name="residual_small", op="rhs", kind="four", m=4, N=2, flux="lf", mesh_seed=1),
        # the explicit time loop on the mixed mesh, N = 4: the ordinary production run
        dict(name="steps_mixed", op="step", kind="mixed", m=16, N=4, flux="lf", steps=2, mesh_seed=2),
        # tetrahedral mesh, low degree, the Roe flux
        dict(name="steps_tets_roe", op="step", kind="kuhn", m=9, N=3, flux="roe", steps=2, mesh_seed=1),
        # viscous vortex on 512 hexahedra, N = 5
        dict(name="viscous_hex", op="step", physics="ns", kind="hex", m=8, N=5, flux="lf", steps=2, mesh_seed=1),
        # viscous vortex on a mesh of all four types, N = 5
        dict(name="viscous_four", op="step", physics="ns", kind="four", m=7, N=5, flux="lf", steps=1, mesh_seed=3),
        # the largest: viscous vortex on a fine mixed mesh
        dict(name="viscous_large", op="step", physics="ns", kind="mixed", m=20, N=4, flux="lf", steps=1, mesh_seed=2),
        # curved elements (every vertex moved): pointwise geometry, dense element mass matrices
        dict(name="steps_curved", op="step", kind="mixed", m=12, N=4, flux="lf", steps=2, mesh_seed=2, perturb=0.1),
        # the mesh in motion: the mass matrices are solved afresh every stage
        dict(name="steps_moving", op="moving", kind="mixed", m=8, N=3, flux="lf", steps=2, mesh_seed=2, perturb=0.1),
        # entropy-stable split form on the hexahedra
        dict(name="steps_split", op="step", kind="mixed", m=10, N=4, flux="lf", steps=1, mesh_seed=2, form="split"),
        # many independent meshes of several degrees as one batch
        dict(name="steps_batch", op="batch", sizes="4:2,7:3,5:4,9:2,6:5,8:3,5:1,4:6", flux="lf", steps=1, mesh_seed=5),
        # gradient of a functional through the residual (adjoint of dg_rhs)
        dict(name="residual_adjoint", op="rhs_vjp", kind="mixed", m=13, N=3, flux="lf", mesh_seed=2),
        # gradient through a viscous trajectory with checkpoints
        dict(name="steps_adjoint", op="rk_vjp", physics="ns", kind="mixed", m=6, N=4, flux="lf", steps=4, every=2,
             mesh_seed=2),
    ]


# no drawn case costs more than the largest listed one
_MAX_FLOPS = 2.7e10


def draw(rng):
    """One more case of the same ranges: any operation, mesh kind, degree 1 to 6, size over its logarithm."""
    while True:
        op = rng.choice(["rhs", "step", "step", "step", "viscous", "curved", "moving", "split", "batch", "rhs_vjp",
                         "rk_vjp"])
        kind = rng.choice(["mixed", "mixed", "four", "hex", "kuhn"])
        N = rng.randint(1, 6)
        m = int(round(math.exp(rng.uniform(math.log(4), math.log(20)))))
        c = dict(op="step", kind=kind, m=m, N=N, flux="lf", steps=rng.randint(1, 3), mesh_seed=rng.randint(1, 99))
        if op == "rhs":
            c.update(op="rhs")
            c.pop("steps")
        elif op == "step":
            c.update(flux=rng.choice(["lf", "lf", "roe"]))
        elif op == "viscous":
            c.update(physics="ns")
        elif op == "curved":
            c.update(kind=rng.choice(["mixed", "four"]), m=min(m, 12), perturb=0.1)
        elif op == "moving":
            c.update(op="moving", kind="mixed", m=min(m, 9), N=min(N, 4), perturb=0.1)
        elif op == "split":
            c.update(kind=rng.choice(["mixed", "hex"]), m=min(m, 12), N=min(N, 5), form="split")
        elif op == "batch":
            k = rng.randint(2, 9)
            c = dict(op="batch", sizes=",".join(f"{rng.randint(4, 9)}:{rng.randint(1, 5)}" for _ in range(k)),
                     flux="lf", steps=rng.randint(1, 2), mesh_seed=rng.randint(1, 99))
        elif op == "rhs_vjp":
            c.update(op="rhs_vjp", flux=rng.choice(["lf", "roe"]), m=min(m, 14))
            c.pop("steps")
        elif op == "rk_vjp":
            c.update(op="rk_vjp", physics=rng.choice(["euler", "ns"]), m=min(m, 6), N=min(N, 4),
                     steps=rng.randint(2, 5), every=rng.randint(1, 3))
        if work(c)["flops"] <= _MAX_FLOPS:
            return c


# --------------------------------------------------------------------------- meshes

class Box:
    """Mesh arrays in the layout the library reads, plus the vertices' periodic identities."""

    def __init__(self, m, kind, seed):
        rng = np.random.Generator(np.random.PCG64([7, m, seed]))
        n1 = m + 1
        ax = -math.pi + 2 * math.pi / m * np.arange(n1)
        k, j, i = (x.ravel() for x in np.meshgrid(np.arange(n1), np.arange(n1), np.arange(n1), indexing="ij"))
        xyz = np.stack([ax[i], ax[j], ax[k]], axis=1)
        pid = (i % m) + m * ((j % m) + m * (k % m))
        ck, cj, ci = (x.ravel() for x in np.meshgrid(np.arange(m), np.arange(m), np.arange(m), indexing="ij"))
        column = rng.random((m, m))[ci, cj] < 0.5             # prism columns along z
        cube = rng.random(m ** 3) < 0.5                        # pyramid cubes elsewhere
        what = {"hex": np.full(m ** 3, HEX), "kuhn": np.full(m ** 3, TET)}.get(kind)
        if what is None:
            what = np.where(column, PRISM, np.where(cube, PYR, HEX))
        split = np.zeros(m ** 3, dtype=int)                    # pyramid cubes with one base cut into two tetrahedra
        if kind == "four":
            w = max(1, m // 4)
            what = np.where(ci < w, TET, np.where((ci == w) | (ci == m - 1), PYR, what))
            split = np.where(ci == w, 1, np.where(ci == m - 1, 2, 0))

        def corner(c, dx, dy, dz):
            return (ci[c] + dx) + n1 * ((cj[c] + dy) + n1 * (ck[c] + dz))

        elems = []                                             # (cube, local index, type, vertices)

        def add(c, loc, t, verts):
            elems.append((c, np.full(len(c), loc), np.full(len(c), t), np.stack(verts, axis=1)))

        c = np.nonzero(what == HEX)[0]
        add(c, 0, HEX, [corner(c, b & 1, (b >> 1) & 1, b >> 2) for b in range(8)])
        c = np.nonzero(what == PRISM)[0]
        for loc, tri in enumerate((((0, 0), (1, 0), (1, 1)), ((0, 0), (1, 1), (0, 1)))):
            add(c, loc, PRISM, [corner(c, a, b, z) for z in (0, 1) for a, b in tri])
        c = np.nonzero(what == TET)[0]
        for loc, perm in enumerate(((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0))):
            d, path = [0, 0, 0], [corner(c, 0, 0, 0)]
            for a in perm:
                d[a] = 1
                path.append(corner(c, *d))
            add(c, loc, TET, path)
        c = np.nonzero(what == PYR)[0]
        centre = np.zeros(m ** 3, dtype=np.int64)
        centre[c] = len(xyz) + np.arange(len(c))
        h = 2 * math.pi / m
        xyz = np.concatenate([xyz, -math.pi + h * (np.stack([ci[c], cj[c], ck[c]], axis=1) + 0.5)])
        pid = np.concatenate([pid, m ** 3 + c])
        for axis in range(3):
            u, w = [d for d in range(3) if d != axis]
            for side in (0, 1):
                cut = split[c] == (1 + side) if axis == 0 else np.zeros(len(c), dtype=bool)

                def base(cc):
                    out = []
                    for bw in (0, 1):
                        for bu in (0, 1):
                            d = [0, 0, 0]
                            d[axis], d[u], d[w] = side, bu, bw
                            out.append(corner(cc, *d))
                    return out
                cp, ct = c[~cut], c[cut]
                add(cp, 2 * axis + side, PYR, base(cp) + [centre[cp]])
                b = base(ct)
                add(ct, 6, TET, [b[0], b[1], b[3], centre[ct]])
                add(ct, 7, TET, [b[0], b[2], b[3], centre[ct]])
        cubes = np.concatenate([e[0] for e in elems])
        locs = np.concatenate([e[1] for e in elems])
        order = np.lexsort((locs, cubes))
        types = np.concatenate([e[2] for e in elems])[order]
        padded = np.concatenate([np.pad(e[3], ((0, 0), (0, 8 - e[3].shape[1])), constant_values=-1) for e in elems])[order]
        self.xyz, self.pid, self.m = xyz, pid, m
        self.etype = types.astype(np.int8)
        self.padded = padded
        self.elem_verts = padded[padded >= 0].astype(np.int64)
        self.elem_vert_off = np.concatenate([[0], np.cumsum((padded >= 0).sum(axis=1))]).astype(np.int64)
        self.period = np.full(3, 2 * math.pi)

    def perturb(self, amp, seed):
        """Move every vertex by up to amp of the cube side per coordinate (periodic images together)."""
        u = np.random.Generator(np.random.PCG64([11, seed])).uniform(-1, 1, size=(self.pid.max() + 1, 3))
        self.xyz = self.xyz + amp * (2 * math.pi / self.m) * u[self.pid]

    def velocity(self, amp=0.1):
        """Constant vertex velocities: a smooth periodic field."""
        x = self.xyz
        return amp * np.stack([np.sin(x[:, 1]) * np.sin(x[:, 2]), np.sin(x[:, 2]) * np.sin(x[:, 0]),
                               np.sin(x[:, 0]) * np.sin(x[:, 1])], axis=1)


def _box(case, m=None, seed=None):
    b = Box(m or case["m"], case.get("kind", "mixed"), case["mesh_seed"] if seed is None else seed)
    if case.get("perturb"):
        b.perturb(case["perturb"], case["mesh_seed"])
    return b


def _instances(case):
    """(box, N) of every mesh of the case."""
    if case["op"] == "batch":
        pairs = [tuple(int(x) for x in s.split(":")) for s in case["sizes"].split(",")]
        return [(_box(case, m, case["mesh_seed"] + i), N) for i, (m, N) in enumerate(pairs)]
    return [(_box(case), case["N"])]


def _dt(m, N):
    return 0.15 * (2 * math.pi / m) / ((2 * N + 1) * (1.0 + 1.0 / MACH))


def _case_dt(case):
    if case["op"] == "batch":
        return min(_dt(int(s.split(":")[0]), int(s.split(":")[1])) for s in case["sizes"].split(","))
    return _dt(case["m"], case["N"])


# --------------------------------------------------------------------------- reference elements

VERTS = {HEX: [[(-1, 1)[b & 1], (-1, 1)[(b >> 1) & 1], (-1, 1)[b >> 2]] for b in range(8)],
         PRISM: [[-1, -1, -1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1], [1, -1, 1], [-1, 1, 1]],
         PYR: [[-1, -1, -1], [1, -1, -1], [-1, 1, -1], [1, 1, -1], [-1, -1, 1]],
         TET: [[-1, -1, -1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]]}
# local faces: the collapsed coordinate held fixed (0, 1, 2 = a, b, c), its end, and the face's vertices
FACES = {HEX: [(2, -1, (0, 1, 2, 3)), (2, 1, (4, 5, 6, 7)), (1, -1, (0, 1, 4, 5)), (1, 1, (2, 3, 6, 7)),
               (0, -1, (0, 2, 4, 6)), (0, 1, (1, 3, 5, 7))],
         PRISM: [(2, -1, (0, 1, 2)), (2, 1, (3, 4, 5)), (1, -1, (0, 1, 3, 4)), (0, -1, (0, 2, 3, 5)),
                 (0, 1, (1, 2, 4, 5))],
         PYR: [(2, -1, (0, 1, 2, 3)), (1, -1, (0, 1, 4)), (0, -1, (0, 2, 4)), (0, 1, (1, 3, 4)), (1, 1, (2, 3, 4))],
         TET: [(2, -1, (0, 1, 2)), (1, -1, (0, 1, 3)), (0, -1, (0, 2, 3)), (0, 1, (1, 2, 3))]}


@functools.lru_cache(maxsize=None)
def _modes(t, N):
    out = []
    for p in range(N + 1):
        for q in range((N - p if t in (PRISM, TET) else N) + 1):
            top = {HEX: N, PRISM: N, TET: N - p - q, PYR: N - max(p, q)}[t]
            out += [(p, q, r) for r in range(top + 1)]
    return out


@functools.lru_cache(maxsize=None)
def _gauss(n):
    """Gauss-Legendre points and weights in extended precision."""
    x = np.polynomial.legendre.leggauss(n)[0].astype(np.longdouble)
    for _ in range(2):
        p0, p1 = np.ones_like(x), x
        for k in range(2, n + 1):
            p0, p1 = p1, ((2 * k - 1) * x * p1 - (k - 1) * p0) / k
        dp = n * (x * p1 - p0) / (x * x - 1)
        x = x - p1 / dp
    return x, 2 / ((1 - x * x) * dp * dp)


def _jacobi(n, al, be, x):
    p0 = np.ones_like(x)
    if n == 0:
        return p0
    p1 = ((al - be) + (al + be + 2) * x) / 2
    for k in range(2, n + 1):
        s = 2 * k + al + be
        p0, p1 = p1, ((s - 1) * (s * (s - 2) * x + al * al - be * be) * p1
                      - 2 * (k + al - 1) * (k + be - 1) * s * p0) / (2 * k * (k + al + be) * (s - 2))
    return p1


def _factor(k, n, al, x):
    """((1-x)/2)^k times the normalised Jacobi polynomial P_n^(al,0), and its derivative."""
    h, nrm = (1 - x) / 2, np.sqrt(np.longdouble(2 * n + al + 1) / 2)
    P = _jacobi(n, al, 0, x) * nrm
    dP = (np.longdouble(n + al + 1) / 2 * _jacobi(n - 1, al + 1, 1, x) * nrm) if n else np.zeros_like(x)
    g = h ** k * P
    return g, (h ** k * dP - (np.longdouble(k) / 2 * h ** (k - 1) * P if k else 0))


def _basis(t, N, abc):
    """phi [points, modes] and its derivatives along a, b, c [3, points, modes]."""
    a, b, c = (np.asarray(x, dtype=np.longdouble) for x in abc)
    ml = _modes(t, N)
    phi, d = np.empty((a.size, len(ml)), np.longdouble), np.empty((3, a.size, len(ml)), np.longdouble)
    for i, (p, q, r) in enumerate(ml):
        fa, da = _factor(0, p, 0, a)
        fb, db = _factor(p, q, 2 * p + 1, b) if t in (PRISM, TET) else _factor(0, q, 0, b)
        kc = {HEX: 0, PRISM: 0, TET: p + q, PYR: max(p, q)}[t]
        fc, dc = _factor(kc, r, 2 * kc + 2 if kc or t in (TET, PYR) else 0, c)
        phi[:, i], d[0, :, i], d[1, :, i], d[2, :, i] = fa * fb * fc, da * fb * fc, fa * db * fc, fa * fb * dc
    return phi, d


def _shape(t, abc):
    """Vertex interpolant at collapsed points: N [points, vertices] and dN/d(a, b, c) [3, points, vertices]."""
    a, b, c = (np.asarray(x, dtype=np.longdouble) for x in abc)
    one = np.ones_like(a)

    def lin(x, s):
        return (1 + s * x) / 2, s * one / 2
    cols = []
    for v in VERTS[t]:
        if t in (HEX, PYR) and not (t == PYR and v[2] == 1):
            f = [lin(x, s) for x, s in zip((a, b, c), v)]
        elif t == PYR:
            f = [(one, 0 * one), (one, 0 * one), lin(c, 1)]
        elif t == PRISM:
            if v[1] == 1:
                f = [(one, 0 * one), lin(b, 1), lin(c, v[2])]
            else:
                f = [lin(a, v[0]), lin(b, -1), lin(c, v[2])]
        else:
            if v[2] == 1:
                f = [(one, 0 * one), (one, 0 * one), lin(c, 1)]
            elif v[1] == 1:
                f = [(one, 0 * one), lin(b, 1), lin(c, -1)]
            else:
                f = [lin(a, v[0]), lin(b, -1), lin(c, -1)]
        cols.append((f[0][0] * f[1][0] * f[2][0], f[0][1] * f[1][0] * f[2][0], f[0][0] * f[1][1] * f[2][0],
                     f[0][0] * f[1][0] * f[2][1]))
    x = [np.stack([col[i] for col in cols], axis=1) for i in range(4)]
    return x[0], np.stack(x[1:])


def _grid(n):
    x, w = _gauss(n)
    g = [y.ravel() for y in np.meshgrid(x, x, x, indexing="ij")]
    return g, np.einsum("i,j,k->ijk", w, w, w).ravel()


def _face_points(t, lf, n):
    """Collapsed coordinates of a local face's n^2 points and the weights of its rule."""
    fixed, end, _ = FACES[t][lf]
    x, w = _gauss(n)
    u, v = (y.ravel() for y in np.meshgrid(x, x, indexing="ij"))
    other = [u, v]
    abc = [np.full(n * n, np.longdouble(end)) if d == fixed else other.pop(0) for d in range(3)]
    return abc, np.outer(w, w).ravel()


def _collapse(t, xi):
    x, y, z = xi.T
    if t == HEX:
        return x, y, z
    if t == PRISM:
        return 2 * (1 + x) / (1 - y) - 1, y, z
    if t == PYR:
        return 2 * (1 + x) / (1 - z) - 1, 2 * (1 + y) / (1 - z) - 1, z
    return 2 * (1 + x) / (-y - z) - 1, 2 * (1 + y) / (1 - z) - 1, z


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _t(x):
    return torch.tensor(np.asarray(x, dtype=np.float64), dtype=torch.float64, device=_dev())


@functools.lru_cache(maxsize=None)
def _volume_ops(t, N):
    """phi, d phi / d(a, b, c), the rule's weights, the vertex interpolant and its derivatives at the volume points."""
    abc, w = _grid(N + 1)
    phi, d = _basis(t, N, abc)
    s, ds = _shape(t, abc)
    return _t(phi), _t(d), _t(w), _t(s), _t(ds)


# --------------------------------------------------------------------------- inputs

def _flow(x, seed):
    """Perturbed Taylor-Green vortex at points x [..., 3]: conservative variables [..., 5]."""
    X, Y, Z = x[..., 0], x[..., 1], x[..., 2]
    p0 = 1.0 / (GAMMA * MACH * MACH)
    prim = [torch.ones_like(X), torch.sin(X) * torch.cos(Y) * torch.cos(Z), -torch.cos(X) * torch.sin(Y) * torch.cos(Z),
            torch.zeros_like(X), p0 + (torch.cos(2 * X) + torch.cos(2 * Y)) * (torch.cos(2 * Z) + 2) / 16]
    ab = np.random.Generator(np.random.PCG64([3, seed])).uniform(-1, 1, size=(5, 4, 3, 2))
    for v in range(5):
        d = torch.zeros_like(X)
        for k in range(4):
            for ax in range(3):
                d = d + float(ab[v, k, ax, 0]) * torch.sin((k + 1) * x[..., ax]) \
                    + float(ab[v, k, ax, 1]) * torch.cos((k + 1) * x[..., ax])
        prim[v] = prim[v] + 0.05 * (p0 if v == 4 else 1.0) * d / float(np.abs(ab[v]).sum())
    r, u, v, w, p = prim
    return torch.stack([r, r * u, r * v, r * w, p / (GAMMA - 1) + 0.5 * r * (u * u + v * v + w * w)], dim=-1)


def _blocks(box):
    """Per type: element indices and vertex ids."""
    return {t: (np.nonzero(box.etype == t)[0], box.padded[box.etype == t][:, :len(VERTS[t])])
            for t in range(4) if (box.etype == t).any()}


def _scatter(box, N, per_type):
    """Per-type blocks [elements, 5, modes] -> the caller's layout (element blocks concatenated)."""
    nM = np.array([len(_modes(t, N)) for t in range(4)])[box.etype]
    off = np.concatenate([[0], np.cumsum(5 * nM)])
    out = torch.empty(int(off[-1]), dtype=torch.float64, device=_dev())
    for t, (e, _) in _blocks(box).items():
        k = 5 * len(_modes(t, N))
        idx = torch.as_tensor(off[e], device=_dev())[:, None] + torch.arange(k, device=_dev())
        out[idx.reshape(-1)] = per_type[t].reshape(-1)
    return out


def _gather(box, N, flat):
    nM = np.array([len(_modes(t, N)) for t in range(4)])[box.etype]
    off = np.concatenate([[0], np.cumsum(5 * nM)])
    out = {}
    for t, (e, _) in _blocks(box).items():
        k = 5 * len(_modes(t, N))
        idx = torch.as_tensor(off[e], device=_dev())[:, None] + torch.arange(k, device=_dev())
        out[t] = flat[idx.reshape(-1)].reshape(len(e), 5, k // 5)
    return out


def _state(box, N, seed):
    """Modal state of the flow, caller's layout (the reference element's projection)."""
    out = {}
    for t, (e, v) in _blocks(box).items():
        phi, _, w, s, _ = _volume_ops(t, N)
        x = torch.einsum("qv,evd->eqd", s, _t(box.xyz[v]))
        unit = torch.einsum("lqv,vd->qld", _volume_ops(t, N)[4], _t(VERTS[t]))
        wj = w * torch.linalg.det(unit).abs()
        mass = torch.einsum("qi,q,qi->i", phi, wj, phi)
        out[t] = torch.einsum("eqv,q,qi->evi", _flow(x, seed), wj, phi) / mass
    return _scatter(box, N, out)


def _inputs(case, seed):
    """(instances, state, cotangent or None): what prepare() and exact() share."""
    inst = _instances(case)
    Q = torch.cat([_state(b, N, seed + 101 * i) for i, (b, N) in enumerate(inst)])
    bar = None
    if case["op"] in ("rhs_vjp", "rk_vjp"):
        bar = _t(np.random.Generator(np.random.PCG64([5, seed])).uniform(-1, 1, size=Q.numel()))
    return inst, Q, bar


# --------------------------------------------------------------------------- what is timed

def prepare(case, seed):
    inst, Q, bar = _inputs(case, seed)
    box, N = inst[0]
    op = case["op"]
    if op == "batch":
        mesh = dg.Batch([b for b, _ in inst], [n for _, n in inst], flux=case["flux"], gamma=GAMMA)
    elif op == "moving":
        mesh = dg.MovingMesh(box, N, box.velocity(), gamma=GAMMA)
    else:
        mesh = dg.Mesh(box, N, flux=case["flux"], gamma=GAMMA, geometry="vertex" if case.get("perturb") else "affine")
    if case.get("form"):
        mesh.set_volume_form(case["form"])
    if case.get("physics") == "ns":
        mesh.set_physics("navier_stokes", MU, PRANDTL)
    state = dict(case=case, mesh=mesh, Q=Q, S=mesh.empty(), K=mesh.empty(), out=torch.empty_like(Q), dt=_case_dt(case))
    if bar is not None:
        state["bar"] = mesh.set_state(bar)
    return state


def run(state):
    case, mesh, S, K, out = state["case"], state["mesh"], state["S"], state["K"], state["out"]
    op = case["op"]
    mesh.set_state(state["Q"], S)
    if op == "rhs":
        mesh.rhs(S, K)
        return mesh.get_state(K, out)
    if op == "rhs_vjp":
        mesh.rhs_vjp(S, state["bar"], K)
        return mesh.get_state(K, out)
    if op == "rk_vjp":
        mesh.rk_vjp(S, state["dt"], case["steps"], case["every"], state["bar"], K)
        return mesh.get_state(K, out)
    if op == "moving":
        mesh.set_time(0.0)
    mesh.rk_step(S, K, state["dt"], case["steps"])
    return mesh.get_state(S, out)


def _counts(m, kind):
    """Elements per type of a box (the expected numbers of the random kinds)."""
    c = m ** 3
    if kind == "hex":
        return {HEX: c}
    if kind == "kuhn":
        return {TET: 6 * c}
    mixed = {HEX: 0.25, PRISM: 2 * 0.5, PYR: 6 * 0.25}
    if kind == "mixed":
        return {t: f * c for t, f in mixed.items()}
    w, s = max(1, m // 4) * m * m, 2 * m * m
    rest = c - w - s
    out = {t: f * rest for t, f in mixed.items()}
    out[PYR] += 5 * s
    out[TET] = 6 * w + 2 * s
    return out


def work(case):
    """Bytes: the state read and the result written (and the cotangent, and a curved or moving mesh's vertices).
    Flops: the sum-factorised operators, fluxes and updates of every residual; the adjoint twice its forward."""
    sizes = [tuple(int(x) for x in s.split(":")) + ("mixed",) for s in case["sizes"].split(",")] \
        if case["op"] == "batch" else [(case["m"], case["N"], case["kind"])]
    dof, flops = 0.0, 0.0
    ns = case.get("physics") == "ns"
    for m, N, kind in sizes:
        n = N + 1
        for t, cnt in _counts(m, kind).items():
            nM, nf = len(_modes(t, N)), len(FACES[t])
            cols = len({(p, q) for p, q, _ in _modes(t, N)})
            transform = 0 if t == HEX else n * nM + cols * n * n + n ** 4
            lin = 2 * transform + 3 * n ** 4 + 2 * nf * n ** 3
            if ns:       # three lifted gradients: derivative, lifting, projection and back, traces
                lin += 3 * (n ** 4 + 2 * transform + 2 * nf * n ** 3)
            per = 10.0 * lin + n ** 3 * (61 + (180 if ns else 0)) + 0.5 * nf * n * n * (88 + (240 if ns else 0)) + 35 * nM
            if case.get("perturb") and t in (PRISM, PYR):
                per += 10.0 * nM * nM
            flops += cnt * per
            dof += cnt * 5 * nM
    stages = 5 * case["steps"] if "steps" in case else 1
    factor = 3 if case["op"] in ("rhs_vjp", "rk_vjp") else 1
    return {"bytes": 8.0 * dof * (3 if factor == 3 else 2), "flops": flops * stages * factor}


# --------------------------------------------------------------------------- the same in plain torch

LSERK_A = [0.0, -567301805773.0 / 1357537059087.0, -2404267990393.0 / 2016746695238.0,
           -3550918686646.0 / 2091501179385.0, -1275806237668.0 / 842570457699.0]
LSERK_B = [1432997174477.0 / 9575080441755.0, 5161836677717.0 / 13612068292357.0, 1720146321549.0 / 2090206949498.0,
           3134564353537.0 / 4481467310338.0, 2277821191437.0 / 14882151754819.0]
LSERK_C = [0.0, 1432997174477.0 / 9575080441755.0, 2526269341429.0 / 6820363183857.0, 2006345519317.0 / 3224310063776.0,
           2802321613138.0 / 2924317926251.0]


class Reference:
    """Dense-operator DG residual on one box (64 bits, torch)."""

    def __init__(self, box, N, case):
        self.box, self.N, self.n, self.case = box, N, N + 1, case
        self.blocks = _blocks(box)
        self.pos = np.zeros(len(box.etype), dtype=np.int64)
        for e, _ in self.blocks.values():
            self.pos[e] = np.arange(len(e))
        self.faces = self._match()
        self.affine = not case.get("perturb")
        self.vel = box.velocity() if case["op"] == "moving" else None
        self.geometry(0.0)

    def _match(self):
        """Faces grouped by (types, local faces, vertex correspondence): owner and neighbour indices, trace operators."""
        box, keys, rec = self.box, [], []
        for t, (e, v) in self.blocks.items():
            for lf, (_, _, fv) in enumerate(FACES[t]):
                ids = box.pid[v[:, fv]]
                keys.append(np.pad(np.sort(ids, axis=1), ((0, 0), (0, 4 - len(fv))), constant_values=-1))
                rec.append(np.stack([e, np.full(len(e), t), np.full(len(e), lf)], axis=1))
                ids = np.pad(ids, ((0, 0), (0, 4 - len(fv))), constant_values=-1)
                rec[-1] = np.concatenate([rec[-1], ids], axis=1)
        keys, rec = np.concatenate(keys), np.concatenate(rec)
        inv = np.unique(keys, axis=0, return_inverse=True)[1].reshape(-1)
        order = np.lexsort((rec[:, 0], inv))
        own, nb = rec[order[0::2]], rec[order[1::2]]
        perm = np.argmax(own[:, 3:, None] == nb[:, None, 3:], axis=2)       # neighbour's vertex of each owner vertex
        label = np.concatenate([own[:, 1:3], nb[:, 1:3], perm], axis=1)
        groups, which = np.unique(label, axis=0, return_inverse=True)
        out = []
        for g, lab in enumerate(groups):
            sel = np.nonzero(which.reshape(-1) == g)[0]
            t0, l0, t1, l1 = (int(x) for x in lab[:4])
            fv0, fv1 = FACES[t0][l0][2], FACES[t1][l1][2]
            abc, w = _face_points(t0, l0, self.n)
            phi0 = _basis(t0, self.N, abc)[0]
            s, ds = _shape(t0, abc)
            xi = sum(s[:, [fv0[k]]] * np.array(VERTS[t1][fv1[lab[4 + k]]], dtype=np.longdouble) for k in range(len(fv0)))
            phi1 = _basis(t1, self.N, _collapse(t1, xi))[0]
            run = [d for d in range(3) if d != FACES[t0][l0][0]]
            out.append(dict(t0=t0, t1=t1, l0=l0, l1=l1, i0=torch.as_tensor(self.pos[own[sel, 0]], device=_dev()),
                            i1=torch.as_tensor(self.pos[nb[sel, 0]], device=_dev()), phi0=_t(phi0), phi1=_t(phi1), s=_t(s),
                            ds=_t(ds[run]), w=_t(w), fv=list(fv0), idx1=None))
        return out

    def geometry(self, t):
        xyz = self.box.xyz + (t * self.vel if self.vel is not None else 0.0)
        self.X, self.V, self.wJ, self.M, self.xdot, self.minv = {}, {}, {}, {}, {}, {}
        for k, (e, v) in self.blocks.items():
            phi, d, w, s, ds = _volume_ops(k, self.N)
            X = _t(xyz[v])
            o = X[:, :1]
            dx = torch.einsum("lqv,evd->eqdl", ds, X - o)                   # dx_d / da_l
            det = torch.linalg.det(dx)
            self.X[k] = X
            self.wJ[k] = w * det.abs()
            self.M[k] = torch.einsum("eq,eqld->eldq", self.wJ[k], torch.linalg.inv(dx))
            if self.vel is not None:
                self.V[k] = _t(self.vel[v])
                self.xdot[k] = torch.einsum("qv,evd->edq", s, self.V[k])
            self.minv[k] = self.factor(k, self.wJ[k])
        for f in self.faces:
            X = self.X[f["t0"]][f["i0"]]
            o = X[:, :1]
            tan = torch.einsum("lpv,evd->lepd", f["ds"], X - o)
            nvec = torch.linalg.cross(tan[0], tan[1])
            out = X[:, f["fv"]].mean(1) - X.mean(1)
            sign = torch.sign((nvec * out[:, None]).sum(-1))
            f["area"] = (nvec * sign[..., None] * f["w"][None, :, None]).transpose(1, 2)   # [faces, 3, points]
            if self.vel is not None:
                f["xdot"] = torch.einsum("pv,evd->edp", f["s"], self.V[f["t0"]][f["i0"]])

    def factor(self, k, wJ):
        phi = _volume_ops(k, self.N)[0]
        if self.affine:
            return 1.0 / torch.einsum("qi,eq,qi->ei", phi, wJ, phi)
        return torch.linalg.cholesky(torch.einsum("qi,eq,qj->eij", phi, wJ, phi))

    def solve(self, k, r, fac=None):
        fac = self.minv[k] if fac is None else fac
        if self.affine:
            return r * fac[:, None]
        return torch.cholesky_solve(r.transpose(1, 2), fac).transpose(1, 2)

    @staticmethod
    def prim(U):
        u = U[:, 1:4] / U[:, :1]
        p = (GAMMA - 1) * (U[:, 4] - 0.5 * (U[:, 1:4] * u).sum(1))
        return torch.cat([U[:, :1], u, p[:, None]], dim=1)

    @staticmethod
    def flux_dir(U, W, nv):
        """F(U).nv for area vectors nv [., 3, points]."""
        un = (W[:, 1:4] * nv).sum(1, keepdim=True)
        return torch.cat([U[:, :1] * un, U[:, 1:4] * un + W[:, 4:] * nv, (U[:, 4:] + W[:, 4:]) * un], dim=1)

    def riemann(self, UL, UR, f):
        nv = f["area"]
        S = nv.norm(dim=1, keepdim=True)
        nh = nv / S
        WL, WR = self.prim(UL), self.prim(UR)
        F = 0.5 * (self.flux_dir(UL, WL, nv) + self.flux_dir(UR, WR, nv))
        uL, uR = (WL[:, 1:4] * nh).sum(1, keepdim=True), (WR[:, 1:4] * nh).sum(1, keepdim=True)
        if self.case["flux"] == "lf":
            cL, cR = torch.sqrt(GAMMA * WL[:, 4:] / WL[:, :1]), torch.sqrt(GAMMA * WR[:, 4:] / WR[:, :1])
            if self.vel is not None:
                sn = (f["xdot"] * nh).sum(1, keepdim=True)
                F = F - 0.5 * S * sn * (UL + UR)
                uL, uR = uL - sn, uR - sn
            return F - 0.5 * S * torch.maximum(uL.abs() + cL, uR.abs() + cR) * (UR - UL)
        sL, sR = torch.sqrt(UL[:, :1]), torch.sqrt(UR[:, :1])
        HL, HR = (UL[:, 4:] + WL[:, 4:]) / UL[:, :1], (UR[:, 4:] + WR[:, 4:]) / UR[:, :1]
        u, H, rho = (sL * WL[:, 1:4] + sR * WR[:, 1:4]) / (sL + sR), (sL * HL + sR * HR) / (sL + sR), sL * sR
        q2, un = (u * u).sum(1, keepdim=True), (u * nh).sum(1, keepdim=True)
        c = torch.sqrt((GAMMA - 1) * (H - 0.5 * q2))
        dr, dp, du = UR[:, :1] - UL[:, :1], WR[:, 4:] - WL[:, 4:], WR[:, 1:4] - WL[:, 1:4]
        dun = (du * nh).sum(1, keepdim=True)
        a1, a5 = (dp - rho * c * dun) / (2 * c * c), (dp + rho * c * dun) / (2 * c * c)
        l1, l5, l2, a2 = (un - c).abs() * a1, (un + c).abs() * a5, un.abs(), dr - dp / (c * c)
        dt = du - dun * nh
        D = torch.cat([l1 + l5 + l2 * a2, l1 * (u - c * nh) + l5 * (u + c * nh) + l2 * (a2 * u + rho * dt),
                       l1 * (H - c * un) + l5 * (H + c * un) + l2 * (0.5 * a2 * q2 + rho * (u * dt).sum(1, keepdim=True))],
                      dim=1)
        return F - 0.5 * S * D

    @staticmethod
    def viscous(W, g):
        """Viscous fluxes [3][., 5, points] from W and its gradient g [3][., 5, points]."""
        div = g[0][:, 1] + g[1][:, 2] + g[2][:, 3]
        kap = MU * GAMMA / ((GAMMA - 1) * PRANDTL)
        out = []
        for d in range(3):
            tau = [MU * (g[d][:, 1 + i] + g[i][:, 1 + d]) - (2.0 / 3.0 * MU * div if i == d else 0.0) for i in range(3)]
            dT = (g[d][:, 4] - W[:, 4] / W[:, 0] * g[d][:, 0]) / W[:, 0]
            out.append(torch.stack([0 * dT] + tau + [W[:, 1] * tau[0] + W[:, 2] * tau[1] + W[:, 3] * tau[2] + kap * dT],
                                   dim=1))
        return out

    def rate(self, Q):
        """vol - surf per type (the mass matrix not yet applied)."""
        ns, split = self.case.get("physics") == "ns", self.case.get("form") == "split"
        U = {k: q @ _volume_ops(k, self.N)[0].T for k, q in Q.items()}
        trace, hexH = {}, None
        if split and HEX in U:
            hexH, trace = self.split_volume(U[HEX])
        ends = []
        for f in self.faces:
            UL, UR = Q[f["t0"]][f["i0"]] @ f["phi0"].T, Q[f["t1"]][f["i1"]] @ f["phi1"].T
            if split:
                UL, UR = self.split_traces(f, trace, UL, UR)
            ends.append((UL, UR))
        G = None
        if ns:
            G = {}
            W = {k: self.prim(u) for k, u in U.items()}
            r = {k: [-sum((W[k] * self.M[k][:, l, d][:, None]) @ _volume_ops(k, self.N)[1][l] for l in range(3))
                     for d in range(3)] for k in U}
            for f, (UL, UR) in zip(self.faces, ends):
                Ws = 0.5 * (self.prim(UL) + self.prim(UR))
                for d in range(3):
                    v = Ws * f["area"][:, d][:, None]
                    r[f["t0"]][d] = r[f["t0"]][d].index_add(0, f["i0"], v @ f["phi0"])
                    r[f["t1"]][d] = r[f["t1"]][d].index_add(0, f["i1"], -(v @ f["phi1"]))
            G = {k: [self.solve(k, x) for x in r[k]] for k in r}
        out = {}
        for k, u in U.items():
            W = self.prim(u)
            phi, dphi = _volume_ops(k, self.N)[:2]
            if split and k == HEX:
                out[k] = hexH @ phi
                continue
            fv = self.viscous(W, [g @ phi.T for g in G[k]]) if ns else None
            acc = 0.0
            for l in range(3):
                F = self.flux_dir(u, W, self.M[k][:, l])
                if ns:
                    F = F - sum(self.M[k][:, l, d][:, None] * fv[d] for d in range(3))
                if self.vel is not None:
                    F = F - (self.M[k][:, l] * self.xdot[k]).sum(1, keepdim=True) * u
                acc = acc + F @ dphi[l]
            out[k] = acc
        for f, (UL, UR) in zip(self.faces, ends):
            F = self.riemann(UL, UR, f)
            if ns:
                vL = self.viscous(self.prim(UL), [g[f["i0"]] @ f["phi0"].T for g in G[f["t0"]]])
                vR = self.viscous(self.prim(UR), [g[f["i1"]] @ f["phi1"].T for g in G[f["t1"]]])
                F = F - 0.5 * sum((vL[d] + vR[d]) * f["area"][:, d][:, None] for d in range(3))
            out[f["t0"]] = out[f["t0"]].index_add(0, f["i0"], -(F @ f["phi0"]))
            out[f["t1"]] = out[f["t1"]].index_add(0, f["i1"], F @ f["phi1"])
        return out

    # ---- entropy-stable split form on the hexahedra (Chandrashekar's two-point flux)
    @staticmethod
    def _lnmean(a, b):
        f = (a - b) / (a + b)
        u = f * f
        s = 1 + u / 3 + u * u / 5 + u ** 3 / 7 + u ** 4 / 9 + u ** 5 / 11 + u ** 6 / 13 + u ** 7 / 15
        far = u > 1e-2
        one = torch.ones_like(a)
        return torch.where(far, (a - b) / torch.where(far, torch.log(a) - torch.log(b), one), 0.5 * (a + b) / s)

    def _two_point(self, PL, PR, m):
        """F#(L, R).m; P = (rho, u, v, w, beta) along dim 1, m [elements, 3] broadcast."""
        rl, bl = self._lnmean(PL[:, 0], PR[:, 0]), self._lnmean(PL[:, 4], PR[:, 4])
        av = 0.5 * (PL + PR)
        ph = av[:, 0] / (2 * av[:, 4])
        sh = (-1,) + (1,) * (rl.dim() - 1)
        mm = [m[:, d].reshape(sh) for d in range(3)]
        F0 = rl * sum(av[:, 1 + d] * mm[d] for d in range(3))
        Fm = [ph * mm[d] + av[:, 1 + d] * F0 for d in range(3)]
        q2 = 0.5 * ((PL[:, 1:4] ** 2).sum(1) + (PR[:, 1:4] ** 2).sum(1))
        FE = (1 / (2 * (GAMMA - 1) * bl) - 0.5 * q2) * F0 + sum(av[:, 1 + d] * Fm[d] for d in range(3))
        return torch.stack([F0] + Fm + [FE], dim=1)

    def split_volume(self, U):
        n = self.n
        x, w1 = (np.asarray(v, dtype=np.longdouble) for v in _gauss(n))
        L = [np.prod([[(y - x[j]) / (x[i] - x[j]) for j in range(n) if j != i] for i in range(n)], axis=1) for y in (-1, 1)]
        D = np.zeros((n, n), np.longdouble)
        lam = np.array([1 / np.prod([x[i] - x[j] for j in range(n) if j != i]) for i in range(n)])
        for i in range(n):
            for j in range(n):
                if i != j:
                    D[i, j] = lam[j] / lam[i] / (x[i] - x[j])
            D[i, i] = -D[i].sum()
        S, E, w1 = _t(w1[:, None] * D - (w1[:, None] * D).T), _t(np.stack(L)), _t(w1)
        ne = U.shape[0]
        W = self.prim(U)
        beta = 0.5 * W[:, 0] / W[:, 4]
        s = torch.log(W[:, 4]) - GAMMA * torch.log(W[:, 0])
        q2 = (W[:, 1:4] ** 2).sum(1)
        ent = torch.stack([(GAMMA - s) / (GAMMA - 1) - beta * q2, 2 * beta * W[:, 1], 2 * beta * W[:, 2],
                           2 * beta * W[:, 3], -2 * beta], dim=1).reshape(ne, 5, n, n, n)
        P = torch.cat([W[:, :4], beta[:, None]], dim=1).reshape(ne, 5, n, n, n)
        H, trace = torch.zeros(ne, 5, n, n, n, dtype=U.dtype, device=U.device), {}
        X = self.X[HEX]
        A = torch.stack([X[:, 1] - X[:, 0], X[:, 2] - X[:, 0], X[:, 4] - X[:, 0]], dim=2)    # columns: edges
        Jm = (torch.linalg.det(A).abs() / 8)[:, None, None] * 2 * torch.linalg.inv(A)          # J dxi_l/dx_d
        for l in range(3):
            m = Jm[:, l]
            p = P.movedim(2 + l, 2).reshape(ne, 5, n, n * n)
            v = ent.movedim(2 + l, 2).reshape(ne, 5, n, n * n)
            F = self._two_point(p[:, :, :, None], p[:, :, None], m)
            r = -(S[None, None, :, :, None] * F).sum(3)
            for end, sg in ((0, -1.0), (1, 1.0)):
                vt = torch.einsum("i,evix->evx", E[end], v)
                b, uu = -0.5 * vt[:, 4], -vt[:, 1:4] / vt[:, 4:]
                sf = GAMMA - (GAMMA - 1) * (vt[:, 0] + b * (uu ** 2).sum(1))
                rho = torch.exp(-(sf + torch.log(2 * b)) / (GAMMA - 1))
                pr = 0.5 * rho / b
                face = torch.cat([rho[:, None], uu, b[:, None]], dim=1)
                Ff = self._two_point(face[:, :, None], p, m)
                r = r + sg * E[end][None, None, :, None] * (torch.einsum("j,evjx->evx", E[end], Ff)[:, :, None] - Ff)
                trace[(l, end)] = torch.cat([rho[:, None], rho[:, None] * uu,
                                             (pr / (GAMMA - 1) + 0.5 * rho * (uu ** 2).sum(1))[:, None]], dim=1)
            wp = (w1[:, None] * w1[None]).reshape(-1)
            H = H + (r * wp).reshape(ne, 5, n, n, n).movedim(2, 2 + l)
        return H.reshape(ne, 5, n ** 3), trace

    def split_traces(self, f, trace, UL, UR):
        """The hexahedra's face states are the entropy-projected ones."""
        if f["t0"] == HEX:
            fx, end, _ = FACES[HEX][f["l0"]]
            UL = trace[(fx, (end + 1) // 2)][f["i0"]]
        if f["t1"] == HEX:
            fx, end, _ = FACES[HEX][f["l1"]]
            if f["idx1"] is None:
                # the neighbour's own points, reordered to the owner's
                abc = _face_points(HEX, f["l1"], self.n)[0]
                own = _t(_basis(HEX, self.N, abc)[0])
                f["idx1"] = torch.cdist(f["phi1"], own).argmin(1)
            UR = trace[(fx, (end + 1) // 2)][f["i1"]][:, :, f["idx1"]]
        return UL, UR

    def rhs(self, Q):
        return {k: self.solve(k, r) for k, r in self.rate(Q).items()}

    def steps(self, Q, dt, nsteps):
        for _ in range(nsteps):
            K = None
            for a, b in zip(LSERK_A, LSERK_B):
                R = self.rhs(Q)
                K = {k: dt * R[k] if K is None else a * K[k] + dt * R[k] for k in Q}
                Q = {k: Q[k] + b * K[k] for k in Q}
        return Q

    def moving_steps(self, Q, dt, nsteps):
        """M Q is advanced; the stage mass matrices follow the scheme's own integral of dJ/dt."""
        T = 1.0
        vand = np.linalg.inv(np.vander(np.arange(4) * T / 3, 4, increasing=True))
        coef = {k: 0.0 for k in Q}
        for i in range(4):
            self.geometry(i * T / 3)
            for k in Q:
                coef[k] = coef[k] + torch.stack([float(vand[p, i]) * self.wJ[k] for p in range(4)])
        t = 0.0
        for _ in range(nsteps):
            J = {k: sum(coef[k][p] * t ** p for p in range(4)) for k in Q}
            mq = {k: self.weigh(k, Q[k], J[k]) for k in Q}
            K = KJ = None
            for a, b, cs in zip(LSERK_A, LSERK_B, LSERK_C):
                Qs = {k: self.solve(k, mq[k], self.factor(k, J[k])) for k in Q}
                ts = t + cs * dt
                self.geometry(ts)
                R = self.rate(Qs)
                dJ = {k: sum(p * coef[k][p] * ts ** (p - 1) for p in range(1, 4)) for k in Q}
                K = {k: dt * R[k] if K is None else a * K[k] + dt * R[k] for k in Q}
                KJ = {k: dt * dJ[k] if KJ is None else a * KJ[k] + dt * dJ[k] for k in Q}
                mq = {k: mq[k] + b * K[k] for k in Q}
                J = {k: J[k] + b * KJ[k] for k in Q}
            Q = {k: self.solve(k, mq[k], self.factor(k, J[k])) for k in Q}
            t += dt
        return Q

    def weigh(self, k, Q, wJ):
        phi = _volume_ops(k, self.N)[0]
        return ((Q @ phi.T) * wJ[:, None]) @ phi


def exact(case, seed):
    inst, Q, bar = _inputs(case, seed)
    dt, op, out, off = _case_dt(case), case["op"], [], 0
    for box, N in inst:
        ref = Reference(box, N, case)
        n = 5 * int(np.array([len(_modes(t, N)) for t in range(4)])[box.etype].sum())
        q = _gather(box, N, Q[off:off + n])
        if bar is not None:
            g = _gather(box, N, bar[off:off + n])
            q = {k: v.clone().requires_grad_(True) for k, v in q.items()}
            r = ref.rhs(q) if op == "rhs_vjp" else ref.steps(q, dt, case["steps"])
            keys = list(q)
            r = dict(zip(keys, torch.autograd.grad(sum((r[k] * g[k]).sum() for k in keys), [q[k] for k in keys])))
        else:
            with torch.no_grad():
                r = {"rhs": lambda: ref.rhs(q), "moving": lambda: ref.moving_steps(q, dt, case["steps"])}.get(
                    op, lambda: ref.steps(q, dt, case["steps"]))()
        out.append(_scatter(box, N, {k: v.detach() for k, v in r.items()}))
        off += n
    return torch.cat(out)
