"""Workloads of the spectral-element Poisson library that its performance is measured on.

Every case is one call (or one short run of calls) a user's program makes through
paper_2108_12188_gb300.sem on a jittered box mesh of hexahedra: applications of the operator,
the gather-scatter's neighbours (inner products, right-hand sides), steps of the conjugate
gradient and whole solves, at the polynomial orders 2..11 the library is used with and from one
small mesh of 64 elements to the 32^3 mesh of 16.8 million points.

A case is a dict: "kind" (ax, dot, rhs, cg, solve, batch), the order "N", the elements per
direction "nx", "ny", "nz", and the kind's options. exact() restates each of them in plain torch
FP64 from the definitions (trilinear map, tensor-product GLL derivatives, QQ^T by index_add).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2108_12188_gb300 import sem

PREC = {"f64": sem.SEM_F64, "f32": sem.SEM_F32, "f64x": sem.SEM_F64X}
VARIANT = {"stored": sem.SEM_AX_STORED, "otf": sem.SEM_AX_OTF, "scale": sem.SEM_AX_OTF_SCALE}
MAX_POINTS = 16_777_216  # local points of the largest case


def listed():
    return [
        # the smallest solve: 64 elements at the paper's order, FP64 CG with the default options, the
        # solution to 1e-10 (latency of launches and reductions)
        {"name": "solve_f64_4cube_n7", "kind": "solve", "N": 7, "nx": 4, "ny": 4, "nz": 4, "mixed": 0, "f64x": False},
        # an ordinary request of a solve service, ragged: FP32 CG with FP64 reliable updates
        {"name": "solve_mixed_n5", "kind": "solve", "N": 5, "nx": 13, "ny": 11, "nz": 12, "mixed": 2, "f64x": False},
        # a dozen small requests of mixed orders that arrived together and are solved in one batch
        {"name": "batch_mixed_12", "kind": "batch", "N": 7, "nx": 4, "ny": 6, "nz": 9, "count": 12},
        # the benchmark's step: FP64 Jacobi-CG iterations on 32^3 elements, N = 7 (16.8M points)
        {"name": "cg_f64_32cube_n7", "kind": "cg", "N": 7, "nx": 32, "ny": 32, "nz": 32, "prec": "f64", "steps": 10},
        # the same iteration with the operator in double-float arithmetic, a ragged mesh
        {"name": "cg_f64x_n7", "kind": "cg", "N": 7, "nx": 24, "ny": 23, "nz": 25, "prec": "f64x", "steps": 10},
        # the paper's A_L with rematerialised factors in FP32, alone (its Figure 1), largest mesh
        {"name": "ax_f32_otf_32cube_n7", "kind": "ax", "N": 7, "nx": 32, "ny": 32, "nz": 32, "prec": "f32",
         "variant": "otf", "assemble": False},
        # assembled FP32 operator with stored factors, ragged, the order sweep's N = 5
        {"name": "ax_f32_stored_n5", "kind": "ax", "N": 5, "nx": 43, "ny": 37, "nz": 41, "prec": "f32",
         "variant": "stored", "assemble": True},
        # assembled FP64 operator on the fly, a medium ragged mesh at N = 9 (odd number of elements)
        {"name": "ax_f64_otf_n9", "kind": "ax", "N": 9, "nx": 13, "ny": 11, "nz": 9, "prec": "f64", "variant": "otf",
         "assemble": True},
        # assembled FP64 operator with stored factors at the lowest order of the sweep, many elements
        {"name": "ax_f64_stored_n3", "kind": "ax", "N": 3, "nx": 61, "ny": 64, "nz": 67, "prec": "f64",
         "variant": "stored", "assemble": True},
        # and at the highest, a small mesh: fewer elements than would fill the GPU twice
        {"name": "ax_f64_stored_n11", "kind": "ax", "N": 11, "nx": 5, "ny": 7, "nz": 6, "prec": "f64",
         "variant": "stored", "assemble": True},
        # the weighted inner product a user's own iteration takes of FP64 vectors
        {"name": "dot_f64_32cube_n7", "kind": "dot", "N": 7, "nx": 32, "ny": 32, "nz": 32, "prec": "f64"},
        # the right-hand side of a new request
        {"name": "rhs_n9", "kind": "rhs", "N": 9, "nx": 20, "ny": 19, "nz": 21, "prec": "f64"},
    ]


def _box(rng, N, points):
    """Elements per direction of a ragged box of about `points` local points at order N."""
    n = max(1.0, points / (N + 1) ** 3) ** (1.0 / 3.0)
    d = [max(1, int(round(n * rng.uniform(0.75, 1.3)))) for _ in range(3)]
    while d[0] * d[1] * d[2] * (N + 1) ** 3 > MAX_POINTS:
        d[d.index(max(d))] -= 1
    return {"N": N, "nx": d[0], "ny": d[1], "nz": d[2]}


def draw(rng):
    kind = rng.choice(["ax", "ax", "ax", "cg", "cg", "solve", "batch", "dot", "rhs"])
    N = rng.choice([2, 3, 4, 5, 5, 6, 7, 7, 7, 8, 9, 9, 10, 11])
    points = math.exp(rng.uniform(math.log(30_000), math.log(MAX_POINTS)))
    if kind == "ax":
        prec = rng.choice(["f64", "f64", "f32", "f32", "f64x"])
        variant = rng.choice(["stored", "otf"] if prec == "f64x" else ["stored", "stored", "otf", "otf", "scale"])
        return {"kind": kind, **_box(rng, N, points), "prec": prec, "variant": variant,
                "assemble": rng.random() < 0.6}
    if kind == "cg":
        return {"kind": kind, **_box(rng, N, points), "prec": rng.choice(["f64", "f64", "f64x"]),
                "steps": rng.randint(5, 10)}
    if kind == "solve":
        mixed = rng.choice([0, 1, 2, 2])
        box = _box(rng, min(N, 9), min(points, 600_000))
        return {"kind": kind, **box, "mixed": mixed, "f64x": mixed == 0 and rng.random() < 0.4}
    if kind == "batch":
        return {"kind": kind, "N": rng.choice([5, 7, 9]), "nx": rng.randint(2, 4), "ny": rng.randint(3, 6),
                "nz": rng.randint(5, 9), "count": rng.randint(3, 16)}
    return {"kind": kind, **_box(rng, N, points), "prec": rng.choice(["f64", "f64", "f32"])}


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------

def _vertices(nx, ny, nz, seed):
    """Vertex coordinates [nv, 3] of the unit cube's box mesh, x fastest, the interior vertices
    moved by U(-0.15 h, 0.15 h) per coordinate."""
    g = np.random.default_rng(seed)
    iz, iy, ix = np.meshgrid(np.arange(nz + 1), np.arange(ny + 1), np.arange(nx + 1), indexing="ij")
    ix, iy, iz = ix.ravel(), iy.ravel(), iz.ravel()
    h = np.array([1.0 / nx, 1.0 / ny, 1.0 / nz])
    xyz = np.stack([ix, iy, iz], axis=1) * h
    inside = (ix > 0) & (ix < nx) & (iy > 0) & (iy < ny) & (iz > 0) & (iz < nz)
    xyz[inside] += g.uniform(-0.15, 0.15, (int(inside.sum()), 3)) * h
    return np.ascontiguousarray(xyz)


def _elements(nx, ny, nz):
    """Vertex ids [E, 8], local vertex a + 2b + 4c, elements x fastest."""
    ez, ey, ex = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    ex, ey, ez = ex.ravel(), ey.ravel(), ez.ravel()
    return np.stack([(ex + a) + (nx + 1) * ((ey + b) + (ny + 1) * (ez + c))
                     for c in range(2) for b in range(2) for a in range(2)], axis=1).astype(np.int64)


def _grid_ids(N, nx, ny, nz):
    """Global GLL-grid id of every local point, int64 [E, Np, Np, Np] in (e, k, j, i) order, on the
    GPU, and the number of grid points."""
    i = torch.arange(N + 1, device="cuda")

    def axis(n):
        return torch.arange(n, device="cuda")[:, None] * N + i  # [n, Np]

    mx, my, mz = nx * N + 1, ny * N + 1, nz * N + 1
    X, Y, Z = axis(nx), axis(ny), axis(nz)
    g = (Z[:, None, None, :, None, None] * my + Y[None, :, None, None, :, None]) * mx + X[None, None, :, None, None, :]
    return g.reshape(nx * ny * nz, N + 1, N + 1, N + 1), mx * my * mz


def _field(case, seed, dtype):
    """One U(-1, 1) value per node of the GLL grid, copied to every local point."""
    ids, n_glob = _grid_ids(case["N"], case["nx"], case["ny"], case["nz"])
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.rand(n_glob, generator=g, device="cuda", dtype=torch.float64) * 2.0 - 1.0
    return u[ids.reshape(-1)].to(dtype)


def _boxes(case):
    """(N, nx, ny, nz) of the problems of a batch: orders and sizes in turn."""
    sizes, orders = [case["nx"], case["ny"], case["nz"]], [case["N"], 5, 9, 7]
    return [(orders[q % 4], sizes[q % 3], sizes[(q + q // 3) % 3], sizes[(q // 2) % 3]) for q in range(case["count"])]


def _mesh(N, nx, ny, nz, seed, flags):
    return sem.Mesh(N, _vertices(nx, ny, nz, seed), _elements(nx, ny, nz), flags=flags)


def _waves(seed):
    g = np.random.default_rng(seed + 77)
    return tuple(int(v) for v in g.integers(1, 4, 3))


def _flags(case):
    if case["kind"] == "ax":
        if case["variant"] == "scale":
            return sem.SEM_MESH_OTF_SCALE
        if case["variant"] == "otf":
            return 0
        return {"f64": sem.SEM_MESH_F64_STORED, "f32": sem.SEM_MESH_F32_STORED,
                "f64x": sem.SEM_MESH_F64X_STORED}[case["prec"]]
    if case["kind"] == "cg" and case["prec"] == "f64x" or case["kind"] == "solve" and case["f64x"]:
        return sem.SEM_MESH_F64_STORED | sem.SEM_MESH_F64X_STORED
    return 0 if case["kind"] in ("dot", "rhs") else sem.SEM_MESH_F64_STORED


class _Cg:
    """A CG handle that is released with the state."""

    def __init__(self, mesh, opts):
        self.mesh, self.handle = mesh, sem.sem_cg_create(mesh.handle, opts)

    def __del__(self):
        sem.sem_cg_destroy(self.handle)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        meshes = [_mesh(*b, seed + q, sem.SEM_MESH_F64_STORED) for q, b in enumerate(_boxes(case))]
        bs = []
        for q, m in enumerate(meshes):
            bs.append(torch.empty(m.n, dtype=torch.float64, device="cuda"))
            sem.sem_rhs_sine(m.handle, *_waves(seed + q), sem.SEM_F64, bs[-1])
        return {"case": case, "meshes": meshes, "bs": bs, "xs": [torch.empty_like(b) for b in bs],
                "opts": sem.sem_cg_default_opts(mixed=2, inner_rtol=0.1)}
    mesh = _mesh(case["N"], case["nx"], case["ny"], case["nz"], seed, _flags(case))
    s = {"case": case, "mesh": mesh}
    dtype = torch.float32 if case.get("prec") == "f32" else torch.float64
    if kind == "ax":
        s["u"] = _field(case, seed, dtype)
        s["w"] = torch.empty_like(s["u"])
    elif kind == "dot":
        s["a"], s["b"] = _field(case, seed, dtype), _field(case, seed + 1, dtype)
        s["a"] += 0.5 * s["b"]  # correlated, as the vectors of an iteration are
        s["result"] = torch.empty(1, dtype=torch.float64, device="cuda")
    elif kind == "rhs":
        s["waves"] = _waves(seed)
        s["rhs"] = torch.empty(mesh.n, dtype=dtype, device="cuda")
    else:
        s["b"] = torch.empty(mesh.n, dtype=torch.float64, device="cuda")
        sem.sem_rhs_sine(mesh.handle, *_waves(seed), sem.SEM_F64, s["b"])
        s["x"] = torch.empty_like(s["b"])
        if kind == "cg":
            s["cg"] = _Cg(mesh, sem.sem_cg_default_opts(f64_arith=int(case["prec"] == "f64x")))
        else:
            s["opts"] = sem.sem_cg_default_opts(mixed=case["mixed"], f64_arith=int(case["f64x"]))
            if case["mixed"] == 2:
                s["opts"].inner_rtol = 0.1
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "ax":
        sem.sem_ax(state["mesh"].handle, VARIANT[case["variant"]], PREC[case["prec"]], state["u"], state["w"],
                   assemble=case["assemble"])
        return state["w"]
    if kind == "dot":
        sem.sem_glsc3(state["mesh"].handle, PREC[case["prec"]], state["a"], state["b"], state["result"])
        return state["result"]
    if kind == "rhs":
        sem.sem_rhs_sine(state["mesh"].handle, *state["waves"], PREC[case["prec"]], state["rhs"])
        return state["rhs"]
    if kind == "cg":
        state["x"].zero_()
        sem.sem_cg_start(state["cg"].handle, state["b"], state["x"])
        sem.sem_cg_iterate(state["cg"].handle, case["steps"])
        return state["x"]
    if kind == "solve":
        state["x"].zero_()
        sem.sem_cg_solve(state["mesh"].handle, state["b"], state["x"], state["opts"])
        return state["x"]
    for x in state["xs"]:
        x.zero_()
    sem.sem_cg_solve_batch(state["meshes"], state["bs"], state["xs"], state["opts"])
    return state["xs"]


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------

def _cg_step(n, N, word):
    """Bytes and flops of one Jacobi-CG iteration with stored factors: six factors and M^-1 read,
    x, r, p read and written, w written and read; the paper's flop count 12 (N + 1) + 25."""
    return 15.0 * word * n, n * (12.0 * (N + 1) + 25.0)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        parts = [work({"kind": "solve", "N": b[0], "nx": b[1], "ny": b[2], "nz": b[3], "mixed": 2, "f64x": False})
                 for b in _boxes(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    N = case["N"]
    E = case["nx"] * case["ny"] * case["nz"]
    n = float(E * (N + 1) ** 3)
    word = 4.0 if case.get("prec") == "f32" else 8.0
    if kind == "ax":
        factors = {"stored": 6.0 * n, "otf": 21.0 * E, "scale": n + 21.0 * E}[case["variant"]]
        return {"bytes": word * (2.0 * n + factors), "flops": n * (12.0 * (N + 1) + 15.0)}
    if kind == "dot":
        return {"bytes": (2.0 * word + 1.0) * n, "flops": 3.0 * n}
    if kind == "rhs":
        return {"bytes": word * n + 8.0 * 24.0 * E, "flops": 60.0 * n}
    if kind == "cg":
        b, f = _cg_step(n, N, 8.0)
        return {"bytes": case["steps"] * b, "flops": case["steps"] * f}
    # a solve to 1e-10 takes about 6.3 N iterations per element along the longest side
    b, f = _cg_step(n, N, 4.0 if case["mixed"] else 8.0)
    its = 6.3 * N * max(case["nx"], case["ny"], case["nz"])
    return {"bytes": its * b, "flops": its * f}


# ---------------------------------------------------------------------------------------------
# the same in plain FP64 torch
# ---------------------------------------------------------------------------------------------

def _gll(N):
    """GLL nodes, weights and D[i, l] = l_l'(x_i) of order N (FP64 tensors on the GPU)."""
    P = np.polynomial.legendre.Legendre.basis(N)
    dP = P.deriv()
    x = np.concatenate([[-1.0], np.sort(dP.roots().real), [1.0]]) if N > 1 else np.array([-1.0, 1.0])
    for _ in range(3):  # Newton on L_N', whose derivative follows from Legendre's equation
        t = x[1:-1]
        x[1:-1] = t - dP(t) * (1 - t * t) / (2 * t * dP(t) - N * (N + 1) * P(t))
    L = P(x)
    w = 2.0 / (N * (N + 1) * L * L)
    d = x[:, None] - x[None, :] + np.eye(N + 1)
    D = L[:, None] / (L[None, :] * d)
    D[np.arange(N + 1), np.arange(N + 1)] = 0.0
    D[0, 0], D[N, N] = -N * (N + 1) / 4.0, N * (N + 1) / 4.0
    return tuple(torch.tensor(v, dtype=torch.float64, device="cuda") for v in (x, w, D))


class _Plain:
    """The assembled operator, weights and diagonal of one mesh from their definitions."""

    def __init__(self, N, nx, ny, nz, seed):
        self.x1, w1, self.D = _gll(N)
        Np = N + 1
        X = torch.tensor(_vertices(nx, ny, nz, seed)[_elements(nx, ny, nz)], device="cuda")  # [E, 8, 3]
        lo, hi = (1 - self.x1) / 2, (1 + self.x1) / 2
        phi = torch.stack([lo, hi])  # [2, Np]
        dphi = torch.stack([torch.full_like(lo, -0.5), torch.full_like(lo, 0.5)])
        X = X.reshape(-1, 2, 2, 2, 3)  # [e, c, b, a, xyz]

        def mapped(fc, fb, fa):
            t = torch.einsum("ecbax,ai->ecbix", X, fa)
            t = torch.einsum("ecbix,bj->ecjix", t, fb)
            return torch.einsum("ecjix,ck->ekjix", t, fc)

        self.xyz = mapped(phi, phi, phi)
        g = [mapped(phi, phi, dphi), mapped(phi, dphi, phi), mapped(dphi, phi, phi)]
        c = [torch.linalg.cross(g[1], g[2]), torch.linalg.cross(g[2], g[0]), torch.linalg.cross(g[0], g[1])]
        det = (g[0] * c[0]).sum(-1)
        del g
        www = w1[:, None, None] * w1[None, :, None] * w1[None, None, :]
        self.B = www * det
        s = www / det
        self.G = [[None] * 3 for _ in range(3)]
        for a in range(3):
            for b in range(a, 3):
                self.G[a][b] = self.G[b][a] = s * (c[a] * c[b]).sum(-1)
        self.ids, self.n_glob = _grid_ids(N, nx, ny, nz)
        self.ids = self.ids.reshape(-1)
        mx, my, mz = nx * N + 1, ny * N + 1, nz * N + 1
        ix, iy, iz = self.ids % mx, self.ids // mx % my, self.ids // (mx * my)
        self.free = ((ix > 0) & (ix < mx - 1) & (iy > 0) & (iy < my - 1) & (iz > 0) & (iz < mz - 1)).double()
        self.c = 1.0 / self.qqt(torch.ones(self.ids.numel(), dtype=torch.float64, device="cuda"))
        self.shape = (nx * ny * nz, Np, Np, Np)

    def qqt(self, u):
        return torch.zeros(self.n_glob, dtype=torch.float64, device="cuda").index_add_(0, self.ids, u)[self.ids]

    def local(self, u):
        D, G = self.D, self.G
        u = u.reshape(self.shape)
        d = [torch.matmul(u, D.T), torch.matmul(D, u), torch.einsum("kl,elji->ekji", D, u)]
        v = [G[a][0] * d[0] + G[a][1] * d[1] + G[a][2] * d[2] for a in range(3)]
        return (torch.matmul(v[0], D) + torch.matmul(D.T, v[1]) + torch.einsum("lk,elji->ekji", D, v[2])).reshape(-1)

    def ax(self, u):
        return self.qqt(self.local(u)) * self.free

    def rhs(self, waves):
        f = math.pi ** 2 * sum(q * q for q in waves) * self.B
        for q, a in zip(waves, range(3)):
            f = f * torch.sin(math.pi * q * self.xyz[..., a])
        return self.qqt(f.reshape(-1)) * self.free

    def minv(self):
        D2, D, G = self.D ** 2, torch.diagonal(self.D), self.G
        d = torch.matmul(G[0][0], D2) + torch.matmul(D2.T, G[1][1]) + torch.einsum("lk,elji->ekji", D2, G[2][2])
        di, dj, dk = D[None, None, :], D[None, :, None], D[:, None, None]
        d = d + 2 * (di * dj * G[0][1] + di * dk * G[0][2] + dj * dk * G[1][2])
        return self.free / self.qqt(d.reshape(-1))

    def dot(self, a, b):
        return (a * b * self.c).sum()

    def cg(self, b, steps=None, rtol=1e-13):
        """`steps` iterations of Jacobi-CG from 0, or as many as rtol takes."""
        m, x, r = self.minv(), torch.zeros_like(b), b.clone()
        z = m * r
        p, rho, bb = z.clone(), self.dot(r, z), self.dot(b, b)
        for k in range(steps or 20_000):
            w = self.ax(p)
            alpha = rho / self.dot(p, w)
            x += alpha * p
            r -= alpha * w
            if steps is None and k % 10 == 9 and bool(self.dot(r, r) <= rtol * rtol * bb):
                break
            z = m * r
            new = self.dot(r, z)
            p = z + (new / rho) * p
            rho = new
        return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for q, b in enumerate(_boxes(case)):
            p = _Plain(*b, seed + q)
            out.append(p.cg(p.rhs(_waves(seed + q))))
        return out
    p = _Plain(case["N"], case["nx"], case["ny"], case["nz"], seed)
    dtype = torch.float32 if case.get("prec") == "f32" else torch.float64
    if kind == "ax":
        u = _field(case, seed, dtype).double()
        return p.ax(u) if case["assemble"] else p.local(u)
    if kind == "dot":
        a, b = _field(case, seed, dtype), _field(case, seed + 1, dtype)
        a += 0.5 * b
        return p.dot(a.double(), b.double()).reshape(1)
    if kind == "rhs":
        return p.rhs(_waves(seed))
    b = p.rhs(_waves(seed))
    return p.cg(b, case["steps"]) if kind == "cg" else p.cg(b)
