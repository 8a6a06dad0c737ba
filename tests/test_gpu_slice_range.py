"""FP64 operator on the tensor cores (orders 3, 5 to 7 and 9 to 11) on elements whose values differ in size: what a
few large values leave of the others, node by node, against long double.

Tolerances. Nodes that share no coordinate plane with a large value see only small ones: FP64 lines in even and odd
parts are within 2 (NP + 2) units of 2^-53 of S = E^T g E |u|, E = |D| + |D reversed|, g_ab = sqrt(G_aa G_bb), and
the factors and sums within 24 more. Elements in fixed point: 1e-14 of their norm."""
import numpy as np
import pytest

from oracle import sem_oracle as so
from synthetic import BoxMesh, local_field

pytestmark = pytest.mark.gpu

L = np.longdouble
ORDERS = [3, 5, 6, 7, 9, 10, 11]


@pytest.fixture(scope="module")
def sem():
    import torch
    from paper_2108_12188_gb300 import build_lib, sem as sem_mod
    build_lib.build()
    sem_mod.load_library()
    torch.cuda.set_device(0)
    return sem_mod


class Exact:
    """The local operator from its definition in long double."""

    def __init__(self, N, mesh, stretch=(1, 1, 1)):
        x = np.sort(np.polynomial.legendre.Legendre.basis(N).deriv().roots().real)
        x = np.concatenate([[-1.0], x, [1.0]]).astype(L)

        def legendre(t):
            p, q = np.ones_like(t), t
            for n in range(1, N):
                p, q = q, ((2 * n + 1) * t * q - n * p) / (n + 1)
            return p, q  # L_(N-1), L_N

        for _ in range(4):  # Newton on L_N', L_N'' from Legendre's equation
            t = x[1:-1]
            p, q = legendre(t)
            d1 = N * (p - t * q) / (1 - t * t)
            x[1:-1] = t - d1 * (1 - t * t) / (2 * t * d1 - N * (N + 1) * q)
        v = legendre(x)[1]
        w = L(2) / (N * (N + 1) * v * v)
        d = x[:, None] - x[None, :] + np.eye(N + 1)
        self.D = v[:, None] / (v[None, :] * d)
        np.fill_diagonal(self.D, 0)
        self.D[0, 0], self.D[N, N] = -L(N * (N + 1)) / 4, L(N * (N + 1)) / 4
        X = (mesh.vert_xyz * stretch)[mesh.elem_verts].astype(L).reshape(-1, 2, 2, 2, 3)
        phi, dphi = np.stack([(1 - x) / 2, (1 + x) / 2]), np.stack([0 * x - L(0.5), 0 * x + L(0.5)])

        def mapped(fc, fb, fa):
            return np.einsum("ecbax,ai,bj,ck->ekjix", X, fa, fb, fc)

        g = [mapped(phi, phi, dphi), mapped(phi, dphi, phi), mapped(dphi, phi, phi)]
        cr = [np.cross(g[1], g[2]), np.cross(g[2], g[0]), np.cross(g[0], g[1])]
        det = (g[0] * cr[0]).sum(-1)
        s = w[:, None, None] * w[None, :, None] * w[None, None, :] / det
        self.G = [[s * (cr[a] * cr[b]).sum(-1) for b in range(3)] for a in range(3)]

    @staticmethod
    def _apply(D, G, u):
        d = [np.einsum("il,ekjl->ekji", D, u), np.einsum("jl,ekli->ekji", D, u), np.einsum("kl,elji->ekji", D, u)]
        v = [sum(G[a][b] * d[b] for b in range(3)) for a in range(3)]
        return (np.einsum("li,ekjl->ekji", D, v[0]) + np.einsum("lj,ekli->ekji", D, v[1])
                + np.einsum("lk,elji->ekji", D, v[2]))

    def ax(self, u):
        return self._apply(self.D, self.G, u.astype(L))

    def size(self, u):
        E = np.abs(self.D) + np.abs(self.D[:, ::-1])
        g = [[np.sqrt(self.G[a][a] * self.G[b][b]) for b in range(3)] for a in range(3)]
        return self._apply(E, g, np.abs(u).astype(L))


def _ax(sem, mesh, u, variant):
    import torch
    ud = torch.tensor(np.ascontiguousarray(u).ravel(), dtype=torch.float64, device="cuda")
    w = torch.full_like(ud, np.nan)
    sem.sem_ax(mesh.handle, variant, sem.SEM_F64, ud, w, assemble=False)
    return w.cpu().numpy().reshape(u.shape)


@pytest.mark.parametrize("variant", ["stored", "otf"])
@pytest.mark.parametrize("N", ORDERS)
def test_few_large_values(sem, N, variant):
    NP = N + 1
    m = BoxMesh(3, 3, 2, jitter=0.15, seed=N)
    mesh = sem.Mesh(N, m.vert_xyz, m.elem_verts, flags=sem.SEM_MESH_F64_STORED if variant == "stored" else 0)
    exact = Exact(N, m)
    u = local_field(mesh.n, seed=N).reshape(-1, NP, NP, NP)
    # a corner, an edge node, an inner node; a plane of values in the last element
    spikes = [(1, 0, 0, 0), (4, 0, N, 1), (9, 1, 2, 2)]
    for s in spikes:
        u[s] = 1e8
    u[17, N] *= 1e8
    want, size = exact.ax(u), exact.size(u)
    v = sem.SEM_AX_STORED if variant == "stored" else sem.SEM_AX_OTF
    got = _ax(sem, mesh, u, v)
    err = np.abs(got - want)
    for e, k, j, i in spikes:
        far = [np.delete(np.arange(NP), q) for q in (k, j, i)]
        at = (e,) + np.ix_(*far)
        assert (err[at] <= (2 * NP + 28) * 2.0 ** -53 * size[at]).all()
    norm = np.sqrt((want ** 2).sum(axis=(1, 2, 3)))
    assert (np.sqrt((err ** 2).sum(axis=(1, 2, 3))) <= 1e-14 * norm).all()


# one thread of a quarter too few, just enough; spikes of all sizes
@pytest.mark.parametrize("N", ORDERS)
def test_on_either_side_of_a_quarter(sem, N):
    NP, P = N + 1, (N + 1) ** 3
    m = BoxMesh(3, 3, 2, jitter=0.15, seed=N + 1)
    mesh = sem.Mesh(N, m.vert_xyz, m.elem_verts, flags=sem.SEM_MESH_F64_STORED)
    exact = Exact(N, m)
    # the pairs of planes, rows and points along i that one thread holds
    hold = (2, 1, 2) if NP <= 8 else (1, 8, 8)
    k, j, i = np.unravel_index(np.arange(P), (NP, NP, NP))
    thread = ((k // hold[0]) * 64 + (j if NP <= 8 else j % 8)) * 64 + (i // 2 if NP <= 8 else i % 8 // 2)
    ids = np.unique(thread)
    few = (len(ids) + 3) // 4
    rng = np.random.default_rng(N)
    u = local_field(mesh.n, seed=N + 7).reshape(-1, P)
    for e in range(u.shape[0]):
        big = rng.choice(ids, few - 1 if e % 2 else few, replace=False)
        one = np.array([np.flatnonzero(thread == t)[0] for t in big])
        u[e] *= 10.0 ** -(1 + e // 2)
        u[e, one] = np.sign(u[e, one])
    u = u.reshape(-1, NP, NP, NP)
    want = exact.ax(u)
    err = np.sqrt(((_ax(sem, mesh, u, sem.SEM_AX_STORED) - want) ** 2).sum(axis=(1, 2, 3)))
    assert (err <= 1e-14 * np.sqrt((want ** 2).sum(axis=(1, 2, 3)))).all()


# values of one size: no further from long double than twice what plain FP64 (the oracle) is, over the mesh; a digit left out
# is 3e-15 and more. Stretched elements: stored factors keep 59 bits of the element's largest only, factors on the fly
# are made from differences of long and short edges.
@pytest.mark.parametrize("stretch", [(1, 1, 1), (10, 1, 1), (1, 30, 1), (1, 1, 30), (1, 1, 100), (1e2, 1, 1)],
                         ids=["1", "r10", "s30", "t30", "t100", "r100"])
@pytest.mark.parametrize("N", ORDERS)
def test_as_exact_as_fp64(sem, N, stretch):
    NP = N + 1
    m = BoxMesh(3, 3, 2, jitter=0.15, seed=N + 2)
    xyz = m.vert_xyz * stretch
    mesh = sem.Mesh(N, xyz, m.elem_verts, flags=sem.SEM_MESH_F64_STORED)
    u = local_field(mesh.n, seed=N + 3).reshape(-1, NP, NP, NP)
    want = Exact(N, m, stretch).ax(u)
    xi, w1 = so.gll_nodes_weights(N)
    G, _ = so.geometric_factors(so.element_vertices(xyz, m.elem_verts), xi, w1)

    def error(w):
        return np.sqrt((((w - want) ** 2).sum() / (want ** 2).sum()).astype(float))

    plain = error(so.ax_local(u, G, so.lagrange_derivative_matrix(xi)))
    for variant in (sem.SEM_AX_STORED, sem.SEM_AX_OTF):
        assert error(_ax(sem, mesh, u, variant)) <= 2 * plain


# b has one value of 1e10 at a vertex: x after two iterations, at the nodes of its elements on none of its planes
@pytest.mark.parametrize("variant", ["stored", "otf"])
@pytest.mark.parametrize("N", [3, 7, 10])
def test_cg(sem, N, variant):
    import torch
    NP = N + 1
    m = BoxMesh(3, 3, 3, jitter=0.15, seed=N)
    mesh = sem.Mesh(N, m.vert_xyz, m.elem_verts, flags=sem.SEM_MESH_F64_STORED if variant == "stored" else 0)
    exact = Exact(N, m)
    glo = sem.sem_mesh_get_glo_num(mesh.handle)
    free = (sem.sem_mesh_get_mask(mesh.handle) == 0).astype(L)
    shape = (-1, NP, NP, NP)

    def dssum(v):
        s = np.zeros(glo.max() + 1, dtype=v.dtype)
        np.add.at(s, glo, v)
        return s[glo]

    c = 1 / dssum(np.ones(mesh.n, dtype=L))
    g = np.random.default_rng(N).uniform(-1, 1, glo.max() + 1)
    vertex = glo[0 + NP ** 3 - 1]  # element 0's last corner: a vertex of eight elements
    g[vertex] = 1e10
    b = g[glo] * free.astype(np.float64)
    minv = torch.empty(mesh.n, dtype=torch.float64, device="cuda")
    sem.sem_jacobi(mesh.handle, sem.SEM_F64, minv)
    minv = minv.cpu().numpy()
    x, r = np.zeros(mesh.n, dtype=L), b.astype(L)
    z = minv * r
    p, rho = z.copy(), (r * z * c).sum()
    for _ in range(2):
        w = dssum(exact.ax(p.reshape(shape)).reshape(-1)) * free
        alpha = rho / (p * w * c).sum()
        x, r = x + alpha * p, r - alpha * w
        z = minv * r
        new = (r * z * c).sum()
        p, rho = z + new / rho * p, new
    bd = torch.tensor(b, device="cuda")
    xd = torch.zeros_like(bd)
    v = sem.SEM_AX_STORED if variant == "stored" else sem.SEM_AX_OTF
    cg = sem.sem_cg_create(mesh.handle, sem.sem_cg_default_opts(variant=v))
    sem.sem_cg_start(cg, bd, xd)
    sem.sem_cg_iterate(cg, 2)
    torch.cuda.synchronize()
    sem.sem_cg_destroy(cg)
    got, x, ids = xd.cpu().numpy().reshape(shape), x.reshape(shape), glo.reshape(shape)
    elems = [e for e in range(ids.shape[0]) if (ids[e] == vertex).any()]
    assert len(elems) == 8
    for e in elems:
        k, j, i = np.argwhere(ids[e] == vertex)[0]
        at = (e,) + np.ix_(*[np.delete(np.arange(1, N), np.flatnonzero(np.arange(1, N) == q)) for q in (k, j, i)])
        assert np.abs(got[at] - x[at]).max() <= 1e-11 * np.abs(x[at]).max()
