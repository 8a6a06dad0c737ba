"""FP64 operator on the tensor cores on meshes of more than two groups of elements per resident block (factor buffer refilled,
buffers reused, a ragged last group), with elements in FP64 among the first: what follows in the same block is right.

Tolerances: the FP64 parity gate, 1e-12 relative 2-norm per element; three CG iterations carry it through factors below
10 each, 1e-10."""
import numpy as np
import pytest

from oracle import sem_oracle as so
from synthetic import BoxMesh, local_field

pytestmark = pytest.mark.gpu

# 152 SMs hold four blocks of eight (N = 3), four to six blocks of one, or one block at 9 and more points per direction
CASES = [(3, (23, 22, 22)), (5, (14, 13, 13)), (6, (13, 12, 11)), (7, (13, 12, 11)), (9, (7, 7, 7)), (10, (7, 7, 7)),
         (11, (7, 7, 7))]
IDS = [f"N{N}" for N, _ in CASES]


@pytest.fixture(scope="module")
def sem():
    import torch
    from paper_2108_12188_gb300 import build_lib, sem as sem_mod
    build_lib.build()
    sem_mod.load_library()
    torch.cuda.set_device(0)
    return sem_mod


@pytest.mark.parametrize("variant", ["stored", "otf"])
@pytest.mark.parametrize("N,dims", CASES, ids=IDS)
def test_operator(sem, N, dims, variant):
    import torch
    m = BoxMesh(*dims, jitter=0.15, seed=N)
    mesh = sem.Mesh(N, m.vert_xyz, m.elem_verts, flags=sem.SEM_MESH_F64_STORED if variant == "stored" else 0)
    xi, w1 = so.gll_nodes_weights(N)
    G, _ = so.geometric_factors(so.element_vertices(m.vert_xyz, m.elem_verts), xi, w1)
    D = so.lagrange_derivative_matrix(xi)
    E, P = m.num_elements, (N + 1) ** 3
    shape = (E, N + 1, N + 1, N + 1)
    v = sem.SEM_AX_STORED if variant == "stored" else sem.SEM_AX_OTF
    u = local_field(E * P, seed=N).reshape(E, P)
    scale = 2.0 ** np.random.default_rng(N).integers(-40, 40, E)
    scale[[1, 70, 151]] = 2.0 ** -1010  # in FP64
    for other in (False, True):
        f = u * (scale[:, None] if other else 1.0)
        if other:
            f[[3, 90, 150, E // 2], 0] *= 1e9  # one large value: in FP64
            f[[20, 100, E - 1], 3] = np.nan
        ud = torch.tensor(f.ravel(), device="cuda")
        w = torch.empty_like(ud)
        sem.sem_ax(mesh.handle, v, sem.SEM_F64, ud, w, assemble=False)
        g = f / (scale[:, None] if other else 1.0)
        got = w.cpu().numpy().reshape(E, P) / (scale[:, None] if other else 1.0)
        keep = np.isfinite(g).all(axis=1)
        want = so.ax_local(np.where(keep[:, None], g, 0.0).reshape(shape), G, D).reshape(E, P)
        err = np.linalg.norm(got - want, axis=1)
        assert (err[keep] <= 1e-12 * np.linalg.norm(want[keep], axis=1)).all()
        assert not np.isfinite(got[~keep]).all(axis=1).any()


@pytest.mark.parametrize("variant", ["stored", "otf"])
@pytest.mark.parametrize("N,dims", CASES, ids=IDS)
def test_cg(sem, N, dims, variant):
    import torch
    m = BoxMesh(*dims, jitter=0.15, seed=N)
    mesh = sem.Mesh(N, m.vert_xyz, m.elem_verts, flags=sem.SEM_MESH_F64_STORED if variant == "stored" else 0)
    v = sem.SEM_AX_STORED if variant == "stored" else sem.SEM_AX_OTF
    b = torch.empty(mesh.n, dtype=torch.float64, device="cuda")
    sem.sem_rhs_sine(mesh.handle, 1, 2, 1, sem.SEM_F64, b)
    # and a value at one vertex that leaves its elements in FP64
    spike = torch.zeros_like(b)
    spike[(N + 1) ** 3 * (dims[0] * (dims[1] + 1) + 2) - 1] = 1e3 * float(b.abs().max())
    sem.sem_dssum(mesh.handle, sem.SEM_F64, spike)
    minv, dot = torch.empty_like(b), torch.empty(1, dtype=torch.float64, device="cuda")
    sem.sem_jacobi(mesh.handle, sem.SEM_F64, minv)

    def inner(p, q):
        sem.sem_glsc3(mesh.handle, sem.SEM_F64, p, q, dot)
        return float(dot)

    for rhs in (b, b + spike):
        x = torch.zeros_like(b)
        cg = sem.sem_cg_create(mesh.handle, sem.sem_cg_default_opts(variant=v))
        sem.sem_cg_start(cg, rhs, x)
        sem.sem_cg_iterate(cg, 3)
        torch.cuda.synchronize()
        sem.sem_cg_destroy(cg)
        y, r, w = torch.zeros_like(b), rhs.clone(), torch.empty_like(b)
        z = minv * r
        p, rho = z.clone(), inner(r, z)
        for _ in range(3):
            sem.sem_ax(mesh.handle, v, sem.SEM_F64, p, w, assemble=True)
            alpha = rho / inner(p, w)
            y, r = y + alpha * p, r - alpha * w
            z = minv * r
            new = inner(r, z)
            p, rho = z + new / rho * p, new
        assert float((x - y).norm()) <= 1e-10 * float(y.norm())
