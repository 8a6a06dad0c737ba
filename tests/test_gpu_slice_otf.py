"""FP64 operator on the tensor cores with factors rebuilt in fixed point (on the fly, with and without the
per-point scale, orders 3, 5 to 7 and 9 to 11) against the oracle, and its choice on distorted meshes.

Tolerances: the FP64 parity gate, 1e-12 relative 2-norm (per element for the scaled fields); five CG
iterations carry it through factors below 10 each, 1e-10."""
import numpy as np
import pytest

from oracle import sem_oracle as so
from synthetic import BoxMesh, local_field

pytestmark = pytest.mark.gpu

# (elements, N): one element; N = 3 blocks of eight elements with some left over; ragged boxes
CASES = [((1, 1, 1), 3), ((3, 3, 1), 3), ((5, 3, 2), 3), ((3, 2, 2), 5), ((2, 2, 1), 6), ((1, 1, 1), 7), ((3, 2, 2), 7),
         ((2, 2, 1), 9), ((2, 1, 2), 10), ((1, 2, 2), 11)]
IDS = [f"{d[0]}x{d[1]}x{d[2]}-N{N}" for d, N in CASES]


@pytest.fixture(scope="module")
def sem():
    import torch
    from paper_2108_12188_gb300 import build_lib, sem as sem_mod
    build_lib.build()
    sem_mod.load_library()
    torch.cuda.set_device(0)
    return sem_mod


def _apply(sem, mesh, u, variant):
    import torch
    ud = torch.tensor(np.ascontiguousarray(u).ravel(), dtype=torch.float64, device="cuda")
    w = torch.full_like(ud, np.nan)
    sem.sem_ax(mesh.handle, variant, sem.SEM_F64, ud, w, assemble=False)
    return w.cpu().numpy()


@pytest.mark.parametrize("dims,N", CASES, ids=IDS)
def test_operator(sem, dims, N):
    m = BoxMesh(*dims, jitter=0.15, seed=N)
    prob = so.SemProblem(N, m.vert_xyz, m.elem_verts)
    mesh = sem.Mesh(N, m.vert_xyz, m.elem_verts, flags=sem.SEM_MESH_OTF_SCALE)
    E = prob.n // (N + 1) ** 3
    u = local_field(prob.n, seed=N)
    # element scales: 2^-500 .. 2^500 in fixed point, the last element at 2^-1010 in FP64
    s = 2.0 ** np.linspace(-500, 500, E).round()
    if E > 1:
        s[-1] = 2.0 ** -1010
    for f in (u, np.zeros(prob.n), (u.reshape(E, -1) * s[:, None]).ravel()):
        want = (prob.ax_local(f.reshape(E, -1) / (s[:, None] if f is not u and f.any() else 1.0)).reshape(E, -1)
                * (s[:, None] if f is not u and f.any() else 1.0))
        for variant in (sem.SEM_AX_OTF, sem.SEM_AX_OTF_SCALE):
            got = _apply(sem, mesh, f, variant).reshape(E, -1)
            # (scaled back, so that the norms of the smallest and largest elements stay in range)
            t = s[:, None] if f is not u and f.any() else 1.0
            d = np.linalg.norm(got / t - want / t, axis=1)
            assert (d <= 1e-12 * np.linalg.norm(want / t, axis=1)).all()


@pytest.mark.parametrize("stretch", [(1, 1, 1), (20, 1, 1), (1, 1e3, 1), (1e-3, 1, 30)])
@pytest.mark.parametrize("N", [3, 7, 9])
def test_stretched(sem, N, stretch):
    m = BoxMesh(2, 2, 2, jitter=0.25, seed=N)
    xyz = m.vert_xyz * np.asarray(stretch, dtype=np.float64)
    prob = so.SemProblem(N, xyz, m.elem_verts)
    mesh = sem.Mesh(N, xyz, m.elem_verts, flags=0)
    u = local_field(prob.n, seed=N)
    want = prob.ax_local(u).ravel()
    assert np.linalg.norm(_apply(sem, mesh, u, sem.SEM_AX_OTF) - want) <= 1e-12 * np.linalg.norm(want)


@pytest.mark.parametrize("N", [3, 6, 7, 10])
def test_cg(sem, N):
    import torch
    m = BoxMesh(4, 3, 3, jitter=0.15, seed=N)
    mesh = sem.Mesh(N, m.vert_xyz, m.elem_verts, flags=sem.SEM_MESH_F64_STORED | sem.SEM_MESH_OTF_SCALE)
    b = torch.empty(mesh.n, dtype=torch.float64, device="cuda")
    sem.sem_rhs_sine(mesh.handle, 1, 2, 1, sem.SEM_F64, b)
    xs = []
    for variant in (sem.SEM_AX_STORED, sem.SEM_AX_OTF, sem.SEM_AX_OTF_SCALE):
        x = torch.zeros_like(b)
        cg = sem.sem_cg_create(mesh.handle, sem.sem_cg_default_opts(variant=variant))
        sem.sem_cg_start(cg, b, x)
        sem.sem_cg_iterate(cg, 5)
        torch.cuda.synchronize()
        sem.sem_cg_destroy(cg)
        xs.append(x)
    for x in xs[1:]:
        assert float((x - xs[0]).norm()) <= 1e-10 * float(xs[0].norm())
