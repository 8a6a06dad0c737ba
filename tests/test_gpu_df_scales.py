"""SEM_F64X on fixed-point factors (meshes made for SEM_F64 only): the size of the mesh, 2^-70 of a unit cube and 2^60 of it, is
a power of two on the factors and on w. Tolerance 2^-46, a quarter of the 48 bits that a float pair has."""
import numpy as np
import pytest

from synthetic import BoxMesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [3, 5, 6, 9, 10])
def test_mesh_scale(N):
    import torch
    from paper_2108_12188_gb300 import build_lib, sem
    build_lib.build()
    sem.load_library()
    m = BoxMesh(3, 2, 2, jitter=0.15, seed=N)
    w = []
    for k in (0, -70, 60):
        mesh = sem.Mesh(N, m.vert_xyz * 2.0 ** k, m.elem_verts, flags=sem.SEM_MESH_F64_STORED)
        u = torch.tensor(np.random.default_rng(N).uniform(-1, 1, mesh.n), device="cuda")
        w.append(torch.empty_like(u))
        sem.sem_ax(mesh.handle, sem.SEM_AX_STORED, sem.SEM_F64X, u, w[-1], assemble=False)
        w[-1] *= 2.0 ** -k
    for v in w[1:]:
        assert float((v - w[0]).norm()) <= 2.0 ** -46 * float(w[0].norm())
