"""Elements so large that their factors overflow FP64 (edges of 1e80: w / det J times c . c): the stored operator gives no
finite number there, as plain FP64 does, and stays right elsewhere (1e-12, the FP64 parity gate)."""
import numpy as np
import pytest

from oracle import sem_oracle as so
from synthetic import BoxMesh, local_field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "f64x"])
@pytest.mark.parametrize("N", [3, 5, 6, 7, 9, 10, 11])
def test_infinite_factors(N, prec):
    import torch
    from paper_2108_12188_gb300 import build_lib, sem
    build_lib.build()
    sem.load_library()
    a, b = BoxMesh(3, 1, 1, jitter=0.15, seed=N), BoxMesh(2, 1, 1, jitter=0.15, seed=N)
    xyz = np.concatenate([a.vert_xyz, 5 + b.vert_xyz * 1e80])
    ev = np.concatenate([a.elem_verts, b.elem_verts + a.num_vertices])
    mesh = sem.Mesh(N, xyz, ev, flags=sem.SEM_MESH_F64_STORED)
    P = (N + 1) ** 3
    u = local_field(5 * P, seed=N)
    want = so.SemProblem(N, a.vert_xyz, a.elem_verts).ax_local(u[:3 * P]).ravel()
    for f in (1.0, 0.0):
        ud = torch.tensor(u * np.repeat([1.0, f], [3 * P, 2 * P]), device="cuda")
        w = torch.zeros_like(ud)
        sem.sem_ax(mesh.handle, sem.SEM_AX_STORED, sem.SEM_F64X if prec == "f64x" else sem.SEM_F64, ud, w, assemble=False)
        w = w.cpu().numpy()
        assert np.linalg.norm(w[:3 * P] - want) <= 1e-12 * np.linalg.norm(want)
        assert not np.isfinite(w[3 * P:]).any()
