"""The per-point scales of SEM_MESH_OTF_SCALE: FP64 ones are kept only where an FP64 operator reads them, and the variant runs
either way (FP64 parity gate, 1e-12)."""
import numpy as np
import pytest

from synthetic import BoxMesh, local_field

pytestmark = pytest.mark.gpu


# on the tensor cores; the same order with flat elements in FP64; an order in FP64
@pytest.mark.parametrize("N,flat,words", [(7, 1.0, 4), (7, 1e5, 12), (4, 1.0, 12)])
def test_scales_held(N, flat, words):
    import torch
    from paper_2108_12188_gb300 import build_lib, sem
    build_lib.build()
    sem.load_library()
    m = BoxMesh(3, 2, 2, jitter=0.15, seed=N)
    xyz = m.vert_xyz * [1.0, 1.0, flat]
    plain, mesh = (sem.Mesh(N, xyz, m.elem_verts, flags=f) for f in (0, sem.SEM_MESH_OTF_SCALE))
    size = [sem.sem_mesh_get_info(q.handle)["device_bytes"] for q in (plain, mesh)]
    assert size[1] - size[0] == words * mesh.n
    u = torch.tensor(local_field(mesh.n, seed=N), device="cuda")
    w, want = torch.empty_like(u), torch.empty_like(u)
    sem.sem_ax(mesh.handle, sem.SEM_AX_OTF_SCALE, sem.SEM_F64, u, w, assemble=False)
    sem.sem_ax(mesh.handle, sem.SEM_AX_OTF, sem.SEM_F64, u, want, assemble=False)
    assert np.isfinite(float(w.norm())) and float((w - want).norm()) <= 1e-12 * float(want.norm())
