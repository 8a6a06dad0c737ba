"""SEM_F64X CG at order 7 on a small mesh: the residual at the start is formed with the operator that the iterations run, also on a
mesh that holds float pairs beside its factors, so both kinds of mesh give the same bits."""
import numpy as np
import pytest

from synthetic import BoxMesh

pytestmark = pytest.mark.gpu


def test_start_runs_the_iterations_operator():
    import torch
    from paper_2108_12188_gb300 import build_lib, sem
    build_lib.build()
    sem.load_library()
    m = BoxMesh(4, 3, 3, jitter=0.15, seed=7)
    xs = []
    for flags in (sem.SEM_MESH_F64_STORED, sem.SEM_MESH_F64X_STORED):
        mesh = sem.Mesh(7, m.vert_xyz, m.elem_verts, flags=flags)
        b = torch.empty(mesh.n, dtype=torch.float64, device="cuda")
        sem.sem_rhs_sine(mesh.handle, 1, 2, 1, sem.SEM_F64, b)
        x = torch.tensor(np.sin(np.arange(mesh.n, dtype=np.float64)), device="cuda")
        sem.sem_dssum(mesh.handle, sem.SEM_F64, x)
        cg = sem.sem_cg_create(mesh.handle, sem.sem_cg_default_opts(f64_arith=1))
        sem.sem_cg_start(cg, b, x)
        sem.sem_cg_iterate(cg, 1)
        torch.cuda.synchronize()
        sem.sem_cg_destroy(cg)
        xs.append(x)
    assert torch.equal(xs[0], xs[1])
