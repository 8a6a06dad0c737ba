"""Admission of solve requests: a server whose budget is one byte short of the arrays that a request holds refuses it."""
import pytest

from synthetic import BoxMesh

pytestmark = pytest.mark.gpu


# float pairs beside fixed-point factors; FP64 factors beside them (persistent kernel); FP32 on many small elements; FP64
# CG on a large mesh (segments in two layouts); the lowest order; fixed-point factors alone
CASES = [("pairs", 7, (13, 14, 14), "F64X_STORED", dict(mixed=2, f64_arith=1, variant=0, inner_rtol=0.1)),
         ("persistent", 11, (5, 5, 6), "F64_STORED", dict(use_graph=2)),
         ("fp32", 3, (50, 50, 50), None, dict(mixed=1, variant=1)),
         ("fp64", 7, (28, 28, 28), None, dict(variant=1)),
         ("order1", 1, (60, 60, 60), "F64_STORED", dict()),
         ("f64x", 7, (13, 14, 14), "F64_STORED", dict(f64_arith=1))]


@pytest.mark.parametrize("N,dims,flag,opts", [c[1:] for c in CASES], ids=[c[0] for c in CASES])
def test_budget_covers_the_arrays(N, dims, flag, opts):
    import torch
    from paper_2108_12188_gb300 import build_lib, sem
    build_lib.build()
    sem.load_library()
    m = BoxMesh(*dims, jitter=0.1, seed=1)
    o = sem.sem_cg_default_opts(**{"rtol": 1e-2, **opts})
    mesh = sem.Mesh(N, m.vert_xyz, m.elem_verts, flags=getattr(sem, "SEM_MESH_" + flag) if flag else 0)
    b = torch.empty(mesh.n, dtype=torch.float64, device="cuda")
    sem.sem_rhs_sine(mesh.handle, 1, 1, 1, sem.SEM_F64, b)
    sem.sem_cg_solve(mesh.handle, b, torch.zeros_like(b), o)
    # with the Jacobi inverse and what the solver added; b, x and the work vectors
    held = sem.sem_mesh_get_info(mesh.handle)["device_bytes"] + mesh.n * (16 + (40 if o.mixed else 32))
    mesh.close()
    srv = sem.sem_server_create(held - 1, 1)
    try:
        with pytest.raises(sem.SemError, match="more device memory than the budget"):
            sem.sem_server_submit(srv, N, m.vert_xyz, m.elem_verts, (1, 1, 1), o)
    finally:
        sem.sem_server_destroy(srv)
