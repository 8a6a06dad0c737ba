"""Double-float operator on the fly on meshes of more element groups than the GPU holds at once, where
it takes the block shape with fewer registers, against the FP64 operator.

Tolerances: the double-float parity gate of the operator, 1e-12 relative 2-norm; five CG iterations carry
that error through factors below 10 each, 1e-10."""
import numpy as np
import pytest

from synthetic import BoxMesh

pytestmark = pytest.mark.gpu

# one group more than 152 SMs hold and a ragged last group: (elements, N)
CASES = [((21, 19, 19), 2), ((16, 15, 13), 4), ((9, 9, 8), 8), ((8, 8, 8), 9), ((8, 8, 8), 10), ((6, 6, 5), 11)]


@pytest.mark.parametrize("dims,N", CASES, ids=[f"N{N}" for _, N in CASES])
def test_on_the_fly(dims, N):
    import torch
    from paper_2108_12188_gb300 import build_lib, sem
    build_lib.build()
    sem.load_library()
    m = BoxMesh(*dims, jitter=0.15, seed=N)
    mesh = sem.Mesh(N, m.vert_xyz, m.elem_verts, flags=0)
    u = torch.tensor(np.random.default_rng(N).uniform(-1, 1, mesh.n), device="cuda")
    w, want = torch.empty_like(u), torch.empty_like(u)
    sem.sem_ax(mesh.handle, sem.SEM_AX_OTF, sem.SEM_F64X, u, w, assemble=False)
    sem.sem_ax(mesh.handle, sem.SEM_AX_OTF, sem.SEM_F64, u, want, assemble=False)
    assert float((w - want).norm()) <= 1e-12 * float(want.norm())
    b = torch.empty_like(u)
    sem.sem_rhs_sine(mesh.handle, 1, 2, 1, sem.SEM_F64, b)
    xs = []
    for arith in (0, 1):
        x = torch.zeros_like(b)
        cg = sem.sem_cg_create(mesh.handle, sem.sem_cg_default_opts(variant=sem.SEM_AX_OTF, f64_arith=arith))
        sem.sem_cg_start(cg, b, x)
        sem.sem_cg_iterate(cg, 5)
        torch.cuda.synchronize()
        sem.sem_cg_destroy(cg)
        xs.append(x)
    assert float((xs[1] - xs[0]).norm()) <= 1e-10 * float(xs[0].norm())


# either side of the size where the plain operator at N = 7 moves to the tensor-core kernel
@pytest.mark.parametrize("dims", [(13, 14, 14), (16, 16, 10)], ids=["pairs", "slices"])
def test_stored_at_order_7(dims):
    import torch
    from paper_2108_12188_gb300 import build_lib, sem
    build_lib.build()
    sem.load_library()
    m = BoxMesh(*dims, jitter=0.15, seed=7)
    mesh = sem.Mesh(7, m.vert_xyz, m.elem_verts, flags=sem.SEM_MESH_F64X_STORED)
    u = torch.tensor(np.random.default_rng(7).uniform(-1, 1, mesh.n), device="cuda")
    w, want = torch.empty_like(u), torch.empty_like(u)
    sem.sem_ax(mesh.handle, sem.SEM_AX_STORED, sem.SEM_F64X, u, w, assemble=False)
    sem.sem_ax(mesh.handle, sem.SEM_AX_OTF, sem.SEM_F64, u, want, assemble=False)
    assert float((w - want).norm()) <= 1e-12 * float(want.norm())
    b = torch.empty_like(u)
    sem.sem_rhs_sine(mesh.handle, 1, 2, 1, sem.SEM_F64, b)
    x = torch.zeros_like(b)
    res = sem.sem_cg_solve(mesh.handle, b, x, sem.sem_cg_default_opts(rtol=1e-10, f64_arith=1))
    r = torch.empty_like(b)
    sem.sem_ax(mesh.handle, sem.SEM_AX_OTF, sem.SEM_F64, x, r, assemble=True)
    assert res["status"] == sem.SEM_OK and float((b - r).norm()) <= 2e-10 * float(b.norm())
