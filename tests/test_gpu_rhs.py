"""Right-hand side of the sine solution over its ways of forming the sines: a thread per row (many
rows), a thread per pair of points (few), every length of the short sums, and elements too large for
them; orders with and without a middle point.

Tolerance: 1e-13 of the largest value, the gate of the parity tests."""
import numpy as np
import pytest

from synthetic import BoxMesh

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sem():
    import torch
    from paper_2108_12188_gb300 import build_lib, sem as sem_mod
    build_lib.build()
    sem_mod.load_library()
    torch.cuda.set_device(0)
    return sem_mod


# 16.7k elements at N = 2 and 2.9k at N = 5 give 512 rows per SM (a thread per row); the box lengths
# spread |a B| = a h / 2 over 1/64 .. 3/2
@pytest.mark.parametrize("dims,N,lengths,waves", [
    ((27, 25, 25), 2, (1.0, 1.0, 1.0), (1, 2, 3)), ((15, 14, 14), 5, (1.0, 2.0, 4.0), (1, 2, 3)),
    ((15, 14, 14), 5, (8.0, 16.0, 1.0), (2, 1, 3)), ((2, 3, 2), 4, (1.0, 1.0, 1.0), (3, 1, 2)),
    ((1, 1, 1), 11, (3.0, 0.1, 1.0), (1, 3, 2)), ((3, 1, 2), 1, (1.0, 1.0, 0.25), (1, 1, 1))],
    ids=["rows-N2", "rows-N5", "rows-N5-coarse", "pairs-N4", "pairs-N11-coarse", "pairs-N1"])
def test_rhs(sem, dims, N, lengths, waves):
    import torch
    m = BoxMesh(*dims, jitter=0.15, seed=N, lengths=lengths)
    mesh = sem.Mesh(N, m.vert_xyz, m.elem_verts, flags=0)
    n = mesh.n
    P = (N + 1) ** 3
    xyz, B = (torch.empty(k * n, dtype=torch.float64, device="cuda") for k in (3, 1))
    sem.sem_mesh_coords(mesh.handle, xyz)
    sem.sem_mesh_geometry(mesh.handle, sem.SEM_F64, None, B)
    x = xyz.cpu().numpy().reshape(3, n)
    f = np.pi ** 2 * sum(q * q for q in waves) * B.cpu().numpy()
    for q, c in zip(waves, x):
        f = f * np.sin(np.pi * q * c)
    glo, mask = sem.sem_mesh_get_glo_num(mesh.handle), sem.sem_mesh_get_mask(mesh.handle)
    want = np.bincount(glo, weights=f)[glo] * (mask == 0)
    assert f.size == m.num_elements * P
    for prec, dt, tol in ((sem.SEM_F64, torch.float64, 1e-13), (sem.SEM_F32, torch.float32, 1.2e-7)):
        rhs = torch.empty(n, dtype=dt, device="cuda")
        sem.sem_rhs_sine(mesh.handle, *waves, prec, rhs)
        np.testing.assert_allclose(rhs.double().cpu().numpy(), want, rtol=0, atol=tol * np.abs(want).max())
