"""FP64 operator on the tensor cores (stored factors, orders 3, 5 to 7 and 9 to 11): A_L against the oracle
where its integer digits, element scales and shared blocks can go wrong.

Tolerance: the FP64 parity gate, 1e-12 relative 2-norm (per element for the scaled fields). The operator is
linear and every element scales its own input, so a power of two on an element's input must come
back as the same power on its output, bit for bit, as long as fixed point takes the element."""
import numpy as np
import pytest

from oracle import sem_oracle as so
from synthetic import BoxMesh, local_field

pytestmark = pytest.mark.gpu

# (elements, N): one element; a block of eight N = 3 elements with one left over; ragged boxes
CASES = [((1, 1, 1), 3), ((3, 3, 1), 3), ((2, 2, 2), 3), ((5, 3, 2), 3), ((1, 1, 1), 5), ((3, 2, 2), 5),
         ((2, 2, 1), 6), ((1, 1, 1), 7), ((3, 2, 2), 7), ((2, 2, 1), 9), ((1, 1, 1), 10), ((2, 1, 2), 10),
         ((1, 2, 2), 11)]
IDS = [f"{d[0]}x{d[1]}x{d[2]}-N{N}" for d, N in CASES]


@pytest.fixture(scope="module")
def sem():
    import torch
    from paper_2108_12188_gb300 import build_lib, sem as sem_mod
    build_lib.build()
    sem_mod.load_library()
    torch.cuda.set_device(0)
    return sem_mod


def _apply(sem, mesh, u, prec=0):
    import torch
    ud = torch.tensor(np.ascontiguousarray(u).ravel(), dtype=torch.float64, device="cuda")
    w = torch.empty_like(ud)
    sem.sem_ax(mesh.handle, sem.SEM_AX_STORED, prec, ud, w, assemble=False)
    return w.cpu().numpy()


@pytest.mark.parametrize("dims,N", CASES, ids=IDS)
def test_operator(sem, dims, N):
    m = BoxMesh(*dims, jitter=0.15, seed=N)
    prob = so.SemProblem(N, m.vert_xyz, m.elem_verts)
    mesh = sem.Mesh(N, m.vert_xyz, m.elem_verts, flags=sem.SEM_MESH_F64_STORED)
    E = prob.n // (N + 1) ** 3
    u = local_field(prob.n, seed=N)
    spike = np.zeros(prob.n)
    spike[prob.n // 2] = -3.0
    for f in (u, spike, np.zeros(prob.n)):
        want = prob.ax_local(f).ravel()
        got = _apply(sem, mesh, f)
        assert np.linalg.norm(got - want) <= 1e-12 * np.linalg.norm(want)
    got = _apply(sem, mesh, u, sem.SEM_F64X)  # the same factors split for the double-float operator
    want = prob.ax_local(u).ravel()
    assert np.linalg.norm(got - want) <= 1e-12 * np.linalg.norm(want)
    # element scales: 2^-500 .. 2^500 in fixed point, the last element at 2^-1010 in FP64
    s = 2.0 ** np.linspace(-500, 500, E).round()
    if E > 1:
        s[-1] = 2.0 ** -1010
    base = _apply(sem, mesh, u).reshape(E, -1)
    got = _apply(sem, mesh, u.reshape(E, -1) * s[:, None]).reshape(E, -1)
    # (an element in FP64 puts its block's other elements there too)
    exact = np.arange(E) < (E - 1) // 8 * 8 if N == 3 else np.arange(E) < E - 1
    np.testing.assert_array_equal(got[exact], (base * s[:, None])[exact])
    err = np.linalg.norm(got / s[:, None] - base, axis=1) / np.linalg.norm(base, axis=1)
    assert err.max() <= 1e-12


@pytest.mark.parametrize("dims,N", [((3, 3, 1), 3), ((3, 2, 2), 7), ((5, 1, 1), 10)], ids=["N3", "N7", "N10"])
def test_non_finite_values_stay_in_their_element(sem, dims, N):
    m = BoxMesh(*dims, jitter=0.15, seed=N)
    prob = so.SemProblem(N, m.vert_xyz, m.elem_verts)
    mesh = sem.Mesh(N, m.vert_xyz, m.elem_verts, flags=sem.SEM_MESH_F64_STORED)
    P = (N + 1) ** 3
    u = local_field(prob.n, seed=N)
    want = _apply(sem, mesh, u).reshape(-1, P)
    u[2 * P + 5], u[4 * P + P // 2] = np.nan, np.inf
    got = _apply(sem, mesh, u).reshape(-1, P)
    with np.errstate(invalid="ignore"):
        finite = np.isfinite(prob.ax_local(u).ravel()).reshape(-1, P)
    np.testing.assert_array_equal(np.isfinite(got), finite)
    keep = [e for e in range(want.shape[0]) if e not in (2, 4)]
    err = np.linalg.norm(got[keep] - want[keep]) / np.linalg.norm(want[keep])
    assert err <= 1e-12
