"""Weighted inner product <a, b, c> where its fast paths end: lengths that are no multiple of four, zeros,
subnormal and non-finite values, multiplicities that are no power of two.

Tolerance: n 2^-53 times the sum of |a b c|, the bound of adding n rounded products in any order."""
import math

import numpy as np
import pytest

from synthetic import BoxMesh, local_field

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sem():
    import torch
    from paper_2108_12188_gb300 import build_lib, sem as sem_mod
    build_lib.build()
    sem_mod.load_library()
    torch.cuda.set_device(0)
    return sem_mod


def _three_hexes():
    """Three hexahedra around one vertical edge: a hexagon cut into three quads, extruded."""
    ring = [(math.cos(math.pi * q / 3), math.sin(math.pi * q / 3)) for q in range(6)]
    xy = [(0.0, 0.0)] + ring
    xyz = np.array([(x, y, z) for z in (0.0, 1.0) for x, y in xy])
    quads = [(0, 1, 3, 2), (0, 3, 5, 4), (0, 5, 1, 6)]  # (origin, first, last, diagonal) around vertex 0
    ev = []
    for o, a, c, d in quads:
        base = [o, 1 + (a - 1), 1 + (c - 1), 1 + (d - 1)]
        ev.append(base + [v + 7 for v in base])
    return xyz, np.array(ev, dtype=np.int64)


def _dot(sem, mesh, prec, a, b):
    import torch
    dt = torch.float32 if prec == 1 else torch.float64
    r = torch.empty(1, dtype=torch.float64, device="cuda")
    sem.sem_glsc3(mesh.handle, prec, torch.tensor(a, dtype=dt, device="cuda"),
                  torch.tensor(b, dtype=dt, device="cuda"), r)
    return float(r)


@pytest.mark.parametrize("prec", [0, 1], ids=["f64", "f32"])
@pytest.mark.parametrize("kind", ["box-N2", "box-N4", "one-N6", "three-N3"])
def test_dot(sem, kind, prec):
    shape, N = kind.split("-N")
    if shape == "three":
        xyz, ev = _three_hexes()
    else:
        m = BoxMesh(*((3, 1, 1) if shape == "box" else (1, 1, 1)), jitter=0.0, seed=1)
        xyz, ev = m.vert_xyz, m.elem_verts
    mesh = sem.Mesh(int(N), xyz, ev, flags=0)
    glo = sem.sem_mesh_get_glo_num(mesh.handle)
    mult = np.bincount(glo)[glo]
    assert (shape == "three") == (3 in mult)
    n = glo.size
    dt = np.float32 if prec == 1 else np.float64
    tiny = 1e-40 if prec == 1 else 1e-310
    a, b = local_field(n, seed=2).astype(dt), local_field(n, seed=3).astype(dt)
    a[1::5] = 0
    b[2::7] = 0
    a[3::11] = tiny
    b[4::13] = -tiny
    terms = a.astype(np.float64) * b.astype(np.float64) / mult
    got = _dot(sem, mesh, prec, a, b)
    assert abs(got - math.fsum(terms)) <= n * 2.0 ** -53 * math.fsum(np.abs(terms))
    a[n // 2], b[n // 2] = np.inf, 1.0
    assert _dot(sem, mesh, prec, a, b) == np.inf
    b[n // 2] = np.nan
    assert math.isnan(_dot(sem, mesh, prec, a, b))
