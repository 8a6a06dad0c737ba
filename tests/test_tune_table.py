"""Tuning results: a variant that was neither timed nor set keeps the launcher's own choice of block shape, results belong to
the kernels that were timed, and the table goes through a file unchanged."""
import pytest

from synthetic import BoxMesh


@pytest.fixture(scope="module")
def sem():
    from paper_2108_12188_gb300 import build_lib, sem as sem_mod
    build_lib.build()
    sem_mod.load_library()
    sem_mod.sem_autotune_clear()
    yield sem_mod
    sem_mod.sem_autotune_clear()


def _lines(sem, path):
    sem.sem_autotune_save(path)
    return [ln.split() for ln in path.read_text().splitlines()[1:]]


def test_setting_one_variant_leaves_the_others(sem, tmp_path):
    sem.sem_autotune_clear()
    sem.sem_autotune_set(7, sem.SEM_F32, sem.SEM_AX_STORED, 0)
    for ln in _lines(sem, tmp_path / "t"):
        assert ln[:6] == ["1", "7", "0", "0", "-1", "-1"]


@pytest.mark.gpu
@pytest.mark.parametrize("N,elements", [(3, 8), (7, 1), (9, 1)])
def test_results_belong_to_the_kernels(sem, tmp_path, N, elements):
    sem.sem_autotune_clear()
    m = BoxMesh(3, 2, 2, jitter=0.15, seed=N)
    mesh = sem.Mesh(N, m.vert_xyz, m.elem_verts, flags=sem.SEM_MESH_F64_STORED)
    rep = sem.sem_autotune(mesh.handle, sem.SEM_F64, reps=2)
    # one tensor-core kernel per variant, with the elements per block that it runs with
    assert [(c["variant"], c["shape"], c["elements_per_block"]) for c in rep["candidates"]] == [
        (sem.SEM_AX_STORED, 0, elements), (sem.SEM_AX_OTF, 0, elements)]
    one = _lines(sem, tmp_path / "a")
    assert len(one) == 1 and one[0][3:6] == ["-1", "-1", "-1"]
    # elements so flat that factors on the fly stay in FP64: another kernel, its own result
    flat = sem.Mesh(N, m.vert_xyz * [1.0, 1.0, 1e5], m.elem_verts, flags=sem.SEM_MESH_F64_STORED)
    shapes = {(c["variant"], c["shape"]) for c in sem.sem_autotune(flat.handle, sem.SEM_F64, reps=2)["candidates"]}
    assert (sem.SEM_AX_STORED, 1) not in shapes and (sem.SEM_AX_OTF, 0) in shapes
    both = _lines(sem, tmp_path / "b")
    assert len(both) == 2 and one[0] in both
    sem.sem_autotune_clear()
    sem.sem_autotune_load(tmp_path / "b")
    assert _lines(sem, tmp_path / "c") == both
    # a table of the earlier format holds for every kind of mesh
    head = (tmp_path / "b").read_text().split("\n")[0].split()
    (tmp_path / "d").write_text(f"{head[0]} 2 {head[2]}\n0 {N} 1 0 1 0 1.0 2.0 3.0\n")
    sem.sem_autotune_clear()
    sem.sem_autotune_load(tmp_path / "d")
    assert [ln[:6] for ln in _lines(sem, tmp_path / "e")] == 2 * [["0", str(N), "1", "0", "1", "0"]]
