"""Tile autotuner and the FP32 engine that the library chooses by itself: its
candidate is timed and can win, and entries timed with other kernels are not
returned."""
import pytest

from paper_2305_05988_gb300 import autotune

torch = pytest.importorskip("torch")


@pytest.fixture
def fake(monkeypatch):
    """Timings in place of a GPU: the library's own choice is the fastest."""
    monkeypatch.setattr(autotune, "_gpu_name", lambda device: "GB300")
    seen = []

    def measure(shape, op_kind, solver, rows, planes, team, iters, dtype=None, device=None):
        seen.append((rows, planes))
        return 1.0 + rows + 0.01 * planes

    monkeypatch.setattr(autotune, "measure", measure)
    return seen


@pytest.mark.parametrize("solver", ["cg", "jacobi"])
def test_own_choice_is_a_candidate(fake, tmp_path, solver):
    e = autotune.tune((128, 128, 128), "laplacian", solver, dtype=torch.float32, path=str(tmp_path / "t.json"))
    assert e["tile_rows"] == 0 and {r for r, _ in fake} == {0, 4, 8, 16}


@pytest.mark.parametrize("shape,solver,dtype,team", [
    ((128, 128, 128), "cg", torch.float64, "grid"), ((128, 128), "cg", torch.float32, "grid"),
    ((128, 128, 128), "bicgstab", torch.float32, "grid"), ((32, 32, 32), "cg", torch.float32, "1")])
def test_rows_elsewhere(fake, tmp_path, shape, solver, dtype, team):
    autotune.tune(shape, "laplacian", solver, team, dtype=dtype, path=str(tmp_path / "t.json"))
    assert {r for r, _ in fake} == ({4, 8, 16} if team == "grid" else {8})


def test_entries_of_other_kernels_are_tuned_again(fake, tmp_path):
    path, shape = str(tmp_path / "t.json"), (64, 64, 64)
    key = autotune.tune_key("GB300", "cg", "laplacian", shape, "f32", "grid")
    autotune.save_cache({key: {"tile_rows": 16, "tile_planes": 8, "ms_per_iter": 0.1}}, path)
    assert autotune.lookup(shape, "laplacian", "cg", dtype=torch.float32, path=path) is None
    assert autotune.tune(shape, "laplacian", "cg", dtype=torch.float32, path=path)["tile_rows"] == 0
    n = len(fake)
    assert autotune.lookup(shape, "laplacian", "cg", dtype=torch.float32, path=path)["tile_rows"] == 0
    assert autotune.tune(shape, "laplacian", "cg", dtype=torch.float32, path=path)["tile_rows"] == 0
    assert len(fake) == n
