"""sdugks_solver_info says what a step launches, also where the tile size was left open."""
import pytest

from paper_2007_07347_gb300 import meshes as M

pytestmark = pytest.mark.gpu

BLOCK = {16: (4, 4), 64: (8, 8), 128: (16, 8), 224: (16, 14), 256: (16, 16)}


def _info(case, precision, **kw):
    from paper_2007_07347_gb300 import sdugks as S
    return S.Solver.from_case(case, precision, **kw).info()


@pytest.mark.parametrize("precision,n,cells,staging", [
    ("fp64", 20, (16,), "loads"), ("fp64", 130, (64, 224), "loads"), ("fp64", 300, (224,), "loads"), ("fp64", 60, (256,), "tma"),
    ("fp32", 100, (128,), "loads"), ("fp32", 256, (224,), "loads"), ("fp32", 100, (128, 224, 256), "tma"),
    ("bf16dev", 300, (128, 224, 256), "loads")])
def test_block_steps(precision, n, cells, staging):
    i = _info(M.cavity(n), precision, staging=staging)
    assert i["march"] == 0 and i["step_cells"] in cells
    bx, by = BLOCK[i["step_cells"]]
    assert i["step_ctas"] == -(-n // bx) * -(-n // by)


def test_marching_steps():
    i = _info(M.cavity(700), "fp32")
    assert i["march"] == 1 and i["step_cells"] == 0
    assert i["step_ctas"] % 12 == 0                        # twelve strips of 60 columns
    assert _info(M.cavity(700), "fp32", staging="tma")["march"] == 0


def test_tile_steps():
    case = M.cylinder(96, 48, first=0.01, r_far=10.0, shuffle_seed=1)
    for kw, most in ((dict(), 64), (dict(tile_cells=128), 128), (dict(tile_cells=100), 100)):
        i = _info(case, "fp32", **kw)
        assert most // 2 < i["step_cells"] <= most and i["step_ctas"] == i["n_tiles"] >= 96 * 48 // most


def test_a_block_asked_for_by_its_size_is_run():
    """tile_cells = 0 marches on a large grid; 256, 224 and 128 are those blocks, so that the autotuner's
    candidates are different launches, with marching among them."""
    from paper_2007_07347_gb300 import sdugks as S
    case = M.cavity(640)
    for cells in (256, 224, 128):
        i = _info(case, "fp32", tile_cells=cells)
        assert i["march"] == 0 and i["step_cells"] == cells
    S.autotune_clear()
    s = S.Solver.tuned(case, "fp32", steps=64)
    assert s.tune["candidates"] == (1 + 3 * 2) * 3 and s.tune["tile_cells"] in (0, 128, 224, 256)
    assert s.info()["march"] == int(s.tune["tile_cells"] == 0)


def test_batch_autotune_without_a_choice_changes_nothing():
    """Only instances with one form: the launch form for others stays one CTA per item, and no step is made.
    With one that walks or not (a symmetry side) it is timed."""
    from paper_2007_07347_gb300 import sdugks as S
    b = S.Batch(64 << 20, "fp32", max_instances=4)
    i = b.add_case(M.cavity(40, Re=100.0))
    b.autotune(4)
    assert b.info()["per_item"] == 1 and b.residual()[i][2] == 0
    mesh = M.cartesian(40, 20, 40.0, 20.0)
    b.add_case(M.Case("mirror", mesh, [(3, M.BC_WALL, (0, 0, 0)), (1, M.BC_WALL, (0, 0, 0)), (0, M.BC_MOVING_WALL, (0.05, 0, 0)),
                                       (2, M.BC_SYMMETRY, (0, 0, 0))], tau=0.05, dt=0.25))
    b.autotune(4)
    assert b.residual()[i][2] == 4 * 10
