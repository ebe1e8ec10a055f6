"""Small unstructured meshes with the tile size left open run on half tiles: the same
results and the same cell order (a raw state) as whole tiles."""
import numpy as np
import pytest

from paper_2007_07347_gb300 import meshes as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16dev"])
@pytest.mark.parametrize("mesh", ["o_mesh", "plate", "hybrid"])
def test_half_tiles_are_neutral(mesh, precision):
    from paper_2007_07347_gb300 import sdugks as S
    if mesh == "o_mesh":
        case = M.cylinder(96, 48, first=0.01, r_far=10.0, shuffle_seed=1)
    elif mesh == "plate":
        case = M.flat_plate(12, 31, 33)
    else:
        m = M.hybrid(31, 23, 31.0, 23.0, jitter=0.15, seed=2)
        case = M.Case("hybrid", m, [(0, M.BC_WALL, (0, 0, 0)), (1, M.BC_WALL, (0, 0, 0)), (3, M.BC_WALL, (0, 0, 0)),
                                    (2, M.BC_MOVING_WALL, (0.1, 0, 0))], tau=0.1, dt=0.2)
    n = case.mesh.n_cells
    rng = np.random.default_rng(3)
    rho, u = 1.0 + 0.005 * rng.standard_normal(n), np.asarray(case.u0) + 0.005 * rng.standard_normal((n, 2))
    half = S.Solver.from_case(case, precision).init(rho, u)
    whole = S.Solver.from_case(case, precision, tile_cells=128).init(rho, u)
    assert half.info()["n_tiles"] > whole.info()["n_tiles"]
    half.step(70)
    whole.step(70)
    for a, b in zip(half.get_state(), whole.get_state()):
        np.testing.assert_array_equal(a, b)
    # the state behind the header (which names the requested tile size) byte for byte
    a, b = half.get_state_raw(), whole.get_state_raw()
    np.testing.assert_array_equal(a[32:], b[32:])
