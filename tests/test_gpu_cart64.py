"""FP64 Cartesian step with plain loads (blocks of 16x14, 8x8 and 4x4 cells, by grid size)
against the FP64 oracle: every side rule at the edges of a block and past them."""
import numpy as np
import pytest

import oracle as O
from paper_2007_07347_gb300 import meshes as M

pytestmark = pytest.mark.gpu


def _case(kind, nx, ny):
    mesh = M.cartesian(nx, ny, float(nx), (1.5 if kind == "open" else 1.0) * ny)
    w = float(nx)
    left_right = {"open": [(3, M.BC_FARFIELD, (1.01, 0.05, 0.01)), (1, M.BC_OUTLET, (0, 0, 0))],
                  "mirror": [(3, M.BC_SYMMETRY, (0, 0, 0)), (1, M.BC_WALL, (0, 0, 0))],
                  "channel": [(3, M.BC_PERIODIC, (1, w, 0.0)), (1, M.BC_PERIODIC, (3, -w, 0.0))]}[kind]
    below_above = {"open": [(0, M.BC_FARFIELD, (1.0, 0.05, 0.0)), (2, M.BC_OUTLET, (0, 0, 0))],
                   "mirror": [(0, M.BC_SYMMETRY, (0, 0, 0)), (2, M.BC_MOVING_WALL, (0.05, 0, 0))],
                   "channel": [(0, M.BC_WALL, (0, 0, 0)), (2, M.BC_MOVING_WALL, (0.05, 0, 0))]}[kind]
    return M.Case(kind, mesh, left_right + below_above, tau=0.05, dt=0.25)


# 4x4 blocks: grids below, at and past one block; 8x8: 100 to 150 a side; 16x14: the rest
CASES = [M.cavity(2, Re=50.0), M.cavity(17, Re=100.0), _case("open", 3, 5), _case("open", 37, 41), _case("mirror", 2, 2),
         _case("mirror", 29, 35), _case("channel", 5, 9), _case("channel", 4, 64), M.periodic_box(2, 2),
         M.periodic_box(45, 31), M.cavity(130, Re=400.0), _case("open", 121, 140), M.cavity(240, Re=1000.0),
         _case("mirror", 210, 215), M.periodic_box(230, 200)]


@pytest.mark.parametrize("q", range(len(CASES)))
def test_fp64_blocks_match_oracle(q):
    from paper_2007_07347_gb300 import sdugks as S
    case = CASES[q]
    n = case.mesh.n_cells
    rng = np.random.default_rng(q)
    rho, u = 1.0 + 0.01 * rng.standard_normal(n), 0.02 * rng.standard_normal((n, 2))
    s = S.Solver.from_case(case, "fp64").init(rho, u)
    s.step(60)
    f, W = s.get_state()
    st = O.init(n, rho=rho, u=u)
    O.run(case, st, 60)
    assert np.abs(f - st.f).max() <= 1e-12 * np.abs(st.f).max()
    assert np.abs(W - st.W).max() <= 1e-12 * np.abs(st.W).max()
