"""What the header promises of results under another launch: FP64 to the bit across stagings."""
import numpy as np
import pytest

from paper_2007_07347_gb300 import meshes as M

pytestmark = pytest.mark.gpu


def _S():
    from paper_2007_07347_gb300 import sdugks as S
    return S


def _state(case, seed):
    rng = np.random.default_rng(seed)
    n = case.mesh.n_cells
    return 1.0 + 0.01 * rng.standard_normal(n), 0.02 * rng.standard_normal((n, 2))


def _channel(nx, ny):
    mesh = M.cartesian(nx, ny, float(nx), float(ny))
    bcs = [(3, M.BC_PERIODIC, (1, float(nx), 0.0)), (1, M.BC_PERIODIC, (3, -float(nx), 0.0)),
           (0, M.BC_SYMMETRY, (0, 0, 0)), (2, M.BC_MOVING_WALL, (0.05, 0.0, 0.0))]
    return M.Case("channel", mesh, bcs, tau=0.05, dt=0.25)


# no interior block; one; interior blocks beside ragged edges, wraps and a mirror
@pytest.mark.parametrize("case", [M.cavity(20, Re=100.0), M.cavity(50, Re=400.0), _channel(52, 40), _channel(75, 67),
                                  M.cavity(173, Re=1000.0), M.periodic_box(64, 80)], ids=lambda c: c.name)
def test_fp64_is_the_same_with_tensor_copies(case):
    S = _S()
    out = []
    for staging in ("loads", "tma"):
        s = S.Solver.from_case(case, "fp64", staging=staging).init(*_state(case, 3))
        s.step(70)
        s.step_forces()
        s.step(9)
        out.append(s.get_state())
    for a, b in zip(*out):
        assert np.isfinite(a).all()
        np.testing.assert_array_equal(a, b)
