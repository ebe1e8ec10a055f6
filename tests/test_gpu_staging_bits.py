"""What the header promises of results under another launch: FP64 to the bit across stagings and
in a diagnostic step, any precision to the bit however a run is cut into calls, FP32 diagnostic
steps to rounding."""
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


@pytest.mark.parametrize("precision,n", [("fp64", 50), ("fp32", 60)])
def test_a_diagnostic_step_is_a_step(precision, n):
    """To the bit in FP64, and in FP32 where all blocks run one code path."""
    S = _S()
    case = M.cavity(n, Re=400.0)
    out = []
    for diag in (False, True):
        s = S.Solver.from_case(case, precision).init(*_state(case, 5))
        s.step(3)
        s.step_forces() if diag else s.step(1)
        out.append(s.get_state())
    for a, b in zip(*out):
        if precision == "fp64":
            np.testing.assert_array_equal(a, b)
        else:
            assert np.abs(a - b).max() <= 2e-7


def test_a_diagnostic_step_of_a_marching_solve():
    """Blocks in the place of marching warps for one step.  A cell's W changes by sums of six fluxes
    of at most 0.05 (the deviations from rest at unit density), each of some eight roundings of 2^-24:
    8 x 6 x 6e-8 x 0.05 = 1.4e-7 at most, and f by as much: 2e-7."""
    S = _S()
    case = M.cavity(511, Re=1000.0)
    out = []
    for diag in (False, True):
        s = S.Solver.from_case(case, "fp32").init(*_state(case, 7))
        assert s.info()["march"] == 1
        s.step(3)
        s.step_forces() if diag else s.step(1)
        out.append(s.get_state())
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= 2e-7


@pytest.mark.parametrize("precision,n", [("fp32", 100), ("fp32", 200), ("fp32", 511), ("bf16dev", 200), ("fp64", 130)])
def test_calls_may_cut_a_run_anywhere(precision, n):
    """One call of 83 steps (graphs of 8, the rest in shorter graphs), calls of other lengths, and
    single launches: where the size was left open, 100^2 and 200^2 run other blocks outside graphs."""
    S = _S()
    case = M.cavity(n, Re=400.0)
    out = []
    for cuts, graph in (([83], 8), ([1] * 5 + [17, 40, 21], 8), ([83], -1)):
        s = S.Solver.from_case(case, precision, graph_steps=graph).init(*_state(case, 9))
        for k in cuts:
            s.step(k)
        out.append(s.get_state())
    for other in out[1:]:
        for a, b in zip(out[0], other):
            np.testing.assert_array_equal(a, b)
