"""The marching-warp form of the FP32 Cartesian step: strips of 64 staged columns, 60
apart, two columns per lane.  A batch steps every uniform FP32 grid this way, whatever its
size, so the sizes where strips begin, end and wrap are run there; single solves take it on
grids of many waves of blocks."""
import numpy as np
import pytest

import oracle as O
from paper_2007_07347_gb300 import meshes as M

pytestmark = pytest.mark.gpu


def _S():
    from paper_2007_07347_gb300 import sdugks as S
    return S


def _channel(nx, ny):
    mesh = M.cartesian(nx, ny, float(nx), float(ny))
    bcs = [(3, M.BC_PERIODIC, (1, float(nx), 0.0)), (1, M.BC_PERIODIC, (3, -float(nx), 0.0)),
           (0, M.BC_WALL, (0, 0, 0)), (2, M.BC_MOVING_WALL, (0.05, 0.0, 0.0))]
    return M.Case("channel", mesh, bcs, tau=0.05, dt=0.25)


def _open(nx, ny):
    """Far field and outlets on oblong cells, both columns of a lane at a side."""
    mesh = M.cartesian(nx, ny, float(nx), 1.5 * ny)
    bcs = [(3, M.BC_FARFIELD, (1.01, 0.05, 0.01)), (1, M.BC_OUTLET, (0, 0, 0)),
           (0, M.BC_FARFIELD, (1.0, 0.05, 0.0)), (2, M.BC_OUTLET, (0, 0, 0))]
    return M.Case("open", mesh, bcs, tau=0.05, dt=0.25)


def _box(nx, ny):
    return M.periodic_box(nx, ny, tau=0.08, dt=0.25)


def _state(case, seed):
    """Cell-to-cell noise, so that a wrong neighbour shows at once."""
    rng = np.random.default_rng(seed)
    n = case.mesh.n_cells
    return 1.0 + 0.01 * rng.standard_normal(n), 0.02 * rng.standard_normal((n, 2))


# one and two strips with walls (<= 64 columns: one; a last strip of 1 .. 60), odd and even
# columns at the right side, wraps inside one strip and across two, grids of two rows
CASES = [M.cavity(2, Re=100.0), M.cavity(33, Re=100.0), M.cavity(64, Re=400.0), M.cavity(65, Re=400.0),
         M.cavity(124, Re=400.0), M.cavity(125, Re=400.0), _channel(4, 64), _channel(62, 9), _channel(120, 33),
         _channel(53, 12), _open(77, 53), _open(3, 5), _open(129, 2), _box(2, 2), _box(60, 7), _box(126, 33)]


def test_strips_against_oracle():
    """40 steps from noise of 1 % in rho and 0.02 in u: rho within 1e-5 and u within 1e-4
    (2-norm) of the FP64 oracle, the FP32 parity tolerances of the other forms."""
    S = _S()
    b = S.Batch(256 << 20, "fp32", max_instances=len(CASES))
    states = [_state(c, 5 + k) for k, c in enumerate(CASES)]
    ids = [b.add_case(c, r, u) for c, (r, u) in zip(CASES, states)]
    b.step(40)
    for c, (r, u), i in zip(CASES, states, ids):
        rho, v = b.macros(i)
        st = O.init(c.mesh.n_cells, rho=r, u=u)
        O.run(c, st, 40)
        what = (c.name, c.mesh.meta["nx"], c.mesh.meta["ny"])
        assert np.abs(rho - st.W[:, 0]).max() <= 1e-5, what
        assert np.sqrt(np.sum((v - st.u) ** 2) / np.sum(st.u ** 2)) <= 1e-4, what


def test_range_of_rows_is_neutral():
    """The rows per warp follow the batch's total size; an instance's results do not: bit
    for bit the same alone (one row a warp) and beside large grids (many rows a warp)."""
    S = _S()
    out = []
    for others in (0, 6):
        b = S.Batch(2 << 30, "fp32", max_instances=16)
        for _ in range(others):
            b.add_case(M.cavity(700, Re=1000.0))
        ids = [b.add_case(c, *_state(c, 9)) for c in (CASES[5], CASES[8], CASES[10], CASES[15])]
        b.step(30)
        out.append([b.macros(i) for i in ids])
    for (r0, u0), (r1, u1) in zip(*out):
        np.testing.assert_array_equal(r0, r1)
        np.testing.assert_array_equal(u0, u1)


def test_more_instances_than_one_group():
    """A group of instances is one launch (96 records); 100 make two."""
    S = _S()
    cases = [M.cavity(20 + k % 9, Re=100.0 + k) for k in range(100)]
    b = S.Batch(256 << 20, "fp32", max_instances=100)
    ids = [b.add_case(c) for c in cases]
    b.step(150)
    for k in (0, 95, 96, 99):
        st = O.init(cases[k].mesh.n_cells)
        O.run(cases[k], st, 150)
        rho, v = b.macros(ids[k])
        assert np.abs(rho - st.W[:, 0]).max() <= 1e-5
        assert np.sqrt(np.sum((v - st.u) ** 2) / np.sum(st.u ** 2)) <= 1e-4


@pytest.mark.parametrize("n", [460, 511])
def test_single_solve_on_a_large_grid_against_oracle(n):
    S = _S()
    case = M.cavity(n, Re=1000.0)
    rho, u = _state(case, 3)
    s = S.Solver.from_case(case, "fp32").init(rho, u)
    s.step(20)
    r, v = s.macros()
    st = O.init(case.mesh.n_cells, rho=rho, u=u)
    O.run(case, st, 20)
    assert np.abs(r - st.W[:, 0]).max() <= 1e-5
    assert np.sqrt(np.sum((v - st.u) ** 2) / np.sum(st.u ** 2)) <= 1e-4


def test_rest_stays_at_rest_and_divergence_is_reported():
    """Zero flux sums leave W exactly as it was; values past FP32's range reach the FP64
    sums as such and are reported."""
    S = _S()
    case = _box(600, 400)
    s = S.Solver.from_case(case, "fp32").init()
    s.step(10)
    rho, u = s.macros()
    assert np.all(rho == 1.0) and np.all(u == 0.0)
    case = M.periodic_box(600, 400, tau=0.001, dt=40.0)      # forty cells a step: unstable
    s = S.Solver.from_case(case, "fp32").init(*_state(case, 4))
    s.step(200)
    with pytest.raises(S.SdugksError) as e:
        s.residual()
    assert e.value.name == "DIVERGED"
