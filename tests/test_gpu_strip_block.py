"""FP32 batches step by marching warps or, where they hold little work, by blocks: the same
results to the last bit, so that an instance's do not depend on what else is in the batch."""
import numpy as np
import pytest

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
    mesh = M.cartesian(nx, ny, float(nx), 1.5 * ny)
    bcs = [(3, M.BC_FARFIELD, (1.01, 0.05, 0.01)), (1, M.BC_OUTLET, (0, 0, 0)),
           (0, M.BC_FARFIELD, (1.0, 0.05, 0.0)), (2, M.BC_OUTLET, (0, 0, 0))]
    return M.Case("open", mesh, bcs, tau=0.05, dt=0.25)


def _box(nx, ny):
    return M.periodic_box(nx, ny, tau=0.08, dt=0.25)


# the smallest grids, one cell less, as many and one more than a block (16 x 8) and a strip (64, then
# 60 columns) hold, interior blocks, wraps within a block and across several
CASES = [M.cavity(2, Re=100.0), M.cavity(33, Re=100.0), M.cavity(65, Re=400.0), M.cavity(125, Re=400.0), M.couette(64),
         _channel(4, 64), _channel(18, 8), _channel(34, 17), _channel(62, 9), _channel(120, 33), M.couette(40, nx=2), M.cavity(3, Re=50.0),
         _open(15, 7), _open(16, 8), _open(17, 9), _open(77, 53), _channel(130, 2), _box(2, 2), _box(16, 8), _box(18, 10),
         _box(48, 40), _box(126, 33)]


def _state(case, seed):
    rng = np.random.default_rng(seed)
    n = case.mesh.n_cells
    return 1.0 + 0.01 * rng.standard_normal(n), 0.02 * rng.standard_normal((n, 2))


def test_both_forms_give_the_same_bits():
    """Alone the grids go by blocks, beside eight of 700^2 cells they march: steps of a graph, single
    steps, and back and forth as the large ones come and go."""
    S = _S()
    big = M.cavity(700, Re=1000.0)
    out = []
    for company in (False, True):
        b = S.Batch(4 << 30, "fp32", max_instances=len(CASES) + 8)
        ids = [b.add_case(c, *_state(c, k)) for k, c in enumerate(CASES)]
        b.step(131)
        assert b.info()["march"] == 0
        others = [b.add_case(big) for _ in range(8)] if company else []
        b.step(131)
        assert b.info()["march"] == int(company)
        for i in others:
            b.remove(i)
        b.step(12)
        assert b.info()["march"] == 0
        out.append([b.macros(i) for i in ids])
    for c, (r0, u0), (r1, u1) in zip(CASES, *out):
        what = (c.name, c.mesh.meta["nx"], c.mesh.meta["ny"])
        assert np.abs(u0).max() > 0.0 and np.isfinite(u0).all(), what
        np.testing.assert_array_equal(r0, r1, err_msg=str(what))
        np.testing.assert_array_equal(u0, u1, err_msg=str(what))
