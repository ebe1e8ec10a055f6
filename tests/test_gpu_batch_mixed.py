"""Batches whose instances step by different kernels, and 16-bit batches, while instances come and
go: every instance's state, residual and mass to the bit as alone."""
import numpy as np
import pytest

from paper_2007_07347_gb300 import meshes as M

pytestmark = pytest.mark.gpu


def _S():
    from paper_2007_07347_gb300 import sdugks as S
    return S


def _mirror(nx, ny):
    mesh = M.cartesian(nx, ny, float(nx), float(ny))
    bcs = [(3, M.BC_PERIODIC, (1, float(nx), 0.0)), (1, M.BC_PERIODIC, (3, -float(nx), 0.0)),
           (0, M.BC_MOVING_WALL, (0.05, 0.0, 0.0)), (2, M.BC_SYMMETRY, (0.0, 0.0, 0.0))]
    return M.Case("mirror", mesh, bcs, tau=0.05, dt=0.25)


def _odd(nx, ny):
    return M.periodic_box(nx, ny, tau=0.08, dt=0.25)


def _state(case, seed):
    rng = np.random.default_rng(seed)
    n = case.mesh.n_cells
    return 1.0 + 0.01 * rng.standard_normal(n), 0.02 * rng.standard_normal((n, 2))


# with FP32 the second and fourth are stepped by the other kernel's blocks (a mirror, an odd wrap)
CASES = [M.cavity(48, Re=400.0), _mirror(40, 20), M.cavity(100, Re=1000.0), _odd(33, 24), M.couette(64)]


def _alone(k, precision, cuts):
    """(residuals after each cut, macros) of one case in a batch of its own"""
    b = _S().Batch(64 << 20, precision, max_instances=2)
    i = b.add_case(CASES[k], *_state(CASES[k], k))
    res = []
    for n in cuts:
        b.step(n)
        res.append(b.residual()[i])
    return res, b.macros(i)


@pytest.mark.parametrize("precision", ["fp32", "bf16dev", "fp16dev"])
def test_instances_that_come_and_go(precision):
    b = _S().Batch(256 << 20, precision, max_instances=8)
    ids = {k: b.add_case(CASES[k], *_state(CASES[k], k)) for k in (0, 1, 2)}
    b.step(150)                                    # graph steps and single ones
    res = [b.residual()]
    late = {k: b.add_case(CASES[k], *_state(CASES[k], k)) for k in (3, 4)}
    b.step(131)                                    # (from an odd buffer)
    res.append(b.residual())
    b.remove(ids[2])
    b.step(140)
    res.append(b.residual())
    assert set(res[2]) == {ids[0], ids[1], late[3], late[4]}
    for k in (0, 1):
        want, (rho, u) = _alone(k, precision, (150, 131, 140))
        for r, w in zip(res, want):
            assert r[ids[k]] == w
        np.testing.assert_array_equal(b.macros(ids[k])[0], rho)
        np.testing.assert_array_equal(b.macros(ids[k])[1], u)
    for k in (3, 4):
        want, (rho, u) = _alone(k, precision, (131, 140))
        for r, w in zip(res[1:], want):
            assert r[late[k]] == w
        np.testing.assert_array_equal(b.macros(late[k])[0], rho)
        np.testing.assert_array_equal(b.macros(late[k])[1], u)
