"""GPU parity of the rarefied step on uniform Cartesian grids (k_dvm_cart.cu) with the FP64
oracle: odd and even velocity grids, every side as a wall (each of them moving) or periodic,
the smallest grids, shuffled cells, lines of one and of several segments, odd step
counts, and the limit dt = tau of the path with the general path beyond it.

Tolerances, those of the general path's tests: FP64 max |gpu - oracle| / max |oracle| <= 1e-12 for
f and W (sums in another order; f = (phi - b feq) / a with a >= 1/2 at most doubles a rounding); FP32
relative L2 of u <= 1e-4, max |rho - rho_oracle| and max |RT - RT_oracle| <= 1e-5.
"""
import numpy as np
import pytest

import oracle as O
from paper_2007_07347_gb300 import meshes as M

pytestmark = pytest.mark.gpu

WALL, MOVING, PERIODIC = M.BC_WALL, M.BC_MOVING_WALL, M.BC_PERIODIC


def _sides(per_x, per_y, moving, lx, ly):
    """Patches bottom 0, right 1, top 2, left 3; `moving`: the sides that move, both ways."""
    out = []
    for s in range(4):
        if per_x and s in (1, 3):
            out.append((s, PERIODIC, (4 - s, lx if s == 3 else -lx, 0.0)))
        elif per_y and s in (0, 2):
            out.append((s, PERIODIC, (2 - s, 0.0, ly if s == 0 else -ly)))
        elif s in moving:
            out.append((s, MOVING, (0.08 - 0.03 * s, 0.05 * (s - 1), 0)))
        else:
            out.append((s, WALL, (0, 0, 0)))
    return out


# sizes above the line below which small solves stay with the general path
CASES = [  # nx, ny, nv, periodic x, periodic y, moving sides, tau, shuffled, steps
    (5, 4, 116, False, False, (0, 1), 0.2, False, 11),
    (7, 3, 59, True, False, (0, 2), 0.2, False, 20),
    (3, 6, 61, False, True, (1, 3), 0.2, True, 20),
    (4, 4, 66, True, True, (), 0.05, False, 23),
    (2, 2, 260, False, False, (2,), 2.0, False, 10),
    (2, 2, 129, True, True, (), 0.2, False, 12),
    (40, 2, 30, False, False, (3,), 0.2, True, 30),
    (2, 33, 34, False, False, (0, 1, 2, 3), 0.2, False, 30),
    (6, 5, 50, False, False, (2,), 0.5, False, 25),
    (19, 24, 40, False, False, (1, 2), 0.5, True, 15),
    (5, 6, 51, False, False, (2,), 0.01, False, 20),        # dt = tau
    (5, 6, 51, False, False, (2,), 0.009, False, 20),       # dt > tau: the general path
]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nx,ny,nv,per_x,per_y,moving,tau,shuffle,steps", CASES)
def test_rarefied_cartesian_step_matches_oracle(nx, ny, nv, per_x, per_y, moving, tau, shuffle, steps, precision):
    from paper_2007_07347_gb300 import sdugks as S
    lx, ly, vmax, RTw, dt = 0.25 * nx, 0.2 * ny, 2.0, 0.5, 0.01
    m = M.cartesian(nx, ny, lx, ly)
    if shuffle:
        m = M.shuffled(m, 5)
    bcs = _sides(per_x, per_y, moving, lx, ly)
    rng = np.random.default_rng(nx + 100 * ny + nv)
    n = m.n_cells
    rho, RT = 1 + 0.02 * rng.uniform(-1, 1, n), 0.5 + 0.01 * rng.uniform(-1, 1, n)
    u = 0.03 * rng.uniform(-1, 1, (n, 2))
    d = S.Dvm(S.Mesh(m, bcs), nv, vmax, RTw, tau, dt, precision, graph_steps=3).init(rho, u, RT)
    d.step(1)
    d.get_state()                                          # between steps: the state is not touched
    d.step(steps - 1)
    xi, w = O.dvm_grid(nv, vmax)
    st = O.dvm_init(n, xi, w, rho=rho, u=u, RT=RT, RT0=RTw)
    O.dvm_run(m, bcs, st, xi, w, RTw, tau, dt, steps)
    if precision == "fp64":
        f, W = d.get_state()
        assert np.abs(f - st.f).max() <= 1e-12 * np.abs(st.f).max()
        assert np.abs(W - st.W).max() <= 1e-12 * np.abs(st.W).max()
    else:
        r, v, T = d.macros()
        assert np.sqrt(np.sum((v - st.u) ** 2) / np.sum(st.u ** 2)) <= 1e-4
        assert np.abs(r - st.rho).max() <= 1e-5
        assert np.abs(T - st.RT).max() <= 1e-5
