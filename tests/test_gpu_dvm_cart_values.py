"""Values of the rarefied step on uniform grids (k_dvm_cart.cu) that agreement over a few
steps does not show: the Maxwellian's exponential over its whole range, and errors that grow
with the number of steps."""
import numpy as np
import pytest

import oracle as O
from paper_2007_07347_gb300 import meshes as M

pytestmark = pytest.mark.gpu


def _S():
    from paper_2007_07347_gb300 import sdugks as S
    return S


def test_initial_maxwellian_to_rounding():
    """f of the initial state, rho = 1, u = 0, R T = 1/2 on nodes that FP32 holds exactly.  A
    value is the product of two exponentials and a factor.  In units of 2^-23: two exponentials
    of up to 1.5 each; the factor, 1 for its constant and product and 0.5 for its product with an
    exponential; 0.5 for the last product; and log2 e rounded, 1.4e-8 of an exponent of up to 8, 1:
    6 in all."""
    S = _S()
    n, nv = 10, 64
    c = M.micro_cavity(n, 1.0, nv=nv)
    d = S.Dvm.from_case(c, "fp32").init()
    f = d.get_state()[0].reshape(n * n, nv, nv)
    x = -2.0 + (np.arange(nv) + 0.5) * (4.0 / nv)
    g = (4.0 / nv) ** 2 / np.pi * np.exp(-(x[None, :] ** 2 + x[:, None] ** 2))
    assert np.abs(f / g - 1.0).max() <= 6 * 2.0 ** -23


@pytest.mark.parametrize("seed", [5, 15, 17])
def test_a_breakdown_does_not_read_as_finite(seed):
    """One step of two cells from a noisy state leaves cells with R T < 0.  In those between -0.02
    and -0.001 one of the outermost nodes, at +-1.97, has an exponent of at least 139 in base 2 for any
    u: the Maxwellian overflows, and f, the only sign of a breakdown that this solver
    gives, is not finite."""
    S = _S()
    n, nv = 10, 64
    c = M.micro_cavity(n, 1.0, nv=nv)
    rng = np.random.default_rng(seed)
    rho, u = np.exp(rng.uniform(-0.8, 0, n * n)), rng.uniform(-0.1, 0.1, (n * n, 2))
    RT, dt = 0.5 * np.exp(rng.uniform(-2, 0, n * n)), 4 * c.dt
    tau = max(c.tau, dt)
    d = S.Dvm(S.Mesh(c.mesh, c.bcs), nv, 2.0, 0.5, tau, dt, "fp32").init(rho, u, RT)
    d.step(1)
    xi, w = O.dvm_grid(nv, 2.0)
    st = O.dvm_init(n * n, xi, w, rho=rho, u=u, RT=RT, RT0=0.5)
    O.dvm_run(c.mesh, c.bcs, st, xi, w, 0.5, tau, dt, 1)
    cold = np.where((st.RT > -0.02) & (st.RT < -0.001))[0]
    f = d.get_state()[0]
    assert len(cold) and not any(np.isfinite(f[i]).all() for i in cold)


def _in_two_patches(case):
    """The same cavity with half of its bottom side on a patch of its own, which takes it to the
    general kernels."""
    m = case.mesh
    nbr, mid = m.neighbour.copy(), m.points[m.face_pts].mean(1)
    half = (nbr < 0) & (mid[:, 1] < 1e-9) & (mid[:, 0] > 0.5 * m.points[:, 0].max())
    same = next(b for b in case.bcs if b[0] == -1 - nbr[half][0])
    nbr[half] = -1 - 9
    return M.Mesh(m.points, m.face_pts, m.owner, nbr, m.n_cells, m.patches), [*case.bcs, (9, *same[1:])]


@pytest.mark.parametrize("n,nv,kn,steps", [(16, 64, 2.0, 200), (14, 94, 0.5, 120), (12, 33, 4.0, 200)])
def test_fp64_error_does_not_grow(n, nv, kn, steps):
    """FP64 over some hundred steps, against the general kernels, which are within 7.5e-15 (2-norm
    of u) of the same steps in another order of their sums: two such are up to 1.5e-14 apart, and 2e-14
    is allowed.  Constants of walls off by 5e-15, alike in every step, show as 1e-13.  (The oracle
    adds its nv^2 terms one by one and is itself 6e-14 off here.)"""
    S = _S()
    c = M.micro_cavity(n, kn, nv=nv)
    rng = np.random.default_rng(n)
    N = n * n
    rho, RT = 1 + 0.01 * rng.uniform(-1, 1, N), 0.5 + 0.005 * rng.uniform(-1, 1, N)
    u = 0.02 * rng.uniform(-1, 1, (N, 2))
    mesh, bcs = _in_two_patches(c)
    v = []
    for m in (S.Mesh(c.mesh, c.bcs), S.Mesh(mesh, bcs)):
        d = S.Dvm(m, nv, 2.0, 0.5, c.tau, c.dt, "fp64").init(rho, u, RT)
        d.step(steps)
        v.append(d.macros()[1])
        device_bytes = d.sizes()["device_bytes"]
    assert device_bytes > 1.5 * N * nv * nv * 16        # the second is the general path, with its face fluxes
    assert np.sqrt(np.sum((v[0] - v[1]) ** 2) / np.sum(v[1] ** 2)) <= 2e-14


@pytest.mark.parametrize("n,nv,kn,steps,bound", [(40, 100, 1.0, 50, 1.2e-8), (40, 33, 8.0, 100, 2e-8)])
def test_fp32_temperature_noise(n, nv, kn, steps, bound):
    """R T in FP32 against FP64, root mean square.  The general kernels, whose rounding errors
    average over nv^2 nodes, are 0.8e-8 and 1.45e-8 off; a rounding that all nodes of a cell share
    (their Maxwellian's temperature or factor) gave 2.3e-8 and 2.7e-8 plus a drift of 2e-8.  About
    half way between."""
    S = _S()
    c = M.micro_cavity(n, kn, nv=nv)
    rng = np.random.default_rng(3)
    N = n * n
    x = (np.arange(n) + 0.5) / n
    s = np.outer(np.sin(np.pi * x), np.sin(np.pi * x)).ravel()
    rho, RT = 1 + 0.01 * s, 0.5 + 0.01 * s
    u = 0.05 * s[:, None] * rng.normal(size=2)
    T = []
    for prec in ("fp64", "fp32"):
        d = S.Dvm.from_case(c, prec).init(rho, u, RT)
        d.step(steps)
        T.append(d.macros()[2])
    assert np.sqrt(np.mean((T[1] - T[0]) ** 2)) <= bound
