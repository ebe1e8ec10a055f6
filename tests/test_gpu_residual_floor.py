"""The floor that rounding sets for the FP32 residual, which decides what solves reach their target."""
import numpy as np
import pytest

from paper_2007_07347_gb300 import meshes as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,re,checks", [(48, 1000.0, 215), (40, 300.0, 90)])
def test_a_batch_has_no_higher_floor_than_single_solves(n, re, checks):
    """The median of the last 15 residuals, taken every 1000 steps past convergence, of a batched
    solve (the marching form's arithmetic) and of a single one (the block kernel's).  The same
    equations in other sums: 10 % for that.  Equilibria rounded in two ways gave 1.65 and 1.14 times."""
    from paper_2007_07347_gb300 import sdugks as S
    case = M.cavity(n, Re=re)
    b = S.Batch(64 << 20, "fp32", max_instances=2)
    i = b.add_case(case)
    s = S.Solver.from_case(case, "fp32").init()
    eps = []
    for _ in range(checks):
        b.step(1000)
        s.step(1000)
        eps.append((b.residual()[i][0], s.residual()[0]))
    last = np.median(np.array(eps[-15:]), axis=0)
    assert last[1] < 1e-6 and last[0] <= 1.1 * last[1], last
