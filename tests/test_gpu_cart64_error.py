"""FP64 on uniform grids where dt/(2 tau) is large: the error of the steps' rounding, against the plain
FP64 restatement of the timed cases."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,re,steps,bound", [(32, 5000.0, 400, 3.6e-13), (48, 4000.0, 300, 1.3e-13), (256, 5000.0, 60, 1.7e-14)])
def test_fp64_rounding_at_high_reynolds_numbers(n, re, steps, bound):
    """2-norm of u; the bounds are the errors of the kernel that rounded each product and sum."""
    from perf import cases
    case = dict(flow="cavity", nx=n, ny=n, re=re, precision="fp64", steps=steps)
    u = cases.run(cases.prepare(case, 11))["u"].cpu().numpy()
    exact = cases.exact(case, 11)["u"].cpu().numpy()
    assert np.sqrt(np.sum((u - exact) ** 2) / np.sum(exact ** 2)) <= bound
