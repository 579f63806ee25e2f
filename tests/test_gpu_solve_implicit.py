"""Implicit buoyancy with FP32-refined temperature solves: the temperature takes the whole
CTA (its block in two halves from 40 blocks on, one below), then the streamfunction,
whose correction lies over the temperature's FP32 arrays.  Against the oracle at the
bars of test_gpu_solve.py, from the zonal flow's CTA on, at N_c just below and above
the split and in the range where the FP32 solves are the default."""
import numpy as np
import pytest

from tests.parity_util import assert_state_close
from tests.test_gpu_solve import bar, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_r,options", [(9, (("theta_fp32", 1),)), (65, (("theta_fp32", 1),)), (129, (("theta_fp32", 1),)),
                                         (257, (("theta_fp32", 1),)), (513, (("theta_fp32", 1),)), (1025, ())])
@pytest.mark.parametrize("scheme", ["SBDF2", "ARS443"])
def test_implicit_buoyancy_with_fp32_temperature_chains(n_r, options, scheme):
    got, ora = run(n_r, 12, scheme, True, options)
    assert_state_close(got, ora.y, bar(n_r), oracle=ora)
    again, _ = run(n_r, 12, scheme, True, options, ora=ora)
    assert all(np.array_equal(a, b) for a, b in zip(got, again))


def test_implicit_buoyancy_solve_beside_the_explicit_one():
    """Solve kernel at N_c = 682 with 257 modes: the temperature's and the streamfunction's
    systems one after the other, two modes an SM, take at most twice the time that they
    take side by side, and a tenth for the coupling (best of ten averages of five)."""
    from paper_1902_07092_gb300 import binding as B
    from paper_1902_07092_gb300 import inputs
    th = inputs.theta_init(1025, 768, 1e-3, 11, cfg=1)
    best = []
    for implicit in (False, True):
        s = B.Solver(1025, 768, 1e-5, 1e7, 1.0, 0.35, "CNAB2", 1e-7, buoy_implicit=implicit)
        s.set_state(th, *inputs.zero_state(1025, 768))
        s.step(3)
        t = np.inf
        for _ in range(10):
            B.pizza_profile_begin(s.ctx, 8)
            s.step(5)
            ms, n = B.pizza_profile_end(s.ctx)
            t = min(t, ms[3] / n[3])
        best.append(t)
        s.close()
    assert best[1] <= 2.2 * best[0], best
