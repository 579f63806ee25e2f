"""The Courant guard (option cfl_alpha) beside values that are not finite: a state
over the limit is reported by the next pizza_synchronize whatever the states
after it hold, since the maxima are over every state evaluated in between."""
import numpy as np
import pytest

from paper_1902_07092_gb300 import inputs

pytestmark = pytest.mark.gpu

ECFL = -5


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("n_phi,options", [(96, ()), (6144, ()), (96, (("azimuthal_dd", 0),)), (96, (("precision", 1),))])
def test_rates_before_a_nan_are_reported(n_phi, options, bad):
    from paper_1902_07092_gb300 import binding as B
    n_r = 17
    th = inputs.theta_init(n_r, n_phi, 1.0, 4, cfg=7, m_min=0)
    ps = inputs.theta_init(n_r, n_phi, 1.0, 5, cfg=8)
    ps[0] = 0.0
    z, zu = inputs.zero_state(n_r, n_phi)
    s = B.Solver(n_r, n_phi, 1e-3, 1.1e5, 1.0, 0.35, "CNAB2", 1e-4)
    for k, v in options:
        B.pizza_set_option(s.ctx, k, v)
    s.set_state(th, ps, zu)
    d = s.diagnostics()
    B.pizza_set_option(s.ctx, "cfl_alpha", 0.5e-4 * max(d["cfl_s"], d["cfl_phi"]))
    s.step(1)
    spoilt = ps.copy()
    spoilt[3, 2] = bad
    s.set_state(th, spoilt, zu)
    s.step(1)
    with pytest.raises(B.PizzaError) as ei:
        B.pizza_synchronize(s.ctx)
    assert ei.value.code == ECFL
    # and alone such a state trips nothing (check_finite and the diagnostics report it)
    s.set_state(th, spoilt, zu)
    s.step(1)
    B.pizza_synchronize(s.ctx)
    s.close()
