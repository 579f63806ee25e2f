"""FP64 radial transforms on request (option radial_dd = 0) in the batched layout, which
runs them in fixed point by default: other bits, the oracle's terms to the bar of
the parity tests, with one, two and four transforms in a pass and with pumping."""
import numpy as np
import pytest

from oracle.explicit import explicit_terms
from tests.test_gpu_fixed_point import errors, state

pytestmark = pytest.mark.gpu


def bar(n_r):
    return max(1e-12, 4 * n_r * n_r * 2.0 ** -53)  # test_gpu_parity.py


def terms(n_r, n_phi, options, pumping=None):
    from paper_1902_07092_gb300 import binding as B
    ps, th, u = state(n_r, n_phi, (1.0, 1.0, 1.0))
    s = B.Solver(n_r, n_phi, 1e-3, 1.1e5, 1.0, 0.35, "CNAB2", 1e-4, pumping_eps=pumping)
    for k, v in options:
        B.pizza_set_option(s.ctx, k, v)
    s.set_state(th, ps, u)
    got = s.explicit_terms()
    s.close()
    return got


@pytest.mark.parametrize("n_r,n_phi,extra", [(9, 24, ()), (33, 96, ()), (129, 48, (("radial_batch", 1),)),
                                             (129, 48, (("radial_batch", 2),)), (257, 24, ()), (513, 24, ()),
                                             (1025, 24, (("radial_lean", 0),)), (2049, 12, (("radial_lean", 0),))])
def test_fp64_transforms_in_the_batched_layout(n_r, n_phi, extra):
    assert max(errors(n_r, n_phi, options=extra + (("radial_dd", 0),))) <= bar(n_r)
    a, b = terms(n_r, n_phi, extra), terms(n_r, n_phi, extra + (("radial_dd", 0),))
    assert not all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("n_r", [33, 257])
def test_fp64_transforms_with_pumping(n_r):
    from oracle.stepper import IntegrationStepper
    got = terms(n_r, 48, (("radial_dd", 0),), pumping=3e-3)
    ps, th, u = state(n_r, 48, (1.0, 1.0, 1.0))
    ps[0] = 0.0
    ora = IntegrationStepper(n_r, 48, 1e-3, 1.1e5, 1.0, 0.35, "CNAB2", 1e-4, pumping_eps=3e-3)
    for a, b in zip(got, explicit_terms(ora.g, ps, th, u)):
        assert np.linalg.norm(a - b) <= bar(n_r) * np.linalg.norm(b)


@pytest.mark.parametrize("n_r", [33, 257])
def test_fp64_transforms_keep_subnormal_values(n_r):
    """A state of 2^-1040: its grid values to the spacing of the subnormal numbers (2^-1074;
    off the walls, where u_phi is scaled by the vanishing v), against those of the state itself."""
    from paper_1902_07092_gb300 import binding as B
    ps, th, u = state(n_r, 24, (1.0, 1.0, 1.0))
    f = 2.0 ** -1040
    s = B.Solver(n_r, 24, 1e-3, 1.1e5, 1.0, 0.35, "CNAB2", 1e-4)
    B.pizza_set_option(s.ctx, "radial_dd", 0)
    s.set_state(th, ps, u)
    ref = s.get_grid()
    s.set_state(th * f, ps * f, u * f)
    for a, b in zip(s.get_grid(), ref):
        assert np.abs(a[1:-1] / f - b[1:-1]).max() <= 1e-3 * np.abs(b).max()
    s.close()
