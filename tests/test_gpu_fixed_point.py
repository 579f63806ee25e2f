"""Fixed-point transforms of the FP64 explicit stage (radial DCT-I in both layouts,
azimuthal products) against the oracle at the edges of their ranges: the smallest
transforms (2 passes), lengths with and without the radix-8 and radix-3 passes,
few modes on many radii and the reverse, every batch of the radial kernels, both
azimuthal buffer layouts, and fields of very different magnitude."""
import numpy as np
import pytest

from oracle.explicit import explicit_terms
from oracle.stepper import IntegrationStepper
from paper_1902_07092_gb300 import inputs
from tests.parity_util import U_FACTOR, zonal_forcing

pytestmark = pytest.mark.gpu

E, RA, PR, ETA = 1e-3, 1.1e5, 1.0, 0.35


def state(n_r, n_phi, scale):
    nc = inputs.n_c_integration(n_r)
    th = inputs.theta_init(n_r, n_phi, scale[0], 3, cfg=7)
    ps = inputs.theta_init(n_r, n_phi, scale[1], 4, cfg=7)
    u = inputs.theta_init(n_r, n_phi, scale[2], 5, cfg=7, m_min=0)[0].real.copy()
    return ps, th, u[:nc]


def errors(n_r, n_phi, scale=(1.0, 1.0, 1.0), options=()):
    from paper_1902_07092_gb300 import binding as B
    ps, th, u = state(n_r, n_phi, scale)
    s = B.Solver(n_r, n_phi, E, RA, PR, ETA, "CNAB2", 1e-4)
    for k, v in options:
        B.pizza_set_option(s.ctx, k, v)
    s.set_state(th, ps, u)
    got = s.explicit_terms()
    s.close()
    ora = IntegrationStepper(n_r, n_phi, E, RA, PR, ETA, "CNAB2", 1e-4)
    ps = ps.copy()
    ps[0] = 0.0
    ref = explicit_terms(ora.g, ps, th, u)
    mean, terms = zonal_forcing(ora, (ps, th, u))
    c_u = np.linalg.norm(terms) / np.linalg.norm(mean)
    e = [np.linalg.norm(a - b) / np.linalg.norm(b) for a, b in zip(got, ref)]
    # the zonal term is a mean that cancels to 1/c_u of its terms, in the oracle too
    return e[0], e[1], e[2] / max(U_FACTOR, c_u)


def bar(n_r):
    # the flux divergence differentiates rounded products: |T_n'| <= n^2
    return max(1e-12, 4 * n_r ** 2 * np.finfo(float).eps)


@pytest.mark.parametrize("n_r,n_phi", [(9, 12), (9, 384), (17, 24), (33, 48), (65, 1536), (129, 12), (257, 192),
                                       (513, 24), (33, 6144)])
def test_explicit_terms(n_r, n_phi):
    assert max(errors(n_r, n_phi)) <= bar(n_r)


@pytest.mark.parametrize("nb", [1, 2, 4])
def test_radial_batches(nb):
    assert max(errors(129, 96, options=(("radial_batch", nb),))) <= bar(129)


@pytest.mark.parametrize("n_r", [129, 257, 1025])
def test_lean_layout(n_r):
    assert max(errors(n_r, 48, options=(("radial_lean", 1), ("radial_dd", 1)))) <= bar(n_r)


@pytest.mark.parametrize("scale", [(1e-90, 1e60, 1.0), (1e80, 1e-70, 1e-20)])
@pytest.mark.parametrize("n_r", [33, 129])
def test_magnitudes_far_apart(n_r, scale):
    lean = (("radial_lean", 1), ("radial_dd", 1)) if n_r == 129 else ()
    # (the zonal term, 1e-70 of the products it is the mean of, is lost in the oracle)
    assert max(errors(n_r, 48, scale, lean)[:2]) <= bar(n_r)


@pytest.mark.parametrize("n_r,n_phi", [(33, 96), (1025, 24)])
def test_infinity_reaches_the_terms(n_r, n_phi):
    from paper_1902_07092_gb300 import binding as B
    ps, th, u = state(n_r, n_phi, (1.0, 1.0, 1.0))
    th[2, 5] = np.inf
    s = B.Solver(n_r, n_phi, E, RA, PR, ETA, "CNAB2", 1e-4)
    s.set_state(th, ps, u)
    e_psi, e_theta, _ = s.explicit_terms()
    s.close()
    assert not np.isfinite(e_theta).all()
