"""Implicit solves at the edges of their forms against the oracle: dense inverses
(N_c <= 42) from the smallest radial grid up, the block chains from one block a
half upward and just past the dense solve's last size, split streamfunction
blocks, and the chains asked for below that size, which must agree with the dense
solve.  Bars as in the parity tests of these sizes (1e-12 up to n_r = 65, 2e-12
at 129 and 257, 5e-12 at 513)."""
import numpy as np
import pytest

from oracle.stepper import IntegrationStepper
from paper_1902_07092_gb300 import inputs
from tests.parity_util import assert_state_close, rel_l2

pytestmark = pytest.mark.gpu


def run(n_r, n_phi, scheme, implicit, options=(), steps=2, ora=None):
    from paper_1902_07092_gb300 import binding as B
    args = (n_r, n_phi, 1e-3, 1.1e5, 1.0, 0.35, scheme, 1e-5)
    th = inputs.theta_init(n_r, n_phi, 1e-2, 11, cfg=1, m_min=0)
    psi = inputs.theta_init(n_r, n_phi, 1e-4, 12, cfg=8)
    psi[0] = 0.0
    u = inputs.theta_init(n_r, n_phi, 1e-2, 13, cfg=9, m_min=0)[0].real.copy()
    s = B.Solver(*args, buoy_implicit=implicit)
    for k, v in options:
        B.pizza_set_option(s.ctx, k, v)
    s.set_state(th, psi, u)
    s.step(steps)
    got = s.get_state()
    s.close()
    if ora is None:
        ora = IntegrationStepper(*args, buoy_implicit=implicit)
        ora.set_state(psi, th, u)
        for _ in range(steps):
            ora.step()
    return got, ora


def bar(n_r):
    return 1e-12 if n_r <= 65 else 2e-12 if n_r <= 257 else 5e-12


@pytest.mark.parametrize("implicit", [False, True])
@pytest.mark.parametrize("n_r,n_phi,scheme", [(9, 12, "ARS443"), (17, 24, "SBDF3"), (33, 48, "BPR353"), (65, 24, "CNAB2"),
                                              (129, 12, "SBDF2"), (513, 12, "CNAB2")])
def test_solve_matches_oracle(n_r, n_phi, scheme, implicit):
    got, ora = run(n_r, n_phi, scheme, implicit)
    assert_state_close(got, ora.y, bar(n_r), oracle=ora)


@pytest.mark.parametrize("options", [(("psi_chain_dd", 0),), (("psi_chain_dd", 1),), (("theta_fp32", 1),),
                                     (("solve_roles", 1),), (("solve_roles", 1), ("psi_chain_dd", 1), ("theta_fp32", 1))])
@pytest.mark.parametrize("n_r,implicit", [(9, False), (17, False), (33, False), (33, True)])
def test_chains_below_the_dense_size(n_r, implicit, options):
    got, ora = run(n_r, 24, "ARS443", implicit, options)
    assert_state_close(got, ora.y, bar(n_r), oracle=ora)
    dense, _ = run(n_r, 24, "ARS443", implicit, ora=ora)
    flat = [np.concatenate([np.ravel(x) for x in y]) for y in (got, dense)]
    assert rel_l2(*flat) <= bar(n_r)


@pytest.mark.parametrize("n_r,n_phi,scheme", [(65, 384, "SBDF2"), (129, 24, "SBDF3"), (129, 384, "ARS443"),
                                              (129, 768, "CNAB2"), (257, 12, "BPR353"), (129, 3072, "CNAB2")])
def test_one_cta_per_system_or_per_mode_by_default(n_r, n_phi, scheme):
    """Either side of the default rule's lines (N_c 64, 152 and 608 modes): the default
    is one of the two arrangements bit by bit, and the two agree."""
    got = [run(n_r, n_phi, scheme, False, o, ora=0)[0] for o in ((), (("solve_roles", 0),), (("solve_roles", 1),))]
    flat = [np.concatenate([np.ravel(x) for x in y]) for y in got]
    per_system = inputs.n_c_integration(n_r) > 64 and not 152 < n_phi // 3 + 1 <= 608
    assert np.array_equal(flat[0], flat[2 if per_system else 1])
    assert rel_l2(flat[1], flat[2]) <= bar(n_r)
