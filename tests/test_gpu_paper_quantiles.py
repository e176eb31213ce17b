"""The paper's problem sampled at 200,003 particles: positions and velocities
against the oracle's bisection. 1.2 million quantiles reach 1e-6 from either
end and from the median of f_v, where the branches of its inverse meet. The
bisection evaluates G itself, whose rounding (2^-53) moves a root by at most
2^-53 / G'(tau): 1e-11 where |tau| > 0.005 (G' = 2 tau^2 / sqrt pi); nearer
the median tau^3 is off by at most 2^-53 of it, so tau by at most 1e-5."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2602_15130_gb300 import Pic, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("t0", [0.0, 0.6])
def test_sampled_quantiles_match_bisection(t0):
    import __graft_entry__ as g

    g.build()
    p = workloads.paper_small(n_particles=200003, K=0, max_ppc=2048)
    sim, orc = Pic(p), O.Oracle(p)
    sim.sample_mms(t0)
    orc.sample(t0)
    (x, v), (xo, vo) = sim.get_state(), orc.state()
    d = np.abs(x - xo)
    assert np.minimum(d, 1.0 - d).max() <= 1e-14
    vh = p["v_bar"] * 1.2
    tol = np.where(np.abs(vo) > 0.005 * vh, 1e-11, 1e-5) * vh
    assert (np.abs(v - vo) <= tol).all()
    assert np.median(np.abs(v - vo)) <= 1e-13 * vh
