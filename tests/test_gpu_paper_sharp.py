"""Positions of the paper's problem sampled where its f_x is nearly zero at one
point (A(t) = e^{t/T}/5 close to one): against the oracle's bisection, to 16
roundings (2^-52) of F over f_x, which is what a root's conditioning allows."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2602_15130_gb300 import Pic, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("t0", [1.5, 1.6, 1.605, 1.6085])
def test_sampled_positions_at_sharp_densities(t0):
    import __graft_entry__ as g

    g.build()
    p = workloads.paper_small(n_particles=200003, K=0, max_ppc=2048)
    sim, orc = Pic(p), O.Oracle(p)
    sim.sample_mms(t0)
    orc.sample(t0)
    x, xo = sim.get_state()[0], orc.state()[0]
    cfg = O.make_cfg(p)
    for d in range(3):
        f = np.array([O.fx(cfg, d, float(v), t0) for v in xo[:, d]])
        e = np.abs(x[:, d] - xo[:, d])
        assert (np.minimum(e, 1.0 - e) <= 16 * 2.0 ** -52 / f).all()
