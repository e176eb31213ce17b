"""Collision calls of the precision form in which the warps of a block share a
cell: two warps (two chunks of 32 outcomes), four (three and more, with a last
round of one to three chunks), cells of one word of particles and of more words
than warps, lists that run over.

The decisions are the oracle's except in cells with a flagged one, and outside
those every particle is within 2e-5 of the oracle's <dv>, the precision form's
stated error; the logging variant gives the same bits."""
import numpy as np
import pytest

import pairlists
from paper_2602_15130_gb300 import Pic, workloads
from test_gpu_mixed import oracle_on_gpu_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ppc,K,dt", [(5, 9, 33, 0.01), (5, 20, 64, 0.01), (4, 70, 65, 0.01), (4, 33, 160, 0.01),
                                        (3, 180, 224, 0.005), (3, 12, 40, 0.05)])
def test_shared_cells_match_oracle(n, ppc, K, dt):
    import __graft_entry__ as g

    g.build()
    p = workloads.mixed(workloads.base(n, ppc * n ** 3 + 7, dt, K, workloads.hard_sphere_sigma0(ppc, 0.01), seed=2,
                                       max_ppc=64 + 3 * ppc // 32 * 32))
    s = Pic(p)
    s.sample_mms(0.0)
    o = oracle_on_gpu_state(p, s)
    s.set_decision_log(1, 1 << 16)
    dv, dvm = s.collide_avg(1)
    s.set_decision_log(2, 1 << 21)
    dv2, dvm2 = s.collide_avg(1)
    assert np.array_equal(dv, dv2) and np.array_equal(dvm, dvm2)
    o.set_pair_log(True)
    dvo, dvmo = o.collide_avg(1)
    assert np.abs(dvo).max() > 0
    flagged, _ = pairlists.compare_flagged(s.decision_log(), o.pair_log())
    reached = np.isin(s.get_sort()[0], [c for _, c in flagged])
    off = (np.abs(dv - dvo) > 2e-5).any(axis=1)
    assert not (off & ~reached).any()
    assert not reached.all()
    assert np.abs(dvm - dvmo).max() <= 1e-5 * max(1.0, np.abs(dvmo).max())
