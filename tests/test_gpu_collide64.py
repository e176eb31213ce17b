"""The FP64 collision call where its branches differ: cells of more than 255
particles and groups beyond the staged FP32 copy, outcomes that change more
particles than their list holds, outcomes shared by several warps of a cell,
the odd-power cross section, and velocities whose FP32 rounding decides
nothing (far from the origin, or not representable): every accept decision
and candidate count equals the oracle's, and the averages agree to 1e-10 of
their magnitude (the parity tests' bar)."""
import numpy as np
import pytest

import inputs
from oracle import oracle as O
from paper_2602_15130_gb300 import Pic, workloads

pytestmark = pytest.mark.gpu

TOL = 1e-10


def _case(name):
    w = workloads
    base = dict(n=4, n_particles=1500, K=40, max_ppc=1024, cg_tol=1e-10)
    if name == "crowded":       # ~500 per cell, unstaged, lists searched by index
        return w.smallest(**base, dt=0.002), inputs.particles(1500, seed=1, clustered_cells=3, n=4)
    if name == "spilled":       # most of a cell changes in every outcome
        return w.smallest(**base, dt=0.05), inputs.particles(1500, seed=2, clustered_cells=12, n=4)
    if name == "parts":         # 8 cells, K = 150: chunks shared by warps
        return w.smallest(n=2, n_particles=700, K=150, cg_tol=1e-10), inputs.particles(700, seed=3)
    if name == "odd_power":
        return w.paper_small(n_particles=4500, K=33), inputs.particles(4500, seed=4, v_mean=0.0, v_sigma=0.1)
    if name == "far":           # FP32 keeps no digit of v_p - v_q
        p, (x, v) = w.smallest(n_particles=4099, K=9), inputs.particles(4099, seed=5)
        return p, (x, v + 3.0e7)
    if name == "beyond_fp32":   # one velocity in ten overflows FP32
        p, (x, v) = w.smallest(n_particles=2000, K=7), inputs.particles(2000, seed=6)
        v[::10] *= 1e39
        return p, (x, v)
    raise ValueError(name)


@pytest.mark.parametrize("name", ["crowded", "spilled", "parts", "odd_power", "far", "beyond_fp32"])
def test_collision_call_matches_oracle(name):
    import __graft_entry__ as g

    g.build()
    p, (x, v) = _case(name)
    sim, orc = Pic(p), O.Oracle(p)
    sim.set_state(x, v, 0.0)
    orc.set_state(x, v, 0.0)
    sim.reset_stats()
    orc.reset_stats()
    dv, dvm = sim.collide_avg(1)
    dvo, dvmo = orc.collide_avg(1)
    st, so = sim.stats(), orc.stats()
    assert st["n_cand"] == so["n_cand"] and st["n_cand"] > 0
    assert abs(st["n_coll"] - so["n_coll"]) <= st["n_near_ties"]
    assert st["n_gmax_exceed"] == so["n_gmax_exceed"]
    if st["n_near_ties"] == 0:
        for a, b in ((dv, dvo), (dvm, dvmo)):
            scale = np.maximum(1.0, np.abs(np.concatenate([b, v], axis=1)).max(axis=1, keepdims=True))
            if name == "beyond_fp32":  # a partner's velocity scales a change
                scale = max(np.abs(v).max(), np.abs(b).max())
            assert (np.abs(a - b) <= TOL * scale).all()
