"""The FP64 collision call in any units: velocities, g_max and cross sections
whose squares or coefficients are subnormal, zero or infinite in FP32 (seconds
and metres with sigma(g) g near 1e-13 are enough for the odd-power cross
section), a drift that FP32 keeps no digit of v_p - v_q beside, and a few
velocities beyond FP32. About a million candidates a case: every decision is
the oracle's outside outcomes with a flagged near tie, and away from those
cells the averages agree to 400 ulps of the largest velocity of the cell (an
outcome scatters a particle some ten times at most, each rounded by a few
ulps on either side)."""
import numpy as np
import pytest

import pairlists
from oracle import oracle as O
from paper_2602_15130_gb300 import Pic, workloads

pytestmark = pytest.mark.gpu

N, CELLS, K, PMAX = 3840, 4, 256, 0.036


def _hard_spheres(g_max):
    s = g_max / (10.0 * np.sqrt(3.0))
    n_phys = PMAX * N / CELLS ** 3 / 0.01  # sigma0 g_max = 1
    return workloads.base(CELLS, N, 0.01, K, 1.0 / g_max, g_max=g_max, v_mean=(0.2 * s,) * 3, v_sigma=s, n_phys=n_phys,
                          max_ppc=256), s


def _odd_power(g_max, sigma_2):
    """sigma(g) g = A (0.1 + 2.4 y - 2.4 y^2), y = g^2 / g_max^2, with the given sigma_2."""
    s = g_max / (10.0 * np.sqrt(3.0))
    A = -sigma_2 * g_max ** 4 / 2.4
    n_phys = PMAX * N / CELLS ** 3 / (1.0 / 16) / (0.7 * A)
    return workloads.paper_small(n=CELLS, n_particles=N, K=K, cg_tol=1e-10, g_max=g_max, v_bar=s, n_phys=n_phys,
                                 max_ppc=256, sigma_n=(0.1 * A, 2.4 * A / g_max ** 2, sigma_2)), s


CASES = {
    "odd_1e8": lambda: _odd_power(1e8, -4e-45),
    "odd_1e11": lambda: _odd_power(1e11, -3.2e-48),
    "odd_1e-12": lambda: _odd_power(1e-12, -1.0),
    "odd_1": lambda: _odd_power(1.0, -1.0),
    "hard_1e-21": lambda: _hard_spheres(1e-21),
    "hard_1e-22": lambda: _hard_spheres(1e-22),
    "hard_1e-120": lambda: _hard_spheres(1e-120),
    "hard_1e-9": lambda: _hard_spheres(1e-9),
    "hard_1e9": lambda: _hard_spheres(1e9),
    "hard_1e25": lambda: _hard_spheres(1e25),
    "hard_1e120": lambda: _hard_spheres(1e120),
    "far": lambda: _hard_spheres(10.0 * np.sqrt(3.0)),
    "beyond_fp32": lambda: _hard_spheres(10.0 * np.sqrt(3.0)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_decisions_in_any_units(name):
    import __graft_entry__ as g

    g.build()
    p, s = CASES[name]()
    rng = np.random.default_rng(11)
    x = rng.random((N, 3))
    v = s * rng.standard_normal((N, 3))
    if name == "far":
        v += 3.0e7
    if name == "beyond_fp32":
        v[rng.choice(N, 8, replace=False)] *= 1e39
    sim, orc = Pic(p), O.Oracle(p)
    sim.set_state(x, v, 0.0)
    orc.set_state(x, v, 0.0)
    dv, dvm = sim.collide_avg(1)
    sim.set_decision_log(2, 1 << 21)
    dv2, dvm2 = sim.collide_avg(1)
    assert np.array_equal(dv, dv2) and np.array_equal(dvm, dvm2)
    orc.set_pair_log(True)
    dvo, dvmo = orc.collide_avg(1)
    flagged, _ = pairlists.compare_flagged(sim.decision_log(), orc.pair_log())
    cell = sim.get_sort()[0]
    there = ~np.isin(cell, [c for _, c in flagged])
    assert there.any()
    top = np.zeros(CELLS ** 3)
    np.maximum.at(top, cell, np.abs(v).max(axis=1))
    for a, b in ((dv, dvo), (dvm, dvmo)):
        tol = 400 * 2.0 ** -52 * (top[cell] + np.abs(b).max(axis=1))
        assert (np.abs(a - b) <= tol[:, None])[there].all()
    assert np.abs(dvo).max() > 0.0
