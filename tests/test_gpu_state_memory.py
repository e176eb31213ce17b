"""Device memory of the precision form. A context takes 188 bytes a particle
when it is created (two sorted copies of 44, the Lorentz and collision terms
and <dv^M> of 12 each, key, rank and perm of 4, 52 of staging), and its reduction slots 32
bytes a block; v^M by pid (16 bytes a particle) and the bins (48 bytes a
record) come with the first state, and where the allocator refuses them every
call gives the same bits without."""
import numpy as np
import pytest

import inputs
import paper_2602_15130_gb300 as M
from paper_2602_15130_gb300 import Pic, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture
def meter(monkeypatch):
    import __graft_entry__ as g

    g.build()
    state = {"sizes": [], "refuse": False}
    real = M._TorchAllocator._alloc

    def alloc(self, user, nbytes):
        if state["refuse"]:
            return None
        state["sizes"].append(int(nbytes))
        return real(self, user, nbytes)

    monkeypatch.setattr(M._TorchAllocator, "_alloc", alloc)
    return state


def _created(meter, n, count):
    meter["sizes"].clear()
    with Pic(workloads.mixed(workloads.base(n, count, 0.01, 0, 1.0))) as s:
        created = list(meter["sizes"])
        s.sample_mms(0.0)
    return created, meter["sizes"][len(created):]


def test_bytes_per_particle_and_record(meter):
    a, _ = _created(meter, 8, 1 << 14)
    b, more = _created(meter, 8, 1 << 15)
    blocks = max(len(a), len(b))
    # the error norms' block partials (14 doubles in 256 particles or more) beside the arrays
    assert sum(b) - sum(a) <= (188 + 14 * 8 / 256) * (1 << 14) + 64 * blocks
    mean = (1 << 15) // 8 ** 3
    assert sum(more) <= 48 * 8 ** 3 * 4 * mean + 16 * (1 << 15) + 64 * 4
    # a mesh of plain CG over 89 blocks: no slots by the square of them beside the
    # 116.5 bytes a node (field 16, b, phi, r, p and q 4, count and start 4, corners 64, rho 8, partials)
    c, _ = _created(meter, 45, 1 << 14)
    assert sum(c) - sum(a) <= 118 * (45 ** 3 - 8 ** 3)


@pytest.mark.parametrize("dist", ["config", "paper"])
def test_refused_extras_change_no_bit(meter, dist):
    import torch

    n, count = 8, 8 ** 3 * 20 + 7
    p = workloads.mixed(workloads.smallest(n=n, n_particles=count, K=4) if dist == "config" else
                        workloads.paper_small(n=n, n_particles=count, K=4))
    x, v = inputs.particles(count, seed=9, v_mean=0.0, v_sigma=0.1)
    runs = []
    for refuse in (False, True):
        meter["refuse"] = False
        out = []
        with Pic(p) as s:
            meter["refuse"] = refuse
            for put in (lambda a: torch.from_numpy(a).cuda(), lambda a: a, lambda a: torch.from_numpy(a).pin_memory(),
                        lambda a: torch.from_numpy(a).cuda(), None):
                if put:
                    s.set_state(put(x), put(v))
                else:
                    s.sample_mms(0.0)
                s.step(1)
                out += list(s.get_state()) + list(s.get_sort()) + [s.mms_error()["array"]] + list(s.collide_avg(0))
        runs.append(out)
        meter["refuse"] = False
    for a, b in zip(*runs):
        assert np.array_equal(a, b)
