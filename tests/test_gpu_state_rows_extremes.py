"""Velocities of a caller's rows at the ends of FP32 through pic_set_state and
pic_get_state in the precision form, bit for bit the conversions' values:
infinite, overflowing to infinity or just not, subnormal, on ties there, signed
zeros. Device, pinned and pageable rows."""
import numpy as np
import pytest

from paper_2602_15130_gb300 import Pic, workloads

pytestmark = pytest.mark.gpu

TOP = float(np.finfo(np.float32).max)
KINDS = np.array([np.inf, 1e39, 1e300, TOP, TOP * (1.0 + 2.0 ** -25), np.nextafter(TOP * (1.0 + 2.0 ** -25), 0.0),
                  np.nextafter(TOP, np.inf), 2.0 ** -126, np.nextafter(2.0 ** -126, 0.0), 1.5 * 2.0 ** -149,
                  2.0 ** -149, 2.0 ** -150, np.nextafter(2.0 ** -150, 1.0), 1e-60, 5e-324, 0.0, 1.0])


@pytest.mark.parametrize("memory", ["device", "pinned", "pageable"])
def test_velocities_at_the_ends_of_fp32(memory):
    import torch

    import __graft_entry__ as g

    g.build()
    count = 1500
    rng = np.random.default_rng(3)
    x = rng.random((count, 3))
    v = rng.choice(KINDS, (count, 3)) * rng.choice([-1.0, 1.0], (count, 3))
    with np.errstate(over="ignore"):
        want = v.astype(np.float32).astype(np.float64)
    with Pic(workloads.mixed(workloads.base(6, count, 0.01, 0, 1.0, cg_maxit=1))) as sim:
        for _ in range(2):
            if memory == "pageable":
                sim.set_state(x, v, allow=(4,))
                got = sim.get_state()[1]
            else:
                put = (lambda a: torch.from_numpy(a).cuda()) if memory == "device" else \
                    (lambda a: torch.from_numpy(a).pin_memory())
                out = tuple(put(np.zeros_like(x)) for _ in range(2))
                sim.set_state(put(x), put(v), allow=(4,))
                got = sim.get_state(out=out)[1].cpu().numpy()
            assert np.array_equal(got.view(np.int64), want.view(np.int64))
