"""A caller's rows through pic_set_state and pic_get_state in the precision
form, bit for bit: the cell floor(x n) with x n rounded to FP64, the offset x n
- cell rounded to FP64 and then to FP32, velocities rounded to FP32, and back
(cell + offset) h in FP64. Coordinates at cell edges, one ulp beside them,
tiny, on rounding ties, and meshes that are and are not powers of two;
velocities on ties, subnormal in FP32, infinite. Device, pinned and pageable
rows take different paths (in place or staged)."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2602_15130_gb300 import Pic, workloads

pytestmark = pytest.mark.gpu


def _coordinates(n, g, count):
    k = g.integers(0, n, count)
    edge = k / n
    kinds = [g.random(count), edge, np.nextafter(edge, 2.0), np.maximum(np.nextafter(edge, -1.0), 0.0),
             edge + (g.integers(0, 1 << 24, count) + 0.5) * 2.0 ** -24 / n, np.ldexp(g.random(count), -g.integers(0, 130, count)),
             1.0 - g.integers(1, 5, count) * 2.0 ** -53]
    x = np.choose(g.integers(0, len(kinds), count), kinds)
    return np.clip(x, 0.0, np.nextafter(1.0, 0.0))


def _velocities(g, count):
    tie = np.float32(g.standard_normal(count)).astype(np.float64)
    tie = tie + 0.5 * np.spacing(np.abs(tie).astype(np.float32)).astype(np.float64)
    kinds = [g.standard_normal(count), tie, np.ldexp(g.standard_normal(count), -g.integers(100, 160, count)),
             np.zeros(count)]
    return np.choose(g.integers(0, len(kinds), count), kinds)


def _expected(x, n):
    out = np.empty_like(x)
    for i, v in enumerate(x):
        c = min(n - 1, int(np.floor(v * n)))
        o = np.float32(float(Fraction(v) * n - c))
        o = np.float32(1.0 - 2.0 ** -24) if o >= 1 else max(o, np.float32(0.0))
        out[i] = (float(c) + float(o)) * (1.0 / n)
    return out


@pytest.mark.parametrize("n", [2, 7, 8, 100])
@pytest.mark.parametrize("memory", ["device", "pinned", "pageable"])
def test_rows_round_as_documented(n, memory):
    import torch

    import __graft_entry__ as g

    g.build()
    rng = np.random.default_rng(n)
    count = 3001
    x = _coordinates(n, rng, 3 * count).reshape(count, 3)
    v = _velocities(rng, 3 * count).reshape(count, 3)
    p = workloads.mixed(workloads.base(n, count, 0.01, 0, 1.0, cg_maxit=1))
    with Pic(p) as sim:
        for _ in range(2):  # the first load also forms v^M
            if memory == "pageable":
                sim.set_state(x, v, allow=(4,))
                xo, vo = sim.get_state()
            else:
                put = (lambda a: torch.from_numpy(a).cuda()) if memory == "device" else \
                    (lambda a: torch.from_numpy(a).pin_memory())
                out = tuple(put(np.zeros_like(x)) for _ in range(2))
                sim.set_state(put(x), put(v), allow=(4,))
                xo, vo = (a.cpu().numpy() for a in sim.get_state(out=out))
            assert np.array_equal(xo.ravel(), _expected(x.ravel(), n))
            with np.errstate(over="ignore"):
                assert np.array_equal(vo, v.astype(np.float32).astype(np.float64))
