"""The FP64 kick's tables: the drift's dG^{-1}/dT (and the general path that
takes over where f_x is too sharp for it) and the Lorentz term's sin and cos,
at positions on, just below and between cell faces, in single steps.

Drift, with q/m = 0: against extended precision (x^M by Newton). x + dt w
rounds twice, w = v + xdot^M - v^M and its terms a few times; xdot^M carries
the 2^-53 (1 + |c t|) of T times |d xdot^M / dT| <= |c| 2 pi A / (1 - A)^3.
Lorentz term, with a field: v_1 - v_0 = (L_0 + L_1)/2 with E as the library
gives it at both ends; 8 node products, three factors of 2 ulp each."""
import numpy as np
import pytest

import inputs
from oracle import oracle as O
from paper_2602_15130_gb300 import Pic, workloads

pytestmark = pytest.mark.gpu
U = 2.0 ** -53
LD = np.longdouble
PI2 = 2 * LD("3.14159265358979323846264338327950288")


def _start(n, seed):
    x, v = inputs.particles(40 * n, seed=seed)
    edge = np.arange(n) / n
    x[:n, 0] = edge
    x[n:2 * n, 1] = np.nextafter(edge, 1.0)
    x[2 * n:3 * n, 2] = np.nextafter(np.roll(edge, -1) + (np.roll(edge, -1) == 0), 0.0)
    x[3 * n] = 0.0
    x[3 * n + 1] = np.nextafter(1.0, 0.0)
    return x, v


@pytest.mark.parametrize("t0", [0.0, 7.3])
@pytest.mark.parametrize("A,c", [(0.3, 0.1), (-0.3, -0.7), (0.0, 0.1), (0.5, 0.1), (0.9, 0.1)])
def test_drift(A, c, t0):
    import __graft_entry__ as g

    g.build()
    n = 6
    x, v = _start(n, 3)
    p = workloads.base(n, len(x), 0.05, 0, 1.0, qm=0.0, fx_amp=A, fx_speed=c)
    o = O.Oracle(p)
    o.set_state(x, v, t0=t0)
    xi = o.xi()[:, :3].astype(LD)
    o.sample(t0)  # (starts at v = v^M)
    vm = o.state()[1]
    with Pic(p) as s:
        s.set_state(x, v, t0=t0)
        s.step(1)
        x1, v1 = s.get_state()
    assert np.array_equal(v1, v)
    t = LD(t0) + LD(p["dt"]) / 2
    a = LD(A) / PI2
    T = xi - LD(c) * t - a * np.cos(PI2 * LD(c) * t)
    y = T.copy()
    for _ in range(60):
        y -= (y - a * np.cos(PI2 * y) - T) / (1 + LD(A) * np.sin(PI2 * y))
    sn = np.sin(PI2 * y)
    xd = LD(A) * LD(c) * (sn + np.sin(PI2 * LD(c) * t)) / (1 + LD(A) * sn)
    ref = x + LD(p["dt"]) * (v + xd - vm)
    slope = abs(c) * 2 * np.pi * abs(A) / (1 - abs(A)) ** 3
    # v^M itself: two inverse normals of 2 ulp
    bound = 4 * U + p["dt"] * U * (16 * (np.abs(v) + np.abs(vm) + abs(c)) + 8 * slope * (1 + abs(c) * (t0 + 1)))
    d = np.abs(x1 - ref)
    d = np.minimum(d, np.abs(1 - d))
    assert np.all(d <= bound), float((d / bound).max())
    assert np.all((x1 >= 0) & (x1 < 1))


@pytest.mark.parametrize("n", [2, 5, 8])
def test_lorentz_term(n):
    import __graft_entry__ as g

    g.build()
    x, v = _start(n, 4)
    p = workloads.base(n, len(x), 0.03, 0, 1.0, phi_amp=2.0)

    def lorentz(x, E, t):
        f = x * n
        i = np.minimum(np.floor(f).astype(int), n - 1)
        f = (f - i).astype(LD)
        E = np.asarray(E).reshape(n, n, n, 3).astype(LD)
        e = np.zeros((len(x), 3), LD)
        for q in range(8):
            b = np.array([q & 1, q >> 1 & 1, q >> 2])
            k = (i + b) % n
            w = np.prod(np.where(b, f, 1 - f), axis=1)
            e += w[:, None] * E[k[:, 2], k[:, 1], k[:, 0]]
        d = PI2 * (x.astype(LD) - np.array(p["phi_shift"]).astype(LD))
        s, c = np.sin(d), np.cos(d)
        amp = PI2 * LD(p["phi_amp"]) * np.exp(LD(t) / (2 * LD(p["phi_T"])))
        em = -amp * np.stack([c[:, 0] * s[:, 1] * s[:, 2], s[:, 0] * c[:, 1] * s[:, 2], s[:, 0] * s[:, 1] * c[:, 2]], 1)
        return LD(p["dt"]) * (e - em), p["dt"] * (np.abs(E).max() + float(amp))

    with Pic(p) as sim:
        sim.set_state(x, v, t0=0.2)
        L0, m0 = lorentz(x, sim.get_field()[2], 0.2)
        sim.step(1)
        x1, v1 = sim.get_state()
        L1, m1 = lorentz(x1, sim.get_field()[2], 0.2 + p["dt"])
    ref = v + (L0 + L1) / 2
    # weights from x n, whose rounding (n U) moves the field by a difference
    # of neighbouring nodes; 24 products and sums, three factors of 2 ulp
    bound = 4 * U * np.abs(v1) + (m0 + m1) * U * (64.0 + 8.0 * n)
    assert np.all(np.abs(v1 - ref) <= bound), float((np.abs(v1 - ref) / bound).max())
