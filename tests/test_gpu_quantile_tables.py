"""Sampling by the FP64 quantile tables (x^M from G^{-1}(T) - T, v^M from the
normal quantile with its tails beyond 2^-13 left to the general path) and by the
path that takes over where f_x is too sharp, and the error norms of both forms,
which use them too.

x^M against Newton in extended precision: T carries 2 roundings of 1 + |c t|,
times dG^{-1}/dT <= 1 / (1 - |A|), and the sum rounds twice. v^M against scipy's
quantile: 16 units of 2^-53 max(1, |z|) for both quantiles' few ulp."""
import numpy as np
import pytest
from scipy.special import ndtri

from oracle import oracle as O
from paper_2602_15130_gb300 import Pic, workloads

pytestmark = pytest.mark.gpu
U = 2.0 ** -53
LD = np.longdouble
PI2 = 2 * LD("3.14159265358979323846264338327950288")


@pytest.mark.parametrize("A,c,t0", [(0.3, 0.1, 0.0), (0.3, 0.1, 11.7), (-0.3, -0.7, 2.5), (0.0, 0.1, 0.4),
                                    (0.9, 0.1, 0.4)])
def test_sample_and_norms(A, c, t0):
    import __graft_entry__ as g

    g.build()
    n, N = 8, 60000  # about 15 values a component in the tails beyond 2^-13
    p = workloads.base(n, N, 0.01, 0, 1.0, fx_amp=A, fx_speed=c, seed=5, max_ppc=1024)
    o = O.Oracle(p)
    xi = o.xi()
    with Pic(p) as s:
        s.sample_mms(t0)
        x, v = s.get_state()
        e = s.mms_error()["array"]
    z = ndtri(xi[:, 3:])
    assert (np.abs(z) > 3.67).any()
    assert np.all(np.abs(v - (np.array(p["v_mean"]) + p["v_sigma"] * z)) <= 16 * U * np.maximum(1, np.abs(z)) + U * np.abs(v))
    t, a = LD(t0), LD(A) / PI2
    T = xi[:, :3].astype(LD) - LD(c) * t - a * np.cos(PI2 * LD(c) * t)
    y = T.copy()
    for _ in range(60):
        y -= (y - a * np.cos(PI2 * y) - T) / (1 + LD(A) * np.sin(PI2 * y))
    ref = y + LD(c) * t
    d = np.abs(x - (ref - np.floor(ref)))
    size = 1 + abs(c) * t0
    bound = U * size * (2 / (1 - abs(A)) + 3)
    assert np.all(np.minimum(d, 1 - d) <= bound)
    # a sampled state is the manufactured one: its norms are rounding
    assert np.all(e[:3] <= 2 * bound) and np.all(e[3:6] <= 1e-14)
    with Pic(workloads.mixed(p)) as s:
        s.sample_mms(t0)
        xm, vm = s.get_state()
        em = s.mms_error()["array"]
    # the precision form's norms, from its own FP32 state
    dx = xm - ref.astype(float)
    dx -= np.floor(dx + 0.5)
    dv = vm - v
    want = np.concatenate([np.sqrt((dx ** 2).mean(0)), np.sqrt((dv ** 2).mean(0))])
    assert np.all(np.abs(em[:6] - want) <= 1e-6 * want + 4 * bound)


@pytest.mark.parametrize("n,N,A,t0,mean", [(8, 200000, 0.3, 0.0, 0.2), (7, 200000, 0.3, 3.3, 0.0), (96, 400000, -0.3, 0.7, 0.2),
                                           (16, 100000, 0.9, 0.1, 0.2)])
def test_precision_sample_is_the_rounded_quantile(n, N, A, t0, mean):
    """The precision form samples cell and FP32 offset of x^M and the FP32 v^M:
    what rounding the FP64 form's values (equal to 1e-14) gives, to within one
    rounding wherever that difference can decide it."""
    import __graft_entry__ as g

    g.build()
    p = workloads.base(n, N, 0.01, 0, 1.0, fx_amp=A, seed=3, v_mean=(mean,) * 3, max_ppc=2048)
    with Pic(p) as s:
        s.sample_mms(t0)
        x, v = s.get_state()
    with Pic(workloads.mixed(p)) as s:
        s.sample_mms(t0)
        xm, vm = s.get_state()
    tol = 2e-14
    lo, hi = (v - tol * (1 + np.abs(v))).astype(np.float32), (v + tol * (1 + np.abs(v))).astype(np.float32)
    assert np.all((vm >= lo) & (vm <= hi))
    u = x * n
    c = np.floor(u)
    o = u - c
    inside = (o > 1e-9) & (o < 1 - 1e-7)
    lo, hi = (o - tol * n).astype(np.float32), (o + tol * n).astype(np.float32)
    om = xm * n - c
    # the state is the cell plus the offset times h: three roundings at most
    slack = 4 * U * n
    assert np.all(((om >= lo.astype(float) - slack) & (om <= hi.astype(float) + slack))[inside])
    assert inside.mean() > 0.999
