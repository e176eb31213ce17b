"""The FP64 Poisson solve at the edges of its launch shapes (one cluster up to
8,192 nodes; a grid with 1, 2, 4 or 8 nodes a thread, edges at 77,824,
155,648, 311,296 and 622,592 nodes on 152 SMs; vectors in memory beyond)
against an FFT solve of the same discrete system.

The solve stops at ||r|| <= tol ||b||, and phi - phi_exact = A^-1 r, so
||phi - phi_exact|| <= tol ||b|| / lambda_min; the 1e-12 ||phi|| beside it is
the FFT's and the recurrence's rounding (some hundred operations of 2^-53)."""
import numpy as np
import pytest

import inputs
from paper_2602_15130_gb300 import Pic, workloads

pytestmark = pytest.mark.gpu

TOL = 1e-10


def _rhs(p, rho, t):
    n, tau = p["n"], 2.0 * np.pi
    g = np.arange(n) / n
    s = [np.sin(tau * (g - sh)) for sh in p["phi_shift"]]
    f = 1.0 + p["fx_amp"] * np.sin(tau * (g - p["fx_speed"] * t))
    phi_m = p["phi_amp"] * np.exp(t / (2.0 * p["phi_T"])) * \
        (s[2][:, None, None] * s[1][None, :, None] * s[0][None, None, :]).ravel()
    rho_m = p["q"] * (f[:, None, None] * f[None, :, None] * f[None, None, :]).ravel()
    b = rho / p["eps0"] + 3.0 * tau ** 2 * phi_m - rho_m / p["eps0"]
    return b - b.mean()


@pytest.mark.parametrize("n", [2, 3, 8, 20, 21, 42, 43, 53, 54, 67, 68, 85, 86])
def test_solve_matches_fft_at_every_launch_shape(n):
    import __graft_entry__ as g

    g.build()
    p = workloads.base(n, 4 * n ** 2 + 7, 0.01, 0, 1.0, cg_tol=TOL)
    x, v = inputs.particles(p["n_particles"], seed=n)
    with Pic(p) as sim:
        for t0 in (0.0, 0.3):  # a cold and a warm start
            sim.set_state(x, v, t0=t0)
            rho, phi, E = sim.get_field()
            b = _rhs(p, rho, t0)
            lam = 2.0 * n * n * (1.0 - np.cos(2.0 * np.pi * np.arange(n) / n))
            lam = lam[:, None, None] + lam[None, :, None] + lam[None, None, :]
            lam_min = np.sort(lam.ravel())[1]
            lam[0, 0, 0] = 1.0
            bh = np.fft.fftn(b.reshape(n, n, n))
            bh[0, 0, 0] = 0.0
            ref = np.fft.ifftn(bh / lam).real
            bound = TOL * np.linalg.norm(b) / lam_min + 1e-12 * np.linalg.norm(ref)
            assert np.linalg.norm(phi - ref.ravel()) <= bound
            f = phi.reshape(n, n, n)
            for d, axis in enumerate((2, 1, 0)):
                e = (np.roll(f, 1, axis) - np.roll(f, -1, axis)) * (0.5 * n)
                assert np.abs(E[:, d] - e.ravel()).max() <= 8.0 * 2.0 ** -53 * n * np.abs(phi).max()
