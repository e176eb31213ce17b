"""The precision form's plain Poisson solve at the edges of its launch shapes
(a cluster of 4, 8 or 16 blocks: edges at 1,024 and 2,048 nodes; 1, 2 or 4
nodes a thread: edges at 16,384 and 32,768; the grid beyond 65,536) against an FFT solve of the same discrete system in FP64.

phi - phi_exact = A^-1 r: the stop gives tol ||b|| / lambda_min; FP32 adds the
rounding of b (eight operations on rho), and the residual's drift from b - A x,
at most a unit in the last place of ||A|| ||phi|| an operation, 20 of them."""
import numpy as np
import pytest

import inputs
from paper_2602_15130_gb300 import Pic, workloads
from test_gpu_cg_shapes import _rhs

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -24


@pytest.mark.parametrize("n", [2, 3, 7, 8, 10, 11, 12, 13, 25, 26, 31, 33, 40, 41])
def test_precision_solve_matches_fft_at_every_launch_shape(n):
    import __graft_entry__ as g

    g.build()
    p = workloads.mixed(workloads.base(n, 4 * n ** 2 + 7, 0.01, 0, 1.0, cg_tol=1e-10))
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
            ref = np.fft.ifftn(bh / lam).real.ravel()
            bound = (p["cg_tol"] * np.linalg.norm(b) + 8 * EPS * np.linalg.norm(np.abs(rho) / p["eps0"] + 1.0)
                     + 20 * EPS * 12.0 * n * n * np.linalg.norm(ref)) / lam_min
            assert np.linalg.norm(phi - ref) <= bound
            assert sim.stats()["cg_iters_last"] > 0
            f = phi.reshape(n, n, n)
            for d, axis in enumerate((2, 1, 0)):
                e = (np.roll(f, 1, axis) - np.roll(f, -1, axis)) * (0.5 * n)
                assert np.abs(E[:, d] - e.ravel()).max() <= 8.0 * EPS * n * np.abs(phi).max()
