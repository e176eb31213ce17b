"""A caller's allocator of 8- and 16-byte granules: each block starts just
beside a 32-byte boundary, the widest access of the kernels. Both forms and a
batch give the bits that they give on torch's own blocks, and every block goes
back under the address the allocator gave."""
import numpy as np
import pytest

import inputs
import paper_2602_15130_gb300 as M
from paper_2602_15130_gb300 import Batch, Pic, workloads

pytestmark = pytest.mark.gpu


def _run(form):
    import torch

    if form == "batch":
        ps = [workloads.mixed(workloads.smallest(n=n, n_particles=n ** 3 * 10 + n, seed=n)) for n in (4, 8)]
        with Batch(ps) as b:
            b.sample_mms(0.0)
            b.step(3)
            return [a for r in range(2) for a in b.get_state(r)]
    n = 16 if form == "precision" else 8  # 2^k >= 16: the multigrid levels too
    p = workloads.smallest(n=n, n_particles=n ** 3 * 9 + 5)
    if form == "precision":
        p = workloads.mixed(p)
    x, v = inputs.particles(p["n_particles"], seed=3)
    with Pic(p) as s:
        s.sample_mms(0.0)
        s.step(1)
        s.set_state(torch.from_numpy(x).cuda(), torch.from_numpy(v).cuda())  # in place: records and bins
        s.step(2)
        out = tuple(torch.zeros(len(x), 3, dtype=torch.float64, device="cuda") for _ in range(2))
        s.get_state(out=out)
        return [a.cpu().numpy() for a in out] + list(s.get_state()) + list(s.get_field()) + list(s.collide_avg(0))


@pytest.mark.parametrize("form", ["fp64", "precision", "batch"])
@pytest.mark.parametrize("granule", [8, 16])
def test_small_granules(form, granule, monkeypatch):
    import torch

    import __graft_entry__ as g

    g.build()
    want = _run(form)
    live = {}

    def alloc(self, user, nbytes):
        block = torch.empty(int(nbytes) + 64, dtype=torch.uint8, device="cuda")
        at = (block.data_ptr() + 31) // 32 * 32 + granule
        live[at] = block
        return at

    def free(self, user, ptr):
        del live[ptr]

    monkeypatch.setattr(M._TorchAllocator, "_alloc", alloc)
    monkeypatch.setattr(M._TorchAllocator, "_free", free)
    got = _run(form)
    assert not live
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
