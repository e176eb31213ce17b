"""A state in pid order in which cells outgrow their bins (precision form): the
caller's rows are read, or a state drawn, by one launch all the same (over the
uniform load one more launch moves the records). From pinned and device rows
the sorted state has the bits that pageable rows, which take no bins, give;
twice, since the second load finds v^M by pid. Sampling the paper's problem at
A(t) = 0.99 crowds its cells eightfold: the sort is by (cell, pid), and the
state is what its own rows load as."""
import numpy as np
import pytest

from paper_2602_15130_gb300 import Pic, workloads

pytestmark = pytest.mark.gpu


def _built():
    import __graft_entry__ as g

    g.build()


def _launches(sim, load):
    a = sim.stats()["kernel_launches"]
    load()
    return sim.stats()["kernel_launches"] - a


@pytest.mark.parametrize("memory", ["device", "pinned"])
@pytest.mark.parametrize("share", [0.01, 0.3, 1.0])
def test_crowded_rows(memory, share):
    import torch

    _built()
    n, count = 6, 6 ** 3 * 40 + 3
    rng = np.random.default_rng(5)
    even = rng.random((count, 3))
    v = rng.standard_normal((count, 3))
    x = even.copy()
    some = rng.random(count) < share
    x[some] = (np.array([1, 2, 3]) + rng.random((int(some.sum()), 3))) / n * (1.0 - 1e-12)
    p = workloads.mixed(workloads.base(n, count, 0.01, 0, 1.0))
    put = (lambda a: torch.from_numpy(a).cuda()) if memory == "device" else (lambda a: torch.from_numpy(a).pin_memory())
    with Pic(p) as sim, Pic(p) as plain:
        launches, binned = [], 0
        for rows in (even, even, x, x):
            c = np.minimum((rows * n).astype(int), n - 1) @ np.array([1, n, n * n])
            binned += np.bincount(c).max() <= 160  # four times the mean, rounded up to 32
            there = put(rows), put(v)
            launches.append(_launches(sim, lambda: sim.set_state(*there)))
            plain.set_state(rows, v)
            assert sim.stats()["binned_loads"] == binned
            for _ in range(2):  # as loaded, and a step later
                got, want = sim.get_state() + tuple(sim.get_sort()), plain.get_state() + tuple(plain.get_sort())
                for a, b in zip(got, want):
                    assert np.array_equal(a, b)
                sim.step(1)
                plain.step(1)
        assert launches[2] <= launches[1] + 1 and launches[3] <= launches[1] + 1


def test_crowded_sample():
    _built()
    p = workloads.mixed(workloads.paper_small(n_particles=20000, K=0, max_ppc=2048))
    with Pic(p) as sim, Pic(p) as plain:
        sim.sample_mms(1.6)
        cell, count, start, perm = sim.get_sort()
        assert count.max() > 160  # four times the mean, rounded up to 32
        assert np.array_equal(np.bincount(cell, minlength=512), count)
        assert np.array_equal(perm, np.lexsort((np.arange(20000), cell)))
        x, v = sim.get_state()
        plain.set_state(x, v, t0=1.6)
        for a, b in zip(sim.get_state(), plain.get_state()):
            assert np.array_equal(a, b)
        assert np.array_equal(sim.mms_error()["array"][[3, 4, 5, 10, 11, 12]],
                              plain.mms_error()["array"][[3, 4, 5, 10, 11, 12]])
