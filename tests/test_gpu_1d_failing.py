"""1D calls of several instances that fail: the call ends soon after the failing step
however many steps it asked for, and leaves what the single contexts leave, also when
the failing step lies behind the first of the call's launches (2^16 steps each)."""
import time

import numpy as np
import pytest

from paper_1905_04597_gb300 import glbm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def _steep(i):
    return np.where(np.arange(64) < 32, 1.0, 0.01 + 0.002 * i), np.zeros(64)


def test_call_ends_soon_after_the_failing_step():
    """Both instances fail within a few steps of a call of 2^24: one launch of 2^16
    steps (at most 24 ms) and the repeat, where 2^24 steps take more than 3 s."""
    cfg = dict(dims=1, nx=64, k=0, tau=0.02, prec=glbm.FP32_DEV)
    lat, one = glbm.Lattice([cfg, cfg]), glbm.Lattice(cfg)
    for i in range(2):
        lat.set_equilibrium(i, *_steep(i))
    one.set_equilibrium(0, *_steep(0))
    with pytest.raises(glbm.UnstableError):
        one.step(400)
    t0 = time.perf_counter()
    with pytest.raises(glbm.UnstableError):
        lat.step(1 << 24)
    assert time.perf_counter() - t0 < 1.0
    np.testing.assert_array_equal(lat.get_populations(0), one.get_populations(0))
    lat.close()
    one.close()


@pytest.mark.parametrize("failing", [0, 1])
def test_late_failure(failing):
    """A uniform flow just beyond linear stability leaves the domain after some 10^5
    steps; beside it an instance at rest. The failing one stops where it stops alone,
    the one before it has taken every step, the one behind it none."""
    n, L = 200000, 16
    cfgs = [dict(dims=1, nx=L, k=0, tau=0.8, bc=glbm.BC_PERIODIC)] * 2
    cfgs[failing] = dict(cfgs[0], tau=5e-5)
    rho = 1 + 1e-7 * np.random.default_rng(1).standard_normal(L)
    fields = [(1 + 0.05 * np.sin(2 * np.pi * np.arange(L) / L), np.zeros(L))] * 2
    fields[failing] = (rho, np.full(L, 0.43))
    lat = glbm.Lattice(cfgs)
    alone = [glbm.Lattice(c) for c in cfgs]
    for i, f in enumerate(fields):
        lat.set_equilibrium(i, *f)
        alone[i].set_equilibrium(0, *f)
    with pytest.raises(glbm.UnstableError):
        alone[failing].step(n)
    stop = alone[failing].time
    assert 1 << 16 < stop < n
    if failing == 1:
        alone[0].step(n)
    with pytest.raises(glbm.UnstableError):
        lat.step(n)
    assert lat.time == (stop if failing == 1 else 0)
    for i in range(2):
        np.testing.assert_array_equal(lat.get_populations(i), alone[i].get_populations(0))
    for x in [lat] + alone:
        x.close()


def test_long_call_through_three_buffers():
    """A call of several launches, then shorter ones: the same states as in single
    contexts."""
    cfgs = [dict(dims=1, nx=40, k=1, tau=0.6 + 0.3 * i, prec=glbm.FP32_DEV)
            for i in range(3)]
    x = np.arange(40) / 40
    lat = glbm.Lattice(cfgs)
    for i in range(3):
        lat.set_equilibrium(i, 1 + 0.04 * np.sin(2 * np.pi * x + i), np.zeros(40))
    calls = [(1 << 16) + 5, 3, (1 << 17) + 1]
    for m in calls:
        lat.step(m)
    assert lat.time == sum(calls)
    for i, c in enumerate(cfgs):
        one = glbm.Lattice(c)
        one.set_equilibrium(0, 1 + 0.04 * np.sin(2 * np.pi * x + i), np.zeros(40))
        one.step(sum(calls))
        np.testing.assert_array_equal(lat.get_populations(i), one.get_populations(0))
        one.close()
    lat.close()


def test_two_threads_with_lattices_of_different_size():
    """The repeat of failing runs in one CTA sets its kernel's shared-memory limit: a
    small lattice in one thread must not refuse the launch of a large one in another."""
    import threading

    import torch
    errors = []

    def work(L):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                lat = glbm.Lattice(dict(dims=1, nx=L, k=0, tau=0.02))
                rho = torch.where(torch.arange(L, device="cuda") < L // 2, 1.0, 0.01).double()
                u = torch.zeros(L, dtype=torch.float64, device="cuda")
                for _ in range(2000):
                    lat.set_equilibrium(0, rho, u)
                    try:
                        lat.step(40)
                        errors.append("no failure")
                    except glbm.UnstableError:
                        pass
                lat.close()
        except Exception as e:
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=(L,)) for L in (40, 2000)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]
