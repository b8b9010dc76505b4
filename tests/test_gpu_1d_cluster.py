"""1D lattices on a cluster of CTAs: against the oracle (1e-12 in FP64, 1e-5 in FP32
deviations, the tolerances of the other 1D runs) and, bit for bit, one call of many
steps against as many calls of one step (other halo exchanges), over chunk sizes
with remainders, clusters of 1 to 16 CTAs, every level, both kinds of ends and
several instances; a run that fails inside a call stops at its failing step."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1905_04597_gb300 import glbm
from parity_helpers import oracle_moments, rel_errors

pytestmark = pytest.mark.gpu
TOL = {glbm.FP64: 1e-12, glbm.FP32_DEV: 1e-5}


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def _check(k, L, bc, prec, steps=37, n=1):
    N = k + 1
    cfgs = [dict(dims=1, nx=L, k=k, tau=0.7 + 0.2 * i, bc=bc, prec=prec) for i in range(n)]
    a, b = glbm.Lattice(cfgs), glbm.Lattice(cfgs)
    rng = np.random.default_rng(L + k)
    x = np.arange(L) / L
    fields = [(1 + 0.05 * np.sin(2 * np.pi * x + rng.uniform()),
               0.04 * np.cos(2 * np.pi * x + rng.uniform())) for _ in range(n)]
    for lat in (a, b):
        for i, f in enumerate(fields):
            lat.set_equilibrium(i, *f)
    n0 = a.kernel_launches
    a.step(steps)
    if prec == glbm.FP32_DEV or L <= 2560:
        assert a.kernel_launches - n0 == (1 if prec == glbm.FP32_DEV or L <= 3072 else n)
    for _ in range(steps):
        b.step(1)
    for i, f in enumerate(fields):
        np.testing.assert_array_equal(a.get_populations(i), b.get_populations(i))
        o = orc.Lattice(1, N, 0, L, 1, bc, cfgs[i]["tau"])
        X, _ = o.run(o.equilibrium(*f), steps)
        want, F = oracle_moments(o, X)
        errs = rel_errors(a.moments(i), want, dims=1, F=F)
        assert max(errs.values()) < TOL[prec], errs
    a.close()
    b.close()


PRECS = pytest.mark.parametrize("prec", [glbm.FP64, glbm.FP32_DEV])
ENDS = pytest.mark.parametrize("bc", [glbm.BC_BOUNCEBACK, glbm.BC_PERIODIC])


@PRECS
@ENDS
@pytest.mark.parametrize("k", range(8))
def test_levels(k, bc, prec):
    _check(k, 270 + k, bc, prec, n=2)


@PRECS
@ENDS
@pytest.mark.parametrize("L", [3, 31, 64, 129, 515, 1000, 3073])
def test_sizes(L, bc, prec):
    _check(2, L, bc, prec, steps=23)


@PRECS
def test_failing_step_inside_a_call(prec):
    """A density step too steep for D1Q3: the call and the one-step calls stop after
    the same step with the same state."""
    def make():
        lat = glbm.Lattice(dict(dims=1, nx=400, k=0, tau=0.02, prec=prec))
        rho = np.where(np.arange(400) < 200, 1.0, 0.01)
        lat.set_equilibrium(0, rho, np.zeros(400))
        return lat
    a, b = make(), make()
    with pytest.raises(glbm.UnstableError):
        a.step(400)
    with pytest.raises(glbm.UnstableError):
        for _ in range(400):
            b.step(1)
    assert 0 < a.time < 400 and a.time == b.time
    np.testing.assert_array_equal(a.get_populations(0), b.get_populations(0))
    a.close()
    b.close()


def test_calls_longer_than_one_launch():
    """A call of more steps than one launch takes equals the same steps in two calls."""
    cfg = dict(dims=1, nx=64, k=0, tau=0.8, prec=glbm.FP32_DEV)
    a, b = glbm.Lattice(cfg), glbm.Lattice(cfg)
    x = np.arange(64) / 64
    for lat in (a, b):
        lat.set_equilibrium(0, 1 + 0.05 * np.sin(2 * np.pi * x), np.zeros(64))
    n0 = a.kernel_launches
    a.step(65536 + 37)
    assert a.kernel_launches - n0 == 2 and a.time == 65536 + 37
    b.step(40000)
    b.step(25536 + 37)
    np.testing.assert_array_equal(a.get_populations(0), b.get_populations(0))
    a.close()
    b.close()
