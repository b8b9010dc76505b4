"""The FP64 step's rows of 16 and more populations (relaxed one after the other) and the
shorter ones beside them, with and without a force, linear and Guo's: against the
oracle to 1e-12, as the other FP64 runs."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1905_04597_gb300 import glbm, inputs
from parity_helpers import oracle_moments, rel_errors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("g", [0.0, 3e-5])
@pytest.mark.parametrize("k,zv", [(6, 0), (7, 0), (5, 3), (6, 3), (7, 3)])
def test_rows(k, zv, g):
    nx, ny, steps, N = 70, 2 * k + 12, 6, k + 1
    lat = glbm.Lattice(dict(dims=2, nx=nx, ny=ny, k=k, tau=0.8, u_wall_lo=-0.03, u_wall_hi=0.04, g=g,
                            zv_axes=zv))
    lat.set_dataflow(1)  # the tiles, however small the lattice
    fields = inputs.random_macro(60 + k, nx, ny)
    lat.set_equilibrium(0, *fields)
    lat.step(steps)
    o = orc.Lattice(2, N, N, nx, ny, orc.BC_WALLS, 0.8, -0.03, 0.04, g, zv=zv)
    X, _ = o.run(o.equilibrium(*fields), steps)
    want, F = oracle_moments(o, X)
    errs = rel_errors(lat.moments(0), want, F=F, q1x=2 * N + 1 + (zv > 0), zv=zv)
    assert max(errs.values()) < 1e-12, errs
    lat.close()
