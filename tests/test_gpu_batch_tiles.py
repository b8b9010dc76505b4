"""Batches whose levels overlap on three streams, bit for bit over 64 steps."""
import numpy as np
import pytest

from paper_1905_04597_gb300 import glbm, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("nx,ny", [(128, 320), (16, 20)])
def test_overlapping_levels(nx, ny):
    """Six levels on three streams, in a captured chunk and launched one by one: a call
    of 64 steps against calls of one step, bit for bit."""
    cfgs = [dict(dims=2, prec=glbm.FP32_DEV, k=k, nx=nx, ny=ny, kn=0.1, u_wall_lo=-0.04,
                 u_wall_hi=0.05) for k in range(2, 8)]
    a, b = glbm.Lattice(cfgs, hetero=True), glbm.Lattice(cfgs, hetero=True)
    for lat in (a, b):
        for i in range(6):
            lat.set_equilibrium(i, *inputs.random_macro(90 + i, nx, ny))
    a.step(64)
    for _ in range(64):
        b.step(1)
    for i in range(6):
        np.testing.assert_array_equal(a.get_populations(i), b.get_populations(i))
    a.close()
    b.close()
