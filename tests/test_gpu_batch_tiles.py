"""Tile shapes a batch starts with at levels 6 and 7: by the padding and the number of
tiles, and bit for bit the uniform context's results (same G) over 64 steps."""
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


@pytest.mark.parametrize("k,nx,ny,n,shape", [
    (5, 32, 128, 16, (4, 2, 1)),     # half of a 64-column tile would be padding
    (5, 64, 128, 4, (4, 2, 1)),      # 512 tiles
    (5, 48, 128, 16, (4, 1, 2)),
    (5, 64, 128, 6, (4, 1, 2)),      # 768 tiles
    (5, 96, 100, 16, (4, 2, 1)),
    (5, 500, 100, 1, (4, 1, 2)),
    (6, 33, 20, 1, (5, 1, 1)),
    (6, 500, 30, 2, (5, 1, 1)),
])
def test_shape_and_state(k, nx, ny, n, shape):
    cfg = dict(dims=2, prec=glbm.FP32_DEV, k=k, nx=nx, ny=ny, kn=0.1, u_wall_lo=-0.05,
               u_wall_hi=0.05, g=1e-5)
    a, b = glbm.Lattice([cfg] * n, hetero=True), glbm.Lattice([cfg] * n)
    assert a.tile_shape(k) == shape
    for lat in (a, b):
        for i in range(n):
            lat.set_equilibrium(i, *inputs.random_macro(70 + i, nx, ny))
        lat.step(64)
    np.testing.assert_array_equal(a.get_populations(0), b.get_populations(0))
    np.testing.assert_array_equal(a.get_populations(n - 1), b.get_populations(n - 1))
    a.close()
    b.close()


def test_mixed_widths():
    """The choice counts every channel of the level, not those of other levels."""
    wide = dict(dims=2, prec=glbm.FP32_DEV, k=5, nx=512, ny=128, kn=0.1)
    narrow, other = dict(wide, nx=32), dict(wide, k=2, nx=32)
    for cfgs, shape in (([wide] * 2 + [other] * 20, (4, 1, 2)),
                        ([wide, narrow], (4, 1, 2)),
                        ([wide] + [narrow] * 8, (4, 2, 1))):
        lat = glbm.Lattice(cfgs, hetero=True)
        assert lat.tile_shape(5) == shape
        lat.close()


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
