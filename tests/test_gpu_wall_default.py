"""The default way the wall densities are summed in FP32 where the tiles would repeat
them for a tenth to a fifth of a step's loads: dataflow chunks only where they were
measured faster than steps launched one after another, and for those a launch of the
sums only where it pays; the same states whichever way."""
import numpy as np
import pytest

from paper_1905_04597_gb300 import glbm, inputs

pytestmark = pytest.mark.gpu
ZV = dict(x_level=1, zv_axes=glbm.ZV_Y)


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


# (k, nx, ny, instances, kind) -> (dataflow, wall launch outside of chunks); ny gives a
# share of 2 V P / (ny Q_y), V the fastest speed and P the (velocity, row) pairs
@pytest.mark.parametrize("k,nx,ny,n,kw,want", [
    (2, 20, 40, 1, {}, (1, 0)),          # level 3: any size
    (2, 1000, 143, 3, ZV, (1, 0)),       # D1Q3 x D1Q8, 10.3 M populations
    (3, 64, 70, 1, {}, (0, 0)),          # D2Q81, 0.36 M
    (3, 1000, 59, 1, {}, (1, 0)),        # 4.8 M
    (3, 1000, 59, 2, {}, (1, 1)),        # 9.6 M
    (4, 256, 100, 1, {}, (1, 0)),        # D2Q121, 3.1 M
    (5, 256, 129, 1, {}, (1, 1)),        # D2Q169, 5.6 M
    (5, 64, 129, 1, {}, (0, 0)),         # 1.4 M
    (5, 1000, 99, 2, {}, (0, 1)),        # 33 M
    (7, 64, 1020, 1, ZV, (0, 1)),        # D1Q3 x D1Q18, 3.5 M
    (5, 200, 80, 1, dict(zv_axes=glbm.ZV_X | glbm.ZV_Y), (0, 1)),  # above a fifth
    (5, 128, 500, 1, dict(zv_axes=glbm.ZV_X | glbm.ZV_Y), (1, 1)),  # D2Q196, 12.5 M
    (4, 1000, 90, 2, dict(force=glbm.FORCE_GUO), (0, 1)),  # Guo, 21.8 M
    (3, 1000, 120, 1, {}, (1, 0)),       # a share below a tenth
    (3, 1000, 40, 1, {}, (0, 1)),        # above a fifth
])
def test_default(k, nx, ny, n, kw, want):
    cfg = dict(dims=2, nx=nx, ny=ny, k=k, kn=0.2, prec=glbm.FP32_DEV, u_wall_lo=-0.03,
               u_wall_hi=0.05, g=2e-5, **kw)
    lats = [glbm.Lattice([cfg] * n) for _ in range(4)]
    a, b, c, d = lats
    assert a.dataflow == want[0] and a.wall_launch == (0 if want[0] else want[1])
    b.set_dataflow(0)
    assert b.wall_launch == want[1]
    c.set_wall_launch(1)
    d.set_wall_launch(0)
    for lat in lats:
        for i in range(n):
            lat.set_equilibrium(i, *inputs.random_macro(40 + i, nx, ny))
    n0 = a.kernel_launches
    a.step(1)
    assert a.kernel_launches - n0 == 1 + want[1]  # one step is not a chunk
    a.step(69)
    for lat in lats[1:]:
        lat.step(70)
    f = a.get_populations(n - 1)
    for lat in lats[1:]:
        np.testing.assert_array_equal(f, lat.get_populations(n - 1))
    a.set_wall_launch(-1)
    assert a.dataflow == want[0]
    for lat in lats:
        lat.close()


def test_adjoint_takes_the_launch():
    """The adjoint's steps are launched one after another: forward, two launches a
    step from level 6 on, the same gradients."""
    cfg = dict(dims=2, nx=256, ny=129, k=5, kn=0.1, prec=glbm.FP32_DEV, g=1e-5)
    out = []
    for mode in (-1, 0):
        lat = glbm.Lattice(cfg)
        lat.set_wall_launch(mode)
        n0 = lat.kernel_launches
        out.append(lat.adjoint_flowrate(4, ckpt_every=4, walls=True))
        out.append(lat.kernel_launches - n0)
        lat.close()
    assert out[1] - out[3] == 4
    for x, y in zip(out[0], out[2]):
        np.testing.assert_array_equal(x, y)
