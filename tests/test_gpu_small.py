"""The FP64 step of small lattices (one thread per node and velocity row) against
the tiles: bit-identical populations after single steps and graph chunks, on every
lattice kind and level, one-column and ragged lattices, as few rows as the walls
allow, several instances, walls (wall densities summed by the node's threads)
and periodic boundaries; the failure contract and the adjoint on top of it."""
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


def _pair(cfgs):
    """A context as created and one on the level's default tile."""
    out = []
    for tiles in (False, True):
        lat = glbm.Lattice(cfgs)
        assert lat.dataflow == 0  # the small step
        if tiles:
            lat.set_tiles([0] * glbm.LEVELS)
        for i, c in enumerate(cfgs):
            lat.set_equilibrium(i, *inputs.random_macro(900 + 3 * i, c["nx"], c["ny"]))
        out.append(lat)
    return out


def _check(cfgs, steps=(1, 5, 66)):
    a, b = _pair(cfgs)
    for n in steps:
        a.step(n)
        b.step(n)
        for i in range(len(cfgs)):
            np.testing.assert_array_equal(a.get_populations(i), b.get_populations(i))
    a.close()
    b.close()


def _cfgs(n=2, **kw):
    return [dict(dims=2, prec=glbm.FP64, kn=0.2 * (i + 1), **kw) for i in range(n)]


WALLS = dict(u_wall_lo=-0.03, u_wall_hi=0.05, g=2e-5)


@pytest.mark.parametrize("k", range(8))
@pytest.mark.parametrize("kind", ["iso", "d1q3", "zv", "zvxy"])
def test_kinds(k, kind):
    kw = {"iso": {}, "d1q3": dict(x_level=1), "zv": dict(x_level=1, zv_axes=glbm.ZV_Y),
          "zvxy": dict(zv_axes=glbm.ZV_X | glbm.ZV_Y)}[kind]
    _check(_cfgs(nx=13, ny=2 * k + 4, k=k, **WALLS, **kw), steps=(1, 6))


@pytest.mark.parametrize("k", range(8, 13))
def test_high_levels(k):
    _check(_cfgs(nx=3, ny=2 * k + 5, k=k, x_level=1, zv_axes=glbm.ZV_Y, **WALLS), steps=(1, 6))


@pytest.mark.parametrize("nx,ny", [(1, 40), (5, 3), (33, 4), (40, 24)])
@pytest.mark.parametrize("bc", [glbm.BC_WALLS, glbm.BC_PERIODIC])
@pytest.mark.parametrize("g", [0.0, 2e-5])
def test_shapes(nx, ny, bc, g):
    wall = dict(u_wall_lo=-0.03, u_wall_hi=0.05) if bc == glbm.BC_WALLS else {}
    _check(_cfgs(n=3, nx=nx, ny=ny, k=2, bc=bc, g=g, **wall))


def test_failure_contract():
    """k = 0, g = 0.01: step 83 fails, inside a graph chunk; later steps do nothing."""
    lat = glbm.Lattice(dict(dims=2, nx=9, ny=8, k=0, tau=0.8, bc=glbm.BC_PERIODIC, g=0.01,
                            prec=glbm.FP64))
    assert lat.dataflow == 0
    with pytest.raises(glbm.UnstableError, match="83 of 200 steps completed"):
        lat.step(200)
    assert lat.time == 83
    np.testing.assert_allclose(lat.moments(0)["ux"], 0.83, rtol=1e-6)
    with pytest.raises(glbm.UnstableError, match="0 of 10 steps completed"):
        lat.step(10)
    lat.close()


def test_large_lattices_and_explicit_choices_take_the_tiles():
    big = glbm.Lattice(dict(dims=2, nx=512, ny=128, k=3, tau=0.8, prec=glbm.FP64))
    assert big.dataflow == 1
    big.close()
    lat = glbm.Lattice(dict(dims=2, nx=32, ny=64, k=1, tau=0.8, prec=glbm.FP64))
    lat.set_dataflow(1)
    lat.set_wall_launch(0)
    assert lat.dataflow == 1
    lat.close()
