"""The moment reducers of FP32 deviations (integer digits with a float
remainder, wall densities from a launch of their own, fields written straight to
the caller's memory) against the oracle's moments of the same stored
populations: every x level and hierarchy, ragged and one-column lattices, few
rows, walls and periodic boundaries, 3D, and deviations beyond the digits'
range. Both sides sum at most 343 terms of one node in FP64 or more exactly,
so they agree to 343 x 2^-53 = 4e-14 of the terms' scale each; 1e-12 is asked."""
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


def _check(cfg, scale, spread=0.5, **orc_kw):
    import torch
    N = cfg["k"] + 1
    lat = glbm.Lattice(dict(cfg, prec=glbm.FP32_DEV, tau=0.9))
    Q, shape = lat.nq(), lat.shape()
    f = inputs.random_populations(31 + N, Q, int(np.prod(shape)), 1, 1 - spread, 1 + spread)
    lat.set_populations(0, scale * f.reshape((Q,) + shape))
    X = lat.get_populations(0)
    bc = cfg.get("bc", glbm.BC_WALLS)
    d3 = cfg["dims"] == 3
    o = orc.Lattice(cfg["dims"], cfg.get("x_level") or N, N, cfg["nx"], cfg["ny"], bc, 0.9,
                    cfg.get("u_wall_lo", 0.0), cfg.get("u_wall_hi", 0.0), 0.0,
                    zv=cfg.get("zv_axes", 0), NZ=N if d3 else 0, Lz=cfg.get("nz", 1))
    want, F = oracle_moments(o, X)
    out = torch.full((len(want),) + shape, float("nan"), dtype=torch.float64, device="cuda")
    got = lat.moments(0, out=out).cpu().numpy()
    host = lat.moments(0)
    names = glbm.FIELDS_3D if d3 else glbm.FIELDS_2D
    errs = rel_errors(dict(zip(names, got)), want, dims=cfg["dims"], F=F,
                      **({} if d3 else dict(q1x=o.cfg.NX * 2 + (2 if o.cfg.zv & 1 else 1),
                                            zv=o.cfg.zv)))
    assert max(errs.values()) < 1e-12, errs
    for i, name in enumerate(names):  # the host call and a few fields alone give the same bits
        assert np.array_equal(host[name], got[i]), name
    mask = glbm.M_UX | glbm.M_QY
    few = lat.moments(0, mask=mask)
    assert np.array_equal(few["ux"], host["ux"]) and np.array_equal(few["qy"], host["qy"])
    mass, jx, jy = lat.conservation(0)
    assert mass == pytest.approx(want[0].sum(), rel=1e-12)
    assert jx == pytest.approx((want[0] * want[1]).sum(), abs=1e-12 * mass)
    assert jy == pytest.approx((want[0] * want[2]).sum(), abs=1e-12 * mass)
    lat.close()


WALLS = dict(u_wall_lo=-0.03, u_wall_hi=0.05)


@pytest.mark.parametrize("k", range(8))
@pytest.mark.parametrize("kind", ["iso", "d1q3", "zv", "zvxy"])
def test_kinds(k, kind):
    kw = {"iso": {}, "d1q3": dict(x_level=1), "zv": dict(x_level=1, zv_axes=glbm.ZV_Y),
          "zvxy": dict(zv_axes=glbm.ZV_X | glbm.ZV_Y)}[kind]
    _check(dict(dims=2, nx=33 + k, ny=2 * k + 5, k=k, **WALLS, **kw), 1.0)


@pytest.mark.parametrize("nx,ny", [(1, 31), (3, 5), (70, 4), (64, 33)])
@pytest.mark.parametrize("bc", [glbm.BC_WALLS, glbm.BC_PERIODIC])
@pytest.mark.parametrize("scale", [1.0, 40.0])
def test_shapes_and_large_deviations(nx, ny, bc, scale):
    """scale 40: deviations of the central velocities beyond 2."""
    wall = WALLS if bc == glbm.BC_WALLS else {}
    _check(dict(dims=2, nx=nx, ny=ny, k=3, bc=bc, **wall), scale)


def test_highest_level():
    _check(dict(dims=2, nx=2, ny=29, k=12, x_level=1, zv_axes=glbm.ZV_Y, **WALLS), 1.0)


@pytest.mark.parametrize("k", [0, 1, 2])
@pytest.mark.parametrize("scale", [1.0, 60.0])
@pytest.mark.parametrize("bc", [glbm.BC_WALLS, glbm.BC_PERIODIC])
def test_3d(k, scale, bc):
    wall = WALLS if bc == glbm.BC_WALLS else {}
    _check(dict(dims=3, nx=13, ny=6, nz=5, k=k, bc=bc, **wall), scale)


def test_non_finite_values_are_reported():
    """An infinite or NaN deviation reaches the nodes that pull it, and no other."""
    lat = glbm.Lattice(dict(dims=2, nx=9, ny=9, k=1, bc=glbm.BC_PERIODIC, prec=glbm.FP32_DEV,
                            tau=0.9))
    f = lat.get_populations(0)
    f[12, 4, 4] = np.inf   # velocity (0, 0)
    f[12, 2, 2] = np.nan
    lat.set_populations(0, f)
    rho = lat.moments(0)["rho"]
    assert np.isinf(rho[4, 4]) and np.isnan(rho[2, 2])
    assert np.isfinite(rho).sum() == 79
    lat.close()
