"""The initial equilibrium (float-pair arithmetic in FP32 deviations) against the
oracle's: a stored deviation is the exact one rounded once, so it differs from the
oracle's FP64 value by at most half a float ulp of the deviation (2^-24 of it) plus the FP64 roundings of f and of the oracle's
factorial sums (1e-14 of the largest population); FP64 storage by the latter alone.
Every lattice kind, 1D to 3D, ragged sizes, the rest state exactly, and fields
beyond the pairs' range."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1905_04597_gb300 import glbm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def _check(cfg, prec, amp=0.05, edit=None):
    N, d = cfg["k"] + 1, cfg["dims"]
    lat = glbm.Lattice(dict(cfg, prec=prec, tau=0.9))
    rest = lat.get_populations(0)
    shape = lat.shape()
    rng = np.random.default_rng(7 + N)
    fields = [1 + amp * rng.standard_normal(shape)] + \
        [amp * rng.standard_normal(shape) for _ in range(d)]
    if edit:
        edit(fields)
    lat.set_equilibrium(0, *fields)
    got = lat.get_populations(0)
    o = orc.Lattice(d, cfg.get("x_level") or N, N, cfg["nx"], cfg.get("ny", 1),
                    orc.BC_BOUNCEBACK if d == 1 else orc.BC_WALLS, 0.9,
                    zv=cfg.get("zv_axes", 0), NZ=N if d == 3 else 0, Lz=cfg.get("nz", 1))
    want = o.equilibrium(*fields)
    one, zero = np.ones(shape), np.zeros(shape)
    W = o.equilibrium(one, *[zero] * d)
    tol = 1e-14 * np.abs(want).max(axis=0)
    if prec == glbm.FP32_DEV:
        tol = tol + 2.0 ** -24 * np.abs(want - W) + 1e-45
    assert (np.abs(got - want) <= tol).all(), float((np.abs(got - want) - tol).max())
    assert np.abs(rest - W).max() < 1e-15  # the rest state of a new context
    lat.set_equilibrium(0, one, *[zero] * d)
    assert np.array_equal(lat.get_populations(0), rest)
    lat.close()


PRECS = pytest.mark.parametrize("prec", [glbm.FP64, glbm.FP32_DEV])


@PRECS
@pytest.mark.parametrize("k", [0, 3, 7])
@pytest.mark.parametrize("kind", ["iso", "d1q3", "zv", "zvxy"])
def test_2d(kind, k, prec):
    kw = {"iso": {}, "d1q3": dict(x_level=1), "zv": dict(x_level=1, zv_axes=glbm.ZV_Y),
          "zvxy": dict(zv_axes=glbm.ZV_X | glbm.ZV_Y)}[kind]
    _check(dict(dims=2, nx=37, ny=2 * k + 4, k=k, **kw), prec)


@PRECS
def test_1d_3d_and_the_highest_level(prec):
    _check(dict(dims=1, nx=45, k=7), prec)
    _check(dict(dims=3, nx=11, ny=5, nz=3, k=2), prec)
    _check(dict(dims=2, nx=1, ny=28, k=12, x_level=1, zv_axes=glbm.ZV_Y), prec)


@PRECS
def test_fields_beyond_the_float_pairs(prec):
    def edit(f):
        f[0][0, 0], f[1][0, 1], f[2][1, 1] = 3e19, 1e-25, -1e-30
        f[0][2, 2], f[1][2, 2] = 1e-19, 0.0
    _check(dict(dims=2, nx=9, ny=4, k=2), prec, edit=edit)


def test_float_pairs_round_like_fp64():
    """The stored deviations are the FP64 formula's, rounded: against the deviations
    of an FP64 context (E^x A there, so equal up to the rounding of its f ~ W) no
    stored float may be further than half an ulp plus 2^-50 W."""
    nx, ny, k = 700, 300, 3
    rng = np.random.default_rng(11)
    fields = [1 + 0.03 * rng.standard_normal((ny, nx))] + \
        [0.04 * rng.standard_normal((ny, nx)) for _ in range(2)]
    a = glbm.Lattice(dict(dims=2, nx=nx, ny=ny, k=k, tau=0.9, prec=glbm.FP32_DEV))
    b = glbm.Lattice(dict(dims=2, nx=nx, ny=ny, k=k, tau=0.9, prec=glbm.FP64))
    W = b.get_populations(0)
    for lat in (a, b):
        lat.set_equilibrium(0, *fields)
    stored = np.empty((81, ny, nx), np.float32)
    a.pack_columns(0, 0, nx, stored)
    d = b.get_populations(0) - W
    s = stored.astype(np.float64)
    ulp = np.spacing(np.abs(stored)).astype(np.float64)
    assert (np.abs(s - d) <= 0.5 * ulp + 2.0 ** -50 * W).all()
    a.close()
    b.close()


def test_infinite_and_nan_fields_stay_in_their_node():
    lat = glbm.Lattice(dict(dims=2, nx=40, ny=6, k=2, tau=0.9, prec=glbm.FP32_DEV))
    rho, u = np.ones((6, 40)), np.zeros((6, 40))
    rho[1, 3], rho[4, 35] = np.inf, np.nan
    lat.set_equilibrium(0, rho, u, u)
    f = lat.get_populations(0)
    bad = ~np.isfinite(f).all(axis=0)
    assert bad[1, 3] and bad[4, 35] and bad.sum() == 2
    assert np.isnan(f[:, 4, 35]).all()
    lat.close()
