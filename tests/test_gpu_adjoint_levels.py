"""The adjoint step's tiles at every level (rows dealt to 1 to 6 warps), ragged and
narrow lattices, few rows, walls and periodic boundaries, segments whose states
come from the forward run or from a recompute, and deviations beyond the integer
digits of the forward moments: against the oracle's forward-mode dual numbers
(1e-9 in FP64, as for the other levels; 1e-4 from FP32 states). A run that leaves
the positivity domain stops as glbm_step does."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1905_04597_gb300 import glbm, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def _compare(cfg, steps, ckpt, rho_scale=1.0):
    N = cfg["k"] + 1
    rtol = 1e-9 if cfg["prec"] == glbm.FP64 else 1e-4
    rho, ux, uy = inputs.random_macro(130 + N, cfg["nx"], cfg["ny"])
    fields = (rho_scale * rho, ux, uy)
    lat = glbm.Lattice(cfg)
    lat.set_equilibrium(0, *fields)
    got = lat.adjoint_flowrate(steps, ckpt, walls=True)
    assert lat.time == steps
    ref = glbm.Lattice(cfg)  # the state afterwards is that of the plain steps
    ref.set_equilibrium(0, *fields)
    ref.step(steps)
    assert np.array_equal(lat.get_populations(0), ref.get_populations(0))
    bc = cfg.get("bc", orc.BC_WALLS)
    o = orc.Lattice(2, N, N, cfg["nx"], cfg["ny"], bc, cfg["tau"], cfg.get("u_wall_lo", 0.0),
                    cfg.get("u_wall_hi", 0.0), cfg.get("g", 0.0))
    want = o.flowrate_grad(o.equilibrium(*fields), steps, walls=True)
    for k, (g, w) in enumerate(zip(got, want)):
        if k >= 3 and bc != orc.BC_WALLS:
            assert g[0] == 0.0 and w == 0.0
        else:
            assert g[0] == pytest.approx(w, rel=rtol), k
    lat.close()
    ref.close()


@pytest.mark.parametrize("k", range(8))
@pytest.mark.parametrize("prec", [glbm.FP64, glbm.FP32_DEV])
def test_every_level(k, prec):
    cfg = dict(dims=2, nx=35, ny=k + 3, k=k, tau=0.8, prec=prec, u_wall_lo=-0.02, u_wall_hi=0.04,
               g=3e-5)
    _compare(cfg, 9, 4)


@pytest.mark.parametrize("nx,ny,ckpt", [(1, 9, 3), (5, 3, 100), (64, 4, 5)])
@pytest.mark.parametrize("bc", [glbm.BC_WALLS, glbm.BC_PERIODIC])
def test_narrow_lattices(nx, ny, ckpt, bc):
    cfg = dict(dims=2, nx=nx, ny=ny, k=2, tau=1.1, prec=glbm.FP64, bc=bc, g=1e-5)
    if bc == glbm.BC_WALLS:
        cfg.update(u_wall_lo=0.03, u_wall_hi=-0.01)
    _compare(cfg, 10, ckpt)


def test_deviations_beyond_the_digits():
    _compare(dict(dims=2, nx=20, ny=11, k=1, tau=0.9, prec=glbm.FP32_DEV, u_wall_hi=0.03, g=1e-5),
             8, 3, rho_scale=7.0)


@pytest.mark.parametrize("ckpt", [4, 100])
def test_failing_step(ckpt):
    k, nx, ny = 0, 32, 8
    cfg = dict(dims=2, nx=nx, ny=ny, k=k, tau=0.8, bc=glbm.BC_PERIODIC, g=0.02)
    ux = np.full((ny, nx), 0.95 * np.sqrt(2 / 3))
    fields = (np.ones((ny, nx)), ux, np.zeros((ny, nx)))
    lat, ref = glbm.Lattice(cfg), glbm.Lattice(cfg)
    for x in (lat, ref):
        x.set_equilibrium(0, *fields)
    with pytest.raises(glbm.UnstableError):
        ref.step(12)
    with pytest.raises(glbm.UnstableError):
        lat.adjoint_flowrate(12, ckpt)
    assert 0 < ref.time < 12 and lat.time == ref.time
    assert np.array_equal(lat.get_populations(0), ref.get_populations(0))
    lat.close()
    ref.close()
