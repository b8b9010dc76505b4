"""The adjoint of FP64 states at any density: without a force the scheme is linear in the
populations, so at a density scaled by a power of two the flow rate and its
derivatives by tau and the wall speeds are scaled by it bit for bit."""
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


@pytest.mark.parametrize("bc", [glbm.BC_WALLS, glbm.BC_PERIODIC])
@pytest.mark.parametrize("k,nx,ny", [(0, 20, 9), (2, 33, 12), (4, 40, 30), (7, 12, 10)])
def test_scaled_density(k, nx, ny, bc):
    cfg = dict(dims=2, nx=nx, ny=ny, k=k, tau=0.9, bc=bc)
    if bc == glbm.BC_WALLS:
        cfg.update(u_wall_lo=-0.03, u_wall_hi=0.05)
    rho, ux, uy = inputs.random_macro(50 + k, nx, ny)
    out = []
    for scale in (1.0, 2.0 ** -20, 2.0 ** 12):
        lat = glbm.Lattice(cfg)
        lat.set_equilibrium(0, scale * rho, ux, uy)
        J, dtau, _, dlo, dhi = lat.adjoint_flowrate(7, 3, walls=True)
        out.append(np.array([J[0], dtau[0], dlo[0], dhi[0]]) / scale)
        lat.close()
    assert out[0][1] != 0.0
    np.testing.assert_array_equal(out[0], out[1])
    np.testing.assert_array_equal(out[0], out[2])
