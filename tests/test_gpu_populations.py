"""Import and export of populations in FP32 deviations (conversions by integer
instructions, several rows per thread): the stored float is f - W rounded to nearest,
ties to even, zeros, subnormals, infinities and NaN included, and the exported value
is that float plus W in FP64, bit for bit; ragged columns and rows, 1D to 3D."""
import numpy as np
import pytest

from paper_1905_04597_gb300 import glbm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("cfg", [dict(dims=1, nx=131, k=2), dict(dims=2, nx=129, ny=17, k=1),
                                 dict(dims=2, nx=3, ny=8, k=1), dict(dims=3, nx=5, ny=7, nz=3, k=0)])
def test_every_bit(cfg):
    lat = glbm.Lattice(dict(cfg, tau=0.9, prec=glbm.FP32_DEV))
    W = lat.get_populations(0)  # the rest state: f - W = 0
    rng = np.random.default_rng(3)
    d = (rng.standard_normal(W.shape) * 2.0 ** rng.integers(-160, 130, W.shape)).ravel()
    d[:8] = [0.0, -0.0, np.inf, -np.inf, np.nan, 3.4028235677973366e38, 2.0 ** -149, 2.0 ** -151]
    k = d.size // 2  # ties: floats plus half an ulp
    half = rng.standard_normal(k - 8).astype(np.float32).astype(np.float64)
    d[8:k] = half * (1 + 2.0 ** -24)
    f = d.reshape(W.shape) + W
    lat.set_populations(0, f)
    rows = int(np.prod(lat.shape()[:-1], dtype=int))
    stored = np.empty((lat.nq(), rows, cfg["nx"]), np.float32)
    lat.pack_columns(0, 0, cfg["nx"], stored)
    with np.errstate(over="ignore", invalid="ignore"):
        want = (f - W).astype(np.float32)
    np.testing.assert_array_equal(stored.reshape(W.shape), want)
    back = lat.get_populations(0)
    w64 = want.astype(np.float64)
    w64[np.abs(w64) < 2.0 ** -126] = 0.0  # subnormal deviations vanish beside W
    np.testing.assert_array_equal(back, w64 + W)
    lat.close()


@pytest.mark.parametrize("cfg", [dict(dims=1, nx=131, k=2), dict(dims=2, nx=129, ny=17, k=1)])
def test_fp64_is_a_copy(cfg):
    lat = glbm.Lattice(dict(cfg, tau=0.9, prec=glbm.FP64))
    f = np.random.default_rng(4).standard_normal(lat.get_populations(0).shape)
    lat.set_populations(0, f)
    np.testing.assert_array_equal(lat.get_populations(0), f)
    lat.close()
