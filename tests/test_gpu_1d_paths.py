"""Which 1D calls step on the cluster and which launch after launch: long lattices, high
FP64 levels and short calls of one instance launch by launch, several instances
side by side on clusters, with the same states either way (a call of n steps against
n calls of one step)."""
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


# (k, L, instances, precision, steps of a call, launches of it)
@pytest.mark.parametrize("k,L,n,prec,steps,launches", [
    (0, 64000, 1, glbm.FP32_DEV, 16, 1),    # three quarters of Q L = 256000
    (0, 64000, 1, glbm.FP32_DEV, 7, 7),
    (0, 85400, 1, glbm.FP32_DEV, 16, 16),   # above 256000
    (0, 85400, 2, glbm.FP32_DEV, 16, 1),
    (2, 8000, 1, glbm.FP32_DEV, 1, 1),
    (2, 8000, 1, glbm.FP32_DEV, 2, 1),
    (7, 8000, 1, glbm.FP32_DEV, 3, 3),
    (7, 8000, 1, glbm.FP32_DEV, 4, 1),
    (7, 15100, 1, glbm.FP32_DEV, 12, 12),
    (7, 2900, 1, glbm.FP64, 3, 1),
    (7, 2901, 1, glbm.FP64, 3, 3),
    (7, 2901, 2, glbm.FP64, 3, 1),
    (5, 3072, 1, glbm.FP64, 2, 1),
    (5, 3073, 1, glbm.FP64, 2, 2),
])
def test_path_and_state(k, L, n, prec, steps, launches):
    cfgs = [dict(dims=1, nx=L, k=k, tau=0.7 + 0.2 * i, prec=prec) for i in range(n)]
    a, b = glbm.Lattice(cfgs), glbm.Lattice(cfgs)
    x = np.arange(L) / L
    for lat in (a, b):
        for i in range(n):
            lat.set_equilibrium(i, 1 + 0.05 * np.sin(2 * np.pi * x + i), 0.03 * np.cos(6 * np.pi * x))
    n0 = a.kernel_launches
    a.step(steps)
    assert a.kernel_launches - n0 == launches
    for _ in range(steps):
        b.step(1)
    for i in range(n):
        np.testing.assert_array_equal(a.get_populations(i), b.get_populations(i))
    a.close()
    b.close()
