"""The FP32 initial equilibrium stores the FP64 formula's deviations rounded once, also
where its terms cancel and where velocities are so small that the low words of the
float pairs underflow. Reference: the formula in numpy's FP64. Every stored float must
be its rounding unless the FP64 value lies within 2^-48 of its terms' magnitudes of a
rounding boundary (the FP64 roundings of N <= 4 levels stay below 2^-49 of them)."""
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


def _axis(C, u):
    """E - W of every velocity and the sum of its terms' magnitudes."""
    Q = C.shape[0]
    N, v = Q // 2, u * u
    d, mag = np.empty((Q,) + u.shape), np.empty((Q,) + u.shape)
    for n in range(N + 1):
        e, me, o, mo = (np.zeros_like(u) for _ in range(4))
        for i in range(N, 0, -1):
            e, me = (e + C[N + n, 2 * i]) * v, (me + abs(C[N + n, 2 * i])) * v
        for i in range(N - 1, -1, -1):
            c = C[N + n, 2 * i + 1] if n else 0.0
            o, mo = o * v + c, mo * v + abs(c)
        for q, s in ((N + n, 1), (N - n, -1)):
            d[q] = e + s * u * o
            mag[q] = me + abs(u) * mo
    return d, mag


def _check(cfg, rho, us):
    lat = glbm.Lattice(dict(cfg, prec=glbm.FP32_DEV, tau=0.9))
    lat.set_equilibrium(0, rho, *us)
    Q = 2 * cfg["k"] + 3
    stored = np.empty((lat.nq(), int(np.prod(rho.shape[:-1])), cfg["nx"]), np.float32)
    lat.pack_columns(0, 0, cfg["nx"], stored)
    lat.close()
    stored = stored.reshape((-1,) + rho.shape)
    C = glbm.eq_table(cfg["k"])
    W, r1 = C[:, 0], rho - 1.0
    (dx, mx), (dy, my) = _axis(C, us[0]), _axis(C, us[1])
    dz, mz = _axis(C, us[2]) if len(us) == 3 else (np.zeros((1,) + rho.shape),) * 2
    bad = 0
    for iz in range(dz.shape[0]):
        wz = W[iz] if len(us) == 3 else 1.0
        for iy in range(Q):
            wyz = W[iy] * wz
            rest = dy[iy] * (wz + dz[iz]) + W[iy] * dz[iz]  # E^y E^z - W^y W^z
            A, B = rho * (wyz + rest), r1 * wyz + rho * rest
            mA = rho * (W[iy] + my[iy]) * (wz + mz[iz])
            mB = abs(r1) * wyz + rho * (my[iy] * (wz + mz[iz]) + W[iy] * mz[iz])
            for ix in range(Q):
                v = W[ix] * B + dx[ix] * A
                mag = W[ix] * mB + mx[ix] * mA
                s = stored[(iz * Q + iy) * Q + ix]
                f = v.astype(np.float32)
                near = np.minimum(*[abs((f.astype(np.float64) + np.nextafter(f, np.float32(x))) / 2 - v)
                                    for x in (-np.inf, np.inf)])
                bad += int(((s != f) & (near > 2.0 ** -48 * mag)).sum())
    assert bad == 0, bad


@pytest.mark.parametrize("k,nx,ny", [(0, 700, 400), (1, 500, 400), (3, 333, 300)])
def test_cancelling_rows_2d(k, nx, ny):
    """Densities that make B = rho E^y - W^y vanish nearly, at one row of every node."""
    rng = np.random.default_rng(20 + k)
    us = [0.05 * rng.standard_normal((ny, nx)) for _ in range(2)]
    C = glbm.eq_table(k)
    d = _axis(C, us[1])[0]
    row = rng.integers(0, d.shape[0], (1, ny, nx))
    d = np.take_along_axis(d, row, 0)[0]
    eps = 10.0 ** rng.uniform(-12, -3, (ny, nx)) * rng.choice([-1, 1], (ny, nx))
    _check(dict(dims=2, k=k, nx=nx, ny=ny), 1 - d / (C[row[0], 0] + d) * (1 + eps), us)


def test_cancelling_rows_3d():
    k, shape = 1, (20, 30, 101)
    rng = np.random.default_rng(31)
    us = [0.05 * rng.standard_normal(shape) for _ in range(3)]
    C = glbm.eq_table(k)
    e = []
    w = 1.0
    for u in us[1:]:
        row = rng.integers(0, 5, (1,) + shape)
        e.append(C[row[0], 0] + np.take_along_axis(_axis(C, u)[0], row, 0)[0])
        w = w * C[row[0], 0]
    eps = 10.0 ** rng.uniform(-12, -3, shape) * rng.choice([-1, 1], shape)
    rho = 1 + (w / (e[0] * e[1]) - 1) * (1 + eps)
    _check(dict(dims=3, k=k, nx=101, ny=30, nz=20), rho, us)


@pytest.mark.parametrize("k", [0, 1, 3])
def test_tiny_velocities(k):
    """Velocities from 1e-19 to 1e-11 beside a density of 1 and near 1: the populations
    at rest along x are of order u^2."""
    rng = np.random.default_rng(40 + k)
    shape = (60, 300)
    u = 10.0 ** rng.uniform(-19, -11, shape) * rng.choice([-1, 1], shape)
    zero = np.zeros(shape)
    cfg = dict(dims=2, k=k, nx=shape[1], ny=shape[0])
    _check(cfg, np.ones(shape), [u, zero])
    _check(cfg, np.ones(shape), [u, 0.03 * rng.standard_normal(shape)])
    _check(cfg, 1 + 1e-15 * rng.integers(-3, 4, shape), [u, u[::-1].copy()])
