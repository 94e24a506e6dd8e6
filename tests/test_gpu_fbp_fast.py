"""The back-projection's tile kernel and the binning's FP32 prefilter against the FP64 oracle,
at the sizes where they can go wrong: voxel tiles with remainders, more angles than one table
holds, bins wide and fine enough for either row width and for the per-row kernel, and
histories whose bins lie at edges, at degenerate chords or outside.

Bounds: bins are decided exactly (counts equal); the back-projection is held to 1e-12 of the
largest value, as for the per-row kernel (each weight moves by about 1e-14 at most).
"""
import math

import numpy as np
import pytest

import oracle
from test_gpu_fbp import _dev, _geoms, _gpu_bin, ntvs, torch  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,n_theta,n_t,dt", [
    (32, 32, 1, 8, 40, 1.0),       # one full tile, one run of angles
    (33, 31, 2, 9, 64, 1.0),       # remainders in both directions and in the angles
    (1, 1, 1, 1, 1, 1.0),
    (65, 7, 3, 257, 50, 0.95),     # a second table of angles
    (40, 34, 1, 11, 300, 0.2),     # about 219 bins a tile: the wide rows
    (40, 34, 1, 11, 900, 0.1),     # finer than the wide rows: the per-row kernel
    (20, 12, 1, 5, 4000, 1.0),     # positions beyond the fixed-point range: the per-row kernel
    (200, 200, 2, 180, 160, 15 / 16),
])
def test_backproject_tiles(ntvs, torch, nx, ny, nz, n_theta, n_t, dt):  # noqa: F811
    go, gd = _geoms(ntvs, nx=nx, ny=ny, nz=nz, dx=1.0, dy=1.0, dz=2.0, n_theta=n_theta, n_t=n_t, dt=dt, theta0=-0.1)
    q = np.random.default_rng(n_theta + nx).standard_normal((nz, n_theta, n_t))
    fo = oracle.fbp_backproject(q, go)
    img = torch.empty(nx * ny * nz, dtype=torch.float64, device="cuda")
    ntvs.ntvs_fbp_backproject(gd, _dev(torch, q.reshape(-1), torch.float64), img)
    torch.cuda.synchronize()
    assert np.abs(img.cpu().numpy() - fo).max() <= 1e-12 * np.abs(fo).max()


@pytest.mark.parametrize("n_theta,n_t,dt,theta0", [(180, 160, 0.9375, -math.pi / 360), (4096, 8192, 0.01, 0.0),
                                                   (7, 3, 40.0, 2.5)])
def test_bin_prefilter_decides_as_fp64(ntvs, torch, n_theta, n_t, dt, theta0):  # noqa: F811
    rng = np.random.default_rng(n_t)
    M = 20_003
    go, gd = _geoms(ntvs, nx=8, ny=8, nz=5, dx=1.0, dy=1.0, dz=1.25, n_theta=n_theta, n_t=n_t, dt=dt, theta0=theta0)
    th = rng.uniform(0, 2 * math.pi, M)
    th[::3] = theta0 + math.pi / n_theta * rng.integers(0, n_theta, th[::3].size)   # on angle-bin edges
    t = rng.uniform(-0.6, 0.6, M) * n_t * dt
    t[1::3] = (np.floor(t[1::3] / dt) + (0.5 if n_t % 2 else 0.0)) * dt             # on lateral edges
    z = rng.uniform(-0.5, 5 * 1.25 + 0.5, M)
    z[2::3] = 1.25 * rng.integers(-1, 7, z[2::3].size)                              # on slice edges
    L = 10.0 ** rng.uniform(-3, 3, M)
    ux, uy = np.cos(th), np.sin(th)
    P = np.zeros((M, 10), np.float32)
    P[:, 0], P[:, 1] = -t * uy - L * ux, t * ux - L * uy
    P[:, 3], P[:, 4] = -t * uy + L * ux, t * ux + L * uy
    P[:, 2] = P[:, 5] = z
    P[5, 3:5] = P[5, 0:2]                 # no chord
    P[6, :6] = [0, 0, 1, 1e-30, 1e-30, 1]  # FP32 would underflow
    P[7, :6] = [1e25, 0, 1, -1e25, 1, 1]
    w = rng.uniform(0.5, 2.0, M)
    so, co = oracle.fbp_bin(P, w, go)
    sg, cg = _gpu_bin(ntvs, torch, gd, P, w)
    assert np.array_equal(cg, co)
    assert np.allclose(sg, so, rtol=1e-13, atol=0.0)
