"""The FP64 gradient to its last digits, in tiles and by voxel, against NumPy in extended precision.

A difference is exact to half an ulp, D = sqrt(eps + |d|^2) takes five more roundings under the root (they
halve) and one for the root, a quotient one: each of the four terms of a voxel is within 4 x 2^-53 of
itself, and their sum adds three roundings: |error| <= 7 x 2^-53 (|d1| + |d2| + |d3|) / D + ... <= 7 x 2^-53 x
(sqrt(3) + 3)."""
import numpy as np
import pytest

from _gpu_util import empty_system, ntvs_module

pytestmark = pytest.mark.gpu


def _gradient(x, eps):
    x = x.astype(np.longdouble)
    d = [np.zeros_like(x) for _ in range(3)]
    d[0][:, :, :-1] = x[:, :, 1:] - x[:, :, :-1]
    d[1][:, :-1] = x[:, 1:] - x[:, :-1]
    d[2][:-1] = x[1:] - x[:-1]
    D = np.sqrt(np.longdouble(eps) + d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
    g = -(d[0] + d[1] + d[2]) / D
    g[:, :, 1:] += (d[0] / D)[:, :, :-1]
    g[:, 1:] += (d[1] / D)[:, :-1]
    g[1:] += (d[2] / D)[:-1]
    return g


@pytest.mark.parametrize("shape", [(64, 50, 9), (32, 32, 1), (2, 3, 30_000)])
def test_fp64_gradient_to_the_last_digits(shape):
    ntvs = ntvs_module()
    nx, ny, nz = shape
    rng = np.random.default_rng(nx)
    x = rng.uniform(0.0, 1.0, (nz, ny, nx)) * 10.0 ** rng.integers(-6, 7, (nz, ny, nx))
    r = empty_system(ntvs, shape)
    try:
        r.set_params(lam=1.0, N=1, alpha=0.5, eps_tv=1e-8)
        r.set_image(x.reshape(-1))
        g, _ = r.tv_gradient(np.float64)
    finally:
        r.close()
    err = np.abs(g.reshape(x.shape) - _gradient(x, 1e-8)).max()
    assert err <= 7 * 2.0 ** -53 * (3.0 + np.sqrt(3.0))
