"""The checked FP32 step forms its gradient from FP64 differences of the master image: neighbours
that differ by less than the split copies resolve (2^-49 of a voxel near 1 + 2^-25) still have
the direction of their difference."""
import numpy as np
import pytest

import oracle
from _gpu_util import ntvs_module
from test_gpu_kernels import _empty32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(9, 7, 3), (31, 5, 1), (70, 65, 20)])
def test_checked_step_sees_the_last_bits(shape):
    ntvs = ntvs_module()
    nx, ny, nz = shape
    x = np.full((nz, ny, nx), 1.0 + 2.0 ** -25 - 2.0 ** -31)
    x[nz // 2, ny // 2, nx // 2] += 3 * 2.0 ** -52       # one voxel three units in the last place above
    x = x.reshape(-1)
    g = oracle.tv_grad(x, shape, 0.0)
    gn = np.linalg.norm(g)
    assert gn > 1.0
    beta = 2 * 2.0 ** -52
    r = _empty32(ntvs, shape)
    try:
        r.set_params(lam=1.0, N=1, alpha=0.5, eps_tv=0.0, tv_check=True)
        r.set_image(x)
        acc, phi, ref = r.perturb_checked(beta)
        got = r.get_image()
    finally:
        r.close()
    want = x - beta / gn * g
    # the step moves voxels by at most 2 units in the last place: equal up to one of them
    assert np.abs(got - want).max() <= 2.0 ** -52
    assert acc == int(oracle.tv(want, shape) <= oracle.tv(x, shape))
    assert not np.array_equal(got, x)
