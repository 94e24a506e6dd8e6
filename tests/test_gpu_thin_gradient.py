"""The FP64 gradient of images too thin for tiles (one thread per voxel there), and of shapes on either
side of that rule, against the oracle with the FP64 bounds of test_gpu_kernels."""
import numpy as np
import pytest

import oracle
from _gpu_util import empty_system, ntvs_module

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 100_000), (1, 2000, 50), (2, 3, 30_000), (33, 33, 100), (31, 15, 400),
                                   (90_001, 1, 1), (5, 300, 100)])
def test_gradient_and_phi_of_thin_images(shape):
    ntvs = ntvs_module()
    rng = np.random.default_rng(shape[0])
    x = rng.uniform(-1.0, 2.0, int(np.prod(shape)))
    x[rng.random(x.size) < 0.3] = 0.0
    r = empty_system(ntvs, shape)
    try:
        r.set_params(lam=1.0, N=1, alpha=0.5, eps_tv=1e-8)
        r.set_image(x)
        g, gn = r.tv_gradient(np.float64)
        _, phi, _ = r.perturb_checked(1e-3)
    finally:
        r.close()
    want = oracle.tv_grad(x, shape, 1e-8)
    np.testing.assert_allclose(g, want, rtol=0, atol=1e-11 * np.abs(want).max())
    assert gn == pytest.approx(np.linalg.norm(want), rel=1e-12)
    assert phi == pytest.approx(oracle.tv(x, shape), rel=1e-12)
