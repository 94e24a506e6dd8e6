"""The tiled TV gradient (31 x 15 voxel tiles marched along z) and the block apply at tile edges,
against the FP64 oracle, with the bounds of test_gpu_kernels: summation order only in FP64
(1e-11 of the gradient's scale), about ten FP32 operations a voxel in FP32 (2e-5)."""
import numpy as np
import pytest

import oracle
from _gpu_util import empty_system, ntvs_module, rel_l2
from test_gpu_kernels import _empty32

pytestmark = pytest.mark.gpu

SHAPES = [(31, 15, 1), (32, 16, 2), (30, 14, 3), (62, 30, 33), (63, 31, 5), (1, 1, 40), (2, 200, 7), (311, 3, 9)]


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("shape", SHAPES)
def test_gradient_and_checked_phi_at_tile_edges(dtype, shape):
    ntvs = ntvs_module()
    rng = np.random.default_rng(shape[0])
    x = rng.uniform(-1.0, 2.0, int(np.prod(shape)))
    x[rng.random(x.size) < 0.3] = 0.0                       # flat runs and exact zeros
    x[rng.random(x.size) < 0.05] *= 1e-12
    x = x.astype(dtype)
    x64 = x.astype(np.float64)
    r = empty_system(ntvs, shape) if dtype == np.float64 else _empty32(ntvs, shape)
    try:
        r.set_params(lam=1.0, N=1, alpha=0.5, eps_tv=1e-8)
        r.set_image(x)
        g, gn = r.tv_gradient(np.float64)
        _, phi, _ = r.perturb_checked(1e-3)
    finally:
        r.close()
    want = oracle.tv_grad(x64, shape, 1e-8)
    scale = max(np.abs(want).max(), 1.0)
    tol = 1e-11 if dtype == np.float64 else 2e-5
    np.testing.assert_allclose(g, want, rtol=0, atol=tol * scale)
    assert gn == pytest.approx(np.linalg.norm(want), rel=1e-12 if dtype == np.float64 else 1e-5, abs=1e-300)
    assert phi == pytest.approx(oracle.tv(x64, shape), rel=1e-12, abs=1e-300)


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_apply_keeps_untouched_voxels_and_their_copies(dtype):
    # rows of one voxel each: exact projections x_j = b_j / a_j with lambda = 1, every other
    # voxel bit for bit as set; a second sweep then gathers the copies the first one left
    ntvs = ntvs_module()
    shape = (37, 5, 3)
    V = int(np.prod(shape))
    rng = np.random.default_rng(9)
    hit = np.sort(rng.permutation(V)[: V // 3]).astype(np.int32)
    val = rng.uniform(0.5, 2.0, hit.size).astype(dtype)
    b = rng.uniform(-1.0, 1.0, hit.size).astype(dtype)
    x0 = rng.uniform(0.1, 2.0, V) * 10.0 ** rng.integers(-30, 30, V)
    r = ntvs.Reconstructor(0)
    try:
        r.load(shape, np.arange(hit.size + 1, dtype=np.int64), hit, val, b, n_blocks=2)
        r.set_params(lam=1.0, N=0, alpha=0.5)
        keep = np.ones(V, bool)
        keep[hit] = False
        r.set_image(x0)
        r.drop_sweep()
        x = r.get_image()
        assert np.array_equal(x[keep], x0[keep])
        # a well-scaled image on a fresh system (the FP32 window's scale follows the residuals it
        # has seen): the projection is exact
        r.load(shape, np.arange(hit.size + 1, dtype=np.int64), hit, val, b, n_blocks=2)
        r.set_params(lam=1.0, N=0, alpha=0.5)
        r.set_image(rng.uniform(0.5, 1.5, V))
        r.drop_sweep()
        want = b.astype(np.float64) / val
        assert rel_l2(r.get_image()[hit], want) <= (1e-15 if dtype == np.float64 else 2e-7)
        proj = r.forward_project(r.get_image())
        assert rel_l2(proj, b.astype(np.float64)) <= (1e-15 if dtype == np.float64 else 3e-7)
    finally:
        r.close()
