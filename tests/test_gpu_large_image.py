"""The kernels over all voxels take four voxels a thread on large images (from 152 SMs x 6144
voxels on): an odd voxel count just above that, and the last voxels, against NumPy in FP64.

Rows of one voxel each with lambda = 1 project it exactly, so every voxel is known: those of the
rows become b_j / a_j, the others keep their value bit for bit."""
import numpy as np
import pytest

import oracle
from _gpu_util import ntvs_module, rel_l2

pytestmark = pytest.mark.gpu

SHAPE = (331, 283, 11)          # 1,030,403 voxels


def _system(dtype):
    V = int(np.prod(SHAPE))
    rng = np.random.default_rng(5)
    hit = np.unique(np.r_[0, rng.integers(0, V, 4000), V - 257, V - 2, V - 1]).astype(np.int32)
    val = rng.uniform(0.5, 2.0, hit.size).astype(dtype)
    b = rng.uniform(0.5, 1.5, hit.size).astype(dtype)
    return V, hit, val, b


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_large_image_copies_step_and_apply(dtype):
    ntvs = ntvs_module()
    V, hit, val, b = _system(dtype)
    x0 = np.random.default_rng(6).uniform(0.5, 1.5, V)
    eps = 1e-15 if dtype == np.float64 else 3e-7       # a few roundings of the type
    r = ntvs.Reconstructor(0)
    try:
        r.load(SHAPE, np.arange(hit.size + 1, dtype=np.int64), hit, val, b, n_blocks=2)
        r.set_params(lam=1.0, N=1, alpha=0.5, eps_tv=1e-6)
        r.set_image(x0)                                # the FP32 copies of every voxel
        assert rel_l2(r.forward_project(x0), val * x0[hit]) <= eps
        g, gn = r.tv_gradient(np.float64)
        want = oracle.tv_grad(x0, SHAPE, 1e-6)
        np.testing.assert_allclose(g, want, rtol=0, atol=(1e-11 if dtype == np.float64 else 2e-5) * np.abs(want).max())
        r.perturb(0.25)                                # the step, from the gradient as the library forms it
        step = x0 - 0.25 / gn * g
        x1 = r.get_image()
        np.testing.assert_allclose(x1, step, rtol=1e-15, atol=1e-15)
        r.drop_sweep()                                 # the apply, and the copies it leaves
        x2 = r.get_image()
        keep = np.ones(V, bool)
        keep[hit] = False
        assert np.array_equal(x2[keep], x1[keep])
        assert rel_l2(x2[hit], b.astype(np.float64) / val) <= eps
        r.drop_sweep()
        np.testing.assert_allclose(r.block_resid(), 0.0, atol=hit.size * (4 * eps) ** 2)
        g2, _ = r.tv_gradient(np.float64)              # reads the split copies
        want = oracle.tv_grad(r.get_image(), SHAPE, 1e-6)
        np.testing.assert_allclose(g2, want, rtol=0, atol=(1e-11 if dtype == np.float64 else 2e-5) * np.abs(want).max())
    finally:
        r.close()


@pytest.mark.parametrize("xt,ot", [("float64", "float64"), ("float64", "float32"), ("float32", "float64")])
def test_fp64_projection_onto_its_own_input(xt, ot):
    """Device input and output that share memory: the image is read before it is overwritten."""
    import torch
    ntvs = ntvs_module()
    rng = np.random.default_rng(7)
    shape, M = (20, 10, 4), 700
    V = int(np.prod(shape))
    n = rng.integers(0, 40, M)
    rp = np.zeros(M + 1, np.int64)
    np.cumsum(n, out=rp[1:])
    col = np.concatenate([np.sort(rng.choice(V, q, replace=False)) for q in n]).astype(np.int32)
    val = rng.uniform(0.1, 1.5, col.size)
    x = rng.uniform(0.0, 1.0, V).astype(xt)
    row = np.repeat(np.arange(M), n)
    want = np.bincount(row, val * x[col], minlength=M)
    r = ntvs.Reconstructor(0)
    try:
        r.load(shape, rp, col, val, np.zeros(M))
        buf = torch.zeros(8 * max(V, M), dtype=torch.uint8, device="cuda")
        xd = buf.view(getattr(torch, xt))[:V]
        xd.copy_(torch.from_numpy(x))
        out = buf.view(getattr(torch, ot))[:M]
        torch.cuda.synchronize()
        r.forward_project(xd, out)
        assert rel_l2(out.cpu().numpy(), want) <= (1e-14 if ot == "float64" else 1e-7)
    finally:
        r.close()
