"""The scale of the int32 scatter window: a sweep of a newly set image does not depend on the
residuals that earlier sweeps saw, and a few rows far above the others (a chord that grazes a
corner) do not coarsen the others' terms.  FP32 bound of test_gpu_kernels: 1e-6 of the image a sweep."""
import numpy as np
import pytest

import oracle
import synth
from _gpu_util import ntvs_module, quantize, rel_l2
from paper_1803_01112_gb300._ffi import NTVS_SCHED_WINDOW

pytestmark = pytest.mark.gpu


def _system(nx, nz, n_hist, unordered, kind):
    s = synth.generate(synth.spec_scaled_3d(nx=nx, ny=nx, nz=nz, n_hist=n_hist, n_angles=36, n_blocks=1, seed=4),
                       val_dtype=np.float32)
    rp, col, val, b = s.row_ptr, s.col, s.val, s.b.astype(np.float32)
    if unordered:
        perm = np.random.default_rng(1).permutation(s.M)
        n = np.diff(rp)[perm]
        rp2 = np.zeros(s.M + 1, np.int64)
        np.cumsum(n, out=rp2[1:])
        at = np.repeat(rp[:-1][perm] - rp2[:-1], n) + np.arange(rp2[-1])
        rp, col, val, b = rp2, col[at], val[at], b[perm]
    store, val64 = (val, val.astype(np.float64)) if kind == "f32" else quantize(val, kind)
    return s, rp, col, store, val64, b


CASES = [(40, 4, 40_000, False, "f32", 3),       # two rows a warp
         (16, 3, 9_000, False, "f32", 2),        # four rows a warp; CTAs with fewer rows than warps
         (160, 2, 20_000, False, "f32", 1),      # a row a warp
         (160, 2, 20_000, False, "bf16", 2),     # DELTA16 words
         (40, 4, 20_000, False, "fp16", 2),      # DELTA16, two rows a warp
         (96, 7, 115_011, True, "f32", 1)]       # detected order, grouped through the index


@pytest.mark.parametrize("scale", [1e8, 300.0])
@pytest.mark.parametrize("nx,nz,n_hist,unordered,kind,blocks", CASES)
def test_sweep_does_not_depend_on_earlier_residuals(nx, nz, n_hist, unordered, kind, blocks, scale):
    ntvs = ntvs_module()
    s, rp, col, val, val64, b = _system(nx, nz, n_hist, unordered, kind)
    bp = synth.block_partition(s.M, blocks)
    x0 = s.xstar * 0.9 + 0.05
    want, _ = oracle.drop_sweep(rp, col, val64, b.astype(np.float64), bp, x0, 1.1)
    r = ntvs.Reconstructor(0)
    try:
        r.load((nx, nx, nz), rp, col, val, b, block_ptr=bp, storage=0 if kind == "f32" else 1)
        assert r.stats()["drop_schedule"] == NTVS_SCHED_WINDOW
        r.set_params(lam=1.1, N=0, alpha=0.5)
        r.set_image(x0 * scale)
        r.drop_sweep()
        r.set_image(x0)
        r.drop_sweep()
        assert rel_l2(r.get_image(), want) <= 1e-6
    finally:
        r.close()


def _graze(nx, nz, rp, col, val, b, chord):
    """Three rows of one short chord each (the first row among them), and their voxels."""
    M = rp.size - 1
    rows = np.array([0, M // 3, M - 1])
    keep = np.ones(rp[-1], bool)
    n = np.diff(rp)
    for i in rows:
        keep[rp[i] + 1:rp[i + 1]] = False
        val[rp[i]] = chord
        n[i] = 1
    rp2 = np.zeros(M + 1, np.int64)
    np.cumsum(n, out=rp2[1:])
    b[rows] = 1.0
    return rp2, col[keep], val[keep], b, col[rp[rows]]


@pytest.mark.parametrize("chord", [2e-4, 0.5])
@pytest.mark.parametrize("nx,nz,n_hist,unordered", [(40, 4, 40_000, False), (160, 2, 20_000, False),
                                                    (96, 7, 115_011, True)])
def test_grazing_rows_do_not_coarsen_the_others(nx, nz, n_hist, unordered, chord):
    ntvs = ntvs_module()
    s, rp, col, val, _, b = _system(nx, nz, n_hist, unordered, "f32")
    rp, col, val, b, hit = _graze(nx, nz, rp, col, val, b, chord)
    bp = np.array([0, s.M], np.int64)
    x0 = s.xstar * 0.9 + 0.05
    want, _ = oracle.drop_sweep(rp, col, val.astype(np.float64), b.astype(np.float64), bp, x0, 1.1)
    other = np.ones(x0.size, bool)
    other[hit] = False
    r = ntvs.Reconstructor(0)
    try:
        r.load((nx, nx, nz), rp, col, val, b, block_ptr=bp)
        assert r.stats()["drop_schedule"] == NTVS_SCHED_WINDOW
        r.set_params(lam=1.1, N=0, alpha=0.5)
        for _ in range(2):   # the scale of the first sweep and of the following ones
            r.set_image(x0)
            r.drop_sweep()
            got = r.get_image()
            assert rel_l2(got[other], want[other]) <= 1e-6
            assert rel_l2(got[hit], want[hit]) <= 1e-6
    finally:
        r.close()


@pytest.mark.parametrize("window", [-1, 16384])
def test_batch_scale_follows_its_rows(window):
    """Members whose first sweep lands every voxel (rows of one entry, lambda = 1) from an image
    1e8 times too large, and a member with grazing rows."""
    ntvs = ntvs_module()
    rng = np.random.default_rng(2)
    shape = (24, 20, 3)
    V = int(np.prod(shape))
    col = np.sort(np.tile(np.arange(V, dtype=np.int32), 8))
    M = col.size
    val = rng.uniform(0.5, 2.0, M).astype(np.float32)
    xt = rng.uniform(0.5, 1.5, V)
    b = (val.astype(np.float64) * xt[col]).astype(np.float32)
    rp = np.arange(M + 1, dtype=np.int64)
    s, rp2, col2, val2, _, b2 = _system(40, 4, 40_000, False, "f32")
    rp2, col2, val2, b2, hit = _graze(40, 4, rp2, col2, val2, b2, 2e-3)
    x2 = s.xstar * 0.9 + 0.05
    bt = ntvs.Batch(0)
    try:
        bt.add(shape, rp, col, val, b, 1, ntvs.Params(lam=1.0, N=0, alpha=0.5), xt * 1e8)
        bt.add((40, 40, 4), rp2, col2, val2, b2, 1, ntvs.Params(lam=1.1, N=0, alpha=0.5), x2)
        if window >= 0:
            bt.set_schedule(256, window)
        bt.finalize(max_cycles=8)
        bt.run(1)
        one = bt.get_image(1)
        bt.run(1)
        zero = bt.get_image(0)
    finally:
        bt.close()
    want, _ = oracle.drop_sweep(rp2, col2, val2.astype(np.float64), b2.astype(np.float64),
                                np.array([0, s.M], np.int64), x2, 1.1)
    other = np.ones(want.size, bool)
    other[hit] = False
    assert rel_l2(one[other], want[other]) <= 1e-6
    x = xt * 1e8
    for _ in range(2):
        x, _ = oracle.drop_sweep(rp, col, val.astype(np.float64), b.astype(np.float64), np.array([0, M], np.int64), x, 1.0)
    assert rel_l2(zero, x) <= 1e-6


@pytest.mark.parametrize("factor", [1e2, 1e6])
@pytest.mark.parametrize("nx,nz,n_hist,unordered", [(40, 4, 40_000, False), (96, 7, 115_011, True)])
def test_a_corrupt_measurement_does_not_coarsen_the_others(nx, nz, n_hist, unordered, factor):
    """One right-hand side far off moves the voxels of its row; the others keep their precision, in the
    sweep itself and in the next block's (whose scale follows the first one's residuals)."""
    ntvs = ntvs_module()
    s, rp, col, val, _, b = _system(nx, nz, n_hist, unordered, "f32")
    bad = s.M // 5
    b[bad] *= factor
    bp = np.array([0, s.M // 2, s.M] if not unordered else [0, s.M], np.int64)
    x0 = s.xstar * 0.9 + 0.05
    want, _ = oracle.drop_sweep(rp, col, val.astype(np.float64), b.astype(np.float64), bp, x0, 1.1)
    # what the bad row moved, directly or through rows that share its voxels, is not compared
    b2 = b.copy()
    b2[bad] /= factor
    clean, _ = oracle.drop_sweep(rp, col, val.astype(np.float64), b2.astype(np.float64), bp, x0, 1.1)
    other = np.abs(want - clean) <= 1e-3
    assert other.mean() > 0.05
    r = ntvs.Reconstructor(0)
    try:
        r.load((nx, nx, nz), rp, col, val, b, block_ptr=bp)
        assert r.stats()["drop_schedule"] == NTVS_SCHED_WINDOW
        r.set_params(lam=1.1, N=0, alpha=0.5)
        for _ in range(2):
            r.set_image(x0)
            r.drop_sweep()
            assert rel_l2(r.get_image()[other], want[other]) <= 1e-6
    finally:
        r.close()
