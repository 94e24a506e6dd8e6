"""The load's fused preparation (validation, remapping, packing, norms, hit counts and column sums
in one pass) at its edges: every storage and arithmetic, blocks without rows, stored zeros, rows
without entries, bad columns and values, and a voxel with more hits in a block than a float
counts.  Counts are exact; hit counts are compared as integers."""
import numpy as np
import pytest

from _gpu_util import ntvs_module

pytestmark = pytest.mark.gpu


def _system(rng, V, M, dtype):
    n = np.minimum(rng.integers(0, 9, M), V)
    rp = np.zeros(M + 1, np.int64)
    np.cumsum(n, out=rp[1:])
    col = np.concatenate([rng.choice(V, min(k, V), replace=False) for k in n] or [np.zeros(0)]).astype(np.int32)
    val = rng.uniform(0.5, 2.0, col.size).astype(dtype)
    val[rng.random(col.size) < 0.1] = 0
    return rp, col, val


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("dtype,compute,storage", [(np.float32, 1, 0), (np.float32, 0, 0), (np.float64, 0, 0),
                                                   (np.float16, 1, 0), (np.float16, 1, 1), (np.float32, 1, 1)])
@pytest.mark.parametrize("shape,M", [((9, 7, 3), 301), ((33, 5, 1), 64), ((1, 1, 1), 5)])
def test_hit_counts_of_every_storage(shape, M, dtype, compute, storage, device):
    import torch
    ntvs = ntvs_module()
    rng = np.random.default_rng(M)
    V = int(np.prod(shape))
    rp, col, val = _system(rng, V, M, dtype)
    if V == 1:
        rp, col, val = np.arange(M + 1, dtype=np.int64), np.zeros(M, np.int32), np.ones(M, dtype)
    b = rng.uniform(0, 1, M).astype(np.float64 if dtype == np.float64 else np.float32)
    bp = np.array([0, M // 3, M // 3, M], np.int64)     # an empty block in the middle
    arrs = (rp, col, val, b)
    if device:
        arrs = tuple(torch.from_numpy(a).cuda() for a in arrs)
    r = ntvs.Reconstructor(0)
    try:
        r.set_compute_dtype(compute)
        r.load(shape, *arrs, block_ptr=bp, storage=storage)
        row = np.repeat(np.arange(M), np.diff(rp))
        for t in range(3):
            keep = (row >= bp[t]) & (row < bp[t + 1]) & (val != 0)
            assert np.array_equal(r.hit_counts(t), np.bincount(col[keep], minlength=V))
        if device:
            assert torch.equal(arrs[1].cpu(), torch.from_numpy(col))     # the caller's columns are untouched
        bad = col.copy()
        if col.size:
            bad[-1] = V
            with pytest.raises(ntvs.NtvsError, match="column"):
                r.load(shape, rp, bad, val, b, block_ptr=bp, storage=storage)
            nan = val.copy()
            nan[0] = np.inf
            with pytest.raises(ntvs.NtvsError, match="non-finite matrix value"):
                r.load(shape, rp, col, nan, b, block_ptr=bp, storage=storage)
    finally:
        r.close()


@pytest.mark.parametrize("half", [False, True])
def test_a_voxel_hit_more_than_2_24_times(half):
    import torch
    ntvs = ntvs_module()
    M = (1 << 24) + 5
    rp = torch.arange(M + 1, dtype=torch.int64, device="cuda")
    col = torch.zeros(M, dtype=torch.int32, device="cuda")
    col[:3] = 1
    val = torch.ones(M, dtype=torch.float16 if half else torch.float32, device="cuda")
    b = torch.ones(M, dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    r = ntvs.Reconstructor(0)
    try:
        r.load((2, 1, 1), rp, col, val, b, n_blocks=1)
        r.set_params(lam=1.0, N=0, alpha=0.5)
        r.set_image(np.zeros(2))
        r.drop_sweep()
        # every row projects its voxel onto 1: delta_j / s_j = 1 needs the full count
        x = r.get_image()
        assert abs(x[1] - 1.0) <= 1e-6
        want = float(np.float32(1.0 / (M - 3)))
        got = r.hit_counts(0)
        assert got[1] == 3 and abs(1.0 / got[0] - want) <= 1e-7 * want
    finally:
        r.close()
