"""Histories stored as detected (rows of all slices mixed): large blocks of FP32 rows are grouped by
home slice for the windowed schedule through an index of the rows.  Sweeps, partial blocks and
the projection keep the stored order's meaning and are compared with the FP64 oracle and with
the plain schedule (FP32 bounds of test_gpu_kernels: 1e-6 of the image a sweep)."""
import numpy as np
import pytest

import oracle
import synth
from _gpu_util import ntvs_module, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz,n_hist,blocks,empty", [(96, 7, 330_011, [0.0, 0.45, 0.45, 1.0], 5000),
                                                       (96, 7, 230_011, [0.0, 0.45, 0.45, 1.0], 0)])
def test_unordered_rows_take_the_window(nx, nz, n_hist, blocks, empty):
    ntvs = ntvs_module()
    from paper_1803_01112_gb300._ffi import NTVS_SCHED_PLAIN, NTVS_SCHED_WINDOW
    s = synth.generate(synth.spec_scaled_3d(nx=nx, ny=nx, nz=nz, n_hist=n_hist, n_angles=36, n_blocks=1, seed=4),
                       val_dtype=np.float32)
    perm = np.random.default_rng(1).permutation(s.M)
    n = np.diff(s.row_ptr)[perm]
    n[:empty] = 0                                           # rows without entries among them
    rp = np.zeros(s.M + 1, np.int64)
    np.cumsum(n, out=rp[1:])
    at = np.repeat(s.row_ptr[:-1][perm] - rp[:-1], n) + np.arange(rp[-1])
    col, val, b = s.col[at], s.val[at], s.b[perm].astype(np.float32)
    bp = (np.array(blocks) * s.M).astype(np.int64)          # an empty block in the middle
    x0 = s.xstar * 0.9 + 0.05
    want, ss = oracle.drop_sweep(rp, col, val.astype(np.float64), b.astype(np.float64), bp, x0, 1.1)
    out = {}
    for sched in (0, NTVS_SCHED_PLAIN):
        r = ntvs.Reconstructor(0)
        try:
            r.load((nx, nx, nz), rp, col, val, b, block_ptr=bp, schedule=sched)
            big = rp[-1] // (bp.size - 1) >= 12_000_000
            assert r.stats()["drop_schedule"] == (NTVS_SCHED_WINDOW if sched == 0 and big else NTVS_SCHED_PLAIN)
            r.set_params(lam=1.1, N=0, alpha=0.5)
            r.set_image(x0)
            r.drop_sweep()
            assert rel_l2(r.get_image(), want) <= 1e-6
            np.testing.assert_allclose(r.block_resid(), ss, rtol=1e-4)
            r.set_image(x0)
            t = bp.size - 2
            whole, _ = r.drop_block_partial(t)
            mid = int(bp[t] + bp[t + 1]) // 2
            halves = r.drop_block_partial(t, r0=int(bp[t]), r1=mid)[0] + r.drop_block_partial(t, r0=mid,
                                                                                             r1=int(bp[t + 1]))[0]
            inv = 1.0 / np.maximum(r.hit_counts(t), 1)      # the window's bar is that of the image
            assert rel_l2(x0 + whole * inv, x0 + halves * inv) <= 1e-6
            out[sched] = r.forward_project(x0)
        finally:
            r.close()
    assert np.array_equal(out[0], out[NTVS_SCHED_PLAIN])
