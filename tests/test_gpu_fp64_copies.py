"""FP64 rows on few voxels scatter into 1, 4 or 16 copies of delta by the entries a voxel of a block (from
100 and 800 on): sweeps, single blocks, partial blocks and the summed delta of a rank against the oracle,
summation order only (1e-12)."""
import numpy as np
import pytest

import oracle
import synth
from _gpu_util import ntvs_module, rel_l2
from paper_1803_01112_gb300._ffi import ALLREDUCE_FN

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("val_dtype", [np.float64, np.float32])
@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("nx,nz,n_hist,blocks", [(16, 1, 900, [0.0, 0.5, 0.5, 1.0]),      # 1 copy; an empty block
                                                 (16, 1, 6_000, [0.0, 0.3, 1.0]),        # 4
                                                 (13, 2, 40_000, [0.0, 0.4, 1.0])])      # 16
def test_copies_sum_to_the_block(nx, nz, n_hist, blocks, storage, val_dtype):
    ntvs = ntvs_module()
    s = synth.generate(synth.spec_scaled_3d(nx=nx, ny=nx, nz=nz, n_hist=n_hist, n_angles=36, n_blocks=1, seed=6))
    val = s.val.astype(val_dtype)
    v64 = val.astype(np.float64)
    b = s.b if val_dtype == np.float64 else s.b.astype(np.float32)
    b64 = b.astype(np.float64)
    bp = (np.array(blocks) * s.M).astype(np.int64)
    x0 = s.xstar * 0.9 + 0.05
    r = ntvs.Reconstructor(0)
    try:
        r.set_compute_dtype(ntvs.NTVS_F64)
        r.load((nx, nx, nz), s.row_ptr, s.col, val, b, block_ptr=bp, storage=storage)
        r.set_params(lam=0.9, N=0, alpha=0.5)
        want, ss = oracle.drop_sweep(s.row_ptr, s.col, v64, b64, bp, x0, 0.9)
        for _ in range(2):                                  # the copies are zero again after a sweep
            r.set_image(x0)
            r.drop_sweep()
            assert rel_l2(r.get_image(), want) <= 1e-12
            np.testing.assert_allclose(r.block_resid(), ss, rtol=1e-12)
        t = bp.size - 2
        r.set_image(x0)
        delta, _ = r.drop_block_partial(t)                  # one array, as a rank hands out
        r.apply_delta(t, delta)
        one = r.get_image()
        r.set_image(x0)
        r.drop_block(t)
        assert rel_l2(r.get_image(), one) <= 1e-12
        fn = ALLREDUCE_FN(lambda buf, n, dtype, stream, user: 0)
        r.set_allreduce(fn)
        r.set_image(x0)
        r.drop_block(t)
        assert rel_l2(r.get_image(), one) <= 1e-12
    finally:
        r.close()
