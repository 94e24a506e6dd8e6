"""Reading a batch member's image into device memory waits for the caller's pending work on the
default stream, whatever the type, and gives the values that host memory gets."""
import numpy as np
import pytest

import synth
from _gpu_util import ntvs_module

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_batch_image_into_a_tensor_with_pending_work(dtype):
    import torch
    ntvs = ntvs_module()
    s = synth.generate(synth.spec_scaled_3d(nx=40, ny=37, nz=3, n_hist=6_000, n_angles=24, n_blocks=2, seed=5))
    bt = ntvs.Batch(0)
    try:
        bt.add((40, 37, 3), s.row_ptr, s.col, s.val.astype(np.float32), s.b.astype(np.float32), 2,
               ntvs.Params(lam=0.5, N=1, alpha=0.75), s.xbar)
        bt.set_schedule(256, 8192)
        bt.finalize(max_cycles=4)
        bt.run(2)
        want = bt.get_image(0, dtype)
        whole = torch.empty(s.xbar.size + 1, dtype=getattr(torch, np.dtype(dtype).name), device="cuda")
        torch.cuda.synchronize()
        for out in (whole[:-1], whole[1:]):        # aligned, and by one element only
            torch.cuda._sleep(100_000_000)         # about 50 ms on the default stream, then a fill
            out.fill_(7.0)
            ntvs.ntvs_batch_get_image(bt._bt, 0, out)
            assert np.array_equal(out.cpu().numpy(), want)
    finally:
        bt.close()
