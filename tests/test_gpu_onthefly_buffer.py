"""The traced DROP rows at the edges of the per-warp piece buffer: rows that fill it, overflow
it at once or after some runs of 16 segments, a single segment, segment counts that are not a
multiple of 16, and voxel tiles from 1 to 16, against an FP64 evaluation of the generator's
stored rows.

The scatter numerators delta_j = lambda sum_i a_ij r_i are compared (not divided by hit counts,
which a piece near min_len may change).  FP32 tracing places a crossing within about 4 ulp of
its coordinate (250 mm: 6e-5 mm) on pieces of about 0.7 mm: 1e-4 of the norm, and 2e-4 of the
residuals' sum of squares.
"""
import numpy as np
import pytest

import synth
from _gpu_util import ntvs_module, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,n_seg,tile,n_hist", [
    (500, 500, 2, 16, 4, 1501),    # near-diagonal rows overflow in the first run of segments
    (500, 480, 1, 64, 4, 600),     # the first runs fit, later ones do not
    (430, 400, 2, 40, 2, 600),     # three runs, the last one partly empty
    (41, 37, 5, 1, 1, 2003),       # one segment a row, odd row count, canonical order
    (64, 50, 3, 17, 16, 2000),
    (3, 2, 1, 16, 4, 7),           # fewer voxels than lanes
])
def test_traced_delta_at_buffer_edges(nx, ny, nz, n_seg, tile, n_hist):
    ntvs = ntvs_module()
    spec = synth.spec_scaled_3d(nx=nx, ny=ny, nz=nz, n_hist=n_hist, n_angles=24, n_blocks=2, seed=n_seg,
                                curved=n_seg > 1).replace(n_seg=n_seg)
    s, pr = synth.generate(spec), synth.generate_paths(spec)
    b = pr.b.astype(np.float32)
    x0 = np.random.default_rng(3).uniform(0.0, 1.0, spec.V)
    row = np.repeat(np.arange(s.M), np.diff(s.row_ptr))
    dot = np.bincount(row, s.val * x0[s.col], minlength=s.M)
    n2 = np.bincount(row, s.val ** 2, minlength=s.M)
    res = np.where(n2 > 0, b - dot, b).astype(np.float64)
    fac = np.where(n2 > 0, 0.7 * res / np.maximum(n2, 1e-300), 0.0)
    bp = s.block_ptr()
    r = ntvs.Reconstructor(0).set_voxel_tile(tile, tile)
    try:
        r.load_paths((nx, ny, nz), (spec.dx, spec.dy, spec.dz), pr.paths, b, n_blocks=2, n_seg=n_seg,
                     min_len=spec.min_len)
        r.set_params(lam=0.7, N=0, alpha=0.5)
        r.set_image(x0)
        for t in range(2):
            keep = (row >= bp[t]) & (row < bp[t + 1])
            want = np.bincount(s.col[keep], (s.val * fac[row])[keep], minlength=spec.V)
            got, ss = r.drop_block_partial(t)
            assert rel_l2(got, want) <= 1e-4
            assert abs(ss - (res[bp[t]:bp[t + 1]] ** 2).sum()) <= 2e-4 * (res[bp[t]:bp[t + 1]] ** 2).sum()
    finally:
        r.close()
