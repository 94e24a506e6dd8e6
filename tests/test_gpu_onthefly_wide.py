"""Traced DROP rows on grids past 430 voxels a side, where a warp's piece buffer takes its two larger
sizes: rows that fit them and rows that overflow them, against an FP64 evaluation of the generator's
stored rows (scatter numerators, as in test_gpu_onthefly_buffer).

FP32 tracing places a crossing within about 4 ulp of its coordinate, at most half the grid's width, on
pieces of about 0.7 mm."""
import numpy as np
import pytest

import synth
from _gpu_util import ntvs_module, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,n_seg,n_hist", [
    (520, 510, 2, 16, 701),      # two CTAs an SM: rows near the diagonal overflow
    (640, 600, 1, 16, 601),      # one CTA an SM: everything fits
    (1000, 950, 1, 16, 601),     # rows near the diagonal overflow it
    (1100, 1000, 1, 16, 401),    # no buffer: every row is walked twice
])
def test_traced_delta_on_wide_grids(nx, ny, nz, n_seg, n_hist):
    ntvs = ntvs_module()
    spec = synth.spec_scaled_3d(nx=nx, ny=ny, nz=nz, n_hist=n_hist, n_angles=24, n_blocks=1,
                                seed=n_seg).replace(n_seg=n_seg)
    s, pr = synth.generate(spec), synth.generate_paths(spec)
    tol = 4 * float(np.spacing(np.float32(0.5 * max(nx * spec.dx, ny * spec.dy)))) / 0.7
    b = pr.b.astype(np.float32)
    x0 = np.random.default_rng(3).uniform(0.0, 1.0, spec.V)
    row = np.repeat(np.arange(s.M), np.diff(s.row_ptr))
    dot = np.bincount(row, s.val * x0[s.col], minlength=s.M)
    n2 = np.bincount(row, s.val ** 2, minlength=s.M)
    res = np.where(n2 > 0, b - dot, b).astype(np.float64)
    want = np.bincount(s.col, (s.val * np.where(n2 > 0, 0.7 * res / np.maximum(n2, 1e-300), 0.0)[row]),
                       minlength=spec.V)
    r = ntvs.Reconstructor(0)
    try:
        r.load_paths((nx, ny, nz), (spec.dx, spec.dy, spec.dz), pr.paths, b, n_seg=n_seg, min_len=spec.min_len)
        r.set_params(lam=0.7, N=0, alpha=0.5)
        r.set_image(x0)
        got, ss = r.drop_block_partial(0)
    finally:
        r.close()
    assert rel_l2(got, want) <= tol
    assert abs(ss - (res ** 2).sum()) <= 2 * tol * (res ** 2).sum()
