"""Forward projection at the edges of its rows-per-warp rule (a warp takes 1 to 8 rows by their number;
8 CTAs of 8 warps on each of 152 SMs: 9728 warps), with rows from empty to long, against NumPy."""
import math

import numpy as np
import pytest

from _gpu_util import ntvs_module

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("M,longest", [(1, 5000), (7, 2049), (300, 3000), (9728, 9), (9729, 300), (68097, 20), (77825, 12)])
def test_projection_by_number_of_rows(M, longest, dtype):
    ntvs = ntvs_module()
    rng = np.random.default_rng(M)
    shape = (40, 30, 6)
    V = int(np.prod(shape))
    n = rng.integers(0, longest + 1, M)
    n[-1] = longest
    rp = np.zeros(M + 1, np.int64)
    np.cumsum(n, out=rp[1:])
    col = rng.integers(0, V, rp[-1]).astype(np.int32)
    val = rng.uniform(0.1, 1.5, rp[-1]).astype(dtype)
    x = rng.uniform(0.0, 1.0, V).astype(dtype)
    terms = val.astype(np.float64) * x[col]
    want = np.array([math.fsum(terms[p:q]) for p, q in zip(rp[:-1], rp[1:])])   # correctly rounded sums
    r = ntvs.Reconstructor(0)
    try:
        r.load(shape, rp, col, val, np.zeros(M, dtype))
        got = r.forward_project(x)
    finally:
        r.close()
    # a lane sums a 32nd of the row, then five more sums: each rounding within half an ulp of the total
    eps = np.finfo(dtype).eps * 0.5 * (n / 32 + 7)
    assert np.all(np.abs(got - want) <= eps * want + 1e-300)
