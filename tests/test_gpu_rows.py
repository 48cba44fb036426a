"""Predictions of many rows a block (64 and 128 test rows a CTA, whole and partial tiles) against the same rows in
small calls (16 rows a CTA).

A row's FP32 operations do not depend on the rows it shares a CTA with; the sums in pairs of floats carry 48 bits, so
over a few thousand terms the two may differ by about 2^-48 x 4,096 = 1.5e-11 relative to the prior's scale.  The
bound is 1e-9."""
import numpy as np
import pytest

from workloads import make_random_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [16, 129, 701, 2003])
@pytest.mark.parametrize("s", [30, 65])
def test_rows_per_cta(rows, s):
    import paper_1411_4510_gb300 as L
    p = make_random_problem(rows + s, (70, 129, 64, 61), d=3, s=s, B=1, test_sizes=(rows, rows - 5, rows, rows - 1))
    model = L.lma_fit(precision=L.MIXED, **L.problem_args(p))
    mean, var = (np.asarray(x) for x in L.lma_predict(model, p.XU, p.test_block_ptr))
    ptr = np.asarray(p.test_block_ptr)
    for start in (0, rows // 2, rows - 9):
        idx = [np.arange(ptr[m] + min(start, ptr[m + 1] - ptr[m] - 4), ptr[m + 1])[:4] for m in range(4)]
        sub = np.concatenate(idx)
        m2, v2 = (np.asarray(x) for x in L.lma_predict(model, p.XU[sub], np.array([0, 4, 8, 12, 16], dtype=np.int64)))
        scale = np.abs(mean).max()
        assert np.abs(m2 - mean[sub]).max() <= 1e-9 * scale
        assert np.abs(v2 - var[sub]).max() <= 1e-9 * np.abs(var).max()
