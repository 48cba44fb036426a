"""The mixed form's gradient with a training point far from every support point.

Such a pair's covariance is 0 in FP64 and in FP32, so it adds nothing to the gradient: the FP64 form stays finite at
any distance, and the mixed form has to agree with it within its bound of 5e-4.  The far point is a block of its own
without a Markov blanket, so that no window holds two points at that distance (the residual's covariances inside a
window are not what is looked at here)."""
import numpy as np
import pytest

from workloads import make_random_problem

pytestmark = pytest.mark.gpu


def _far_problem(sizes, d, s, lengths, seed=21, **kw):
    p = make_random_problem(seed, sizes + (1,), d=d, s=s, B=0, sigma_n=0.2, **kw)
    near = np.random.default_rng(seed).choice(sum(sizes), size=s, replace=False)
    p.S = p.X[np.sort(near)].copy()
    p.X[-1, 0] += lengths * np.exp(p.log_ell[0])
    return p


@pytest.mark.parametrize("lengths", [45.0, 1.4e4, 1.4e6, 3e9, 1e20])
@pytest.mark.parametrize("sizes, d, s", [((60, 70, 65), 2, 33), ((40, 90), 11, 40), ((1200,) * 4, 3, 1001)])
def test_gradient_with_a_far_point(sizes, d, s, lengths):
    """d2 / 2 from 1e3 through 1e8, 1e12 and 5e18 to beyond the range of a float, on 64-wide tiles with the dimension
    padded to 8 and to 24, and on 128-wide ones."""
    import paper_1411_4510_gb300 as L
    p = _far_problem(sizes, d, s, lengths, ell=0.15 if d == 3 else 0.4)
    ll64, g64 = L.lma_loglik_grad(precision=L.FP64, **L.problem_args(p))
    ll, g = L.lma_loglik_grad(precision=L.MIXED, **L.problem_args(p))
    assert np.isfinite(ll64) and np.all(np.isfinite(g64))
    assert np.isfinite(ll) and np.all(np.isfinite(g)), g
    assert np.linalg.norm(g - g64) <= 5e-4 * np.linalg.norm(g64)
