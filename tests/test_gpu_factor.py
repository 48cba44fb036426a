"""The FP64 dataflow factorisation of Sigma_SS and I + A and the FP32 diagonal
block factorisation at the edges of their tiles, against the oracle.

The bounds are the repository's: 1e-9 for the FP64 form; for the mixed form
1e-4 on the mean and, as FP32 windows allow, 6e-4 on the variance and 1.5e-4 on
the log-likelihood."""
import numpy as np
import pytest

from oracle import lma_oracle as O2
from workloads import make_random_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import paper_1411_4510_gb300 as L
    yield L
    L.lma_autotune_pin(None)


def _rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b)))


def _errors(L, p, precision):
    f = O2.fit(p)
    m_ref, v_ref = O2.predict(f)
    model = L.lma_fit(precision=precision, **L.problem_args(p))
    assert L.lma_model_precision(model) == precision
    mean, var = L.lma_predict(model, p.XU, p.test_block_ptr)
    return _rel(mean, m_ref), _rel(var, v_ref), abs(L.lma_model_loglik(model) - f.loglik) / abs(f.loglik)


@pytest.mark.parametrize("s", [1, 15, 16, 17, 32, 33, 47, 49, 64, 65, 161])
def test_dataflow_factor_at_tile_edges(L, s):
    """One to eleven 16-column panels, the last one full or not, with the appended identity rows and the y row."""
    p = make_random_problem(40 + s, (60, 55, 70), d=3, s=s, B=1, test_sizes=(5, 0, 7))
    L.lma_autotune_pin(None)
    L.lma_autotune_pin("fp64 factor", 5)
    em, ev, el = _errors(L, p, L.FP64)
    assert em <= 1e-9 and ev <= 1e-9 and el <= 1e-9, (em, ev, el)


@pytest.mark.parametrize("sizes", [(1, 1, 1), (63, 1, 64), (64, 64, 64), (65, 63, 66), (129, 128, 1)])
def test_diagonal_blocks_at_tile_edges(L, sizes):
    """Windows of one to five 64-column panels, full and padded ones, first and second panels of a group."""
    p = make_random_problem(7, sizes, d=2, s=min(20, sum(sizes)), B=1, test_sizes=(3, 4, 5))
    em, ev, el = _errors(L, p, L.MIXED)
    assert em <= 1e-4 and ev <= 6e-4 and el <= 1.5e-4, (em, ev, el)


@pytest.mark.parametrize("sizes, s, B", [((1, 1, 1, 1), 3, 3), ((15, 17, 1, 16, 33), 18, 2), ([5 + k % 13 for k in range(71)], 9, 3),
                                         ((70, 200, 30, 90), 40, 1)])
def test_fp64_windows_at_tile_edges(L, sizes, s, B):
    """Windows of one point up to seventeen 16-column panels, more windows than one launch and than its chains take,
    test blocks of no, one and more than 16 points; the gradient reads the 64-wide inverses."""
    test_sizes = [(0, 1, 17, 5)[k % 4] for k in range(len(sizes))]
    p = make_random_problem(11, sizes, d=3, s=s, B=B, test_sizes=test_sizes)
    em, ev, el = _errors(L, p, L.FP64)
    assert em <= 1e-9 and ev <= 1e-9 and el <= 1e-9, (em, ev, el)
    _, g = L.lma_loglik_grad(precision=L.FP64, **L.problem_args(p))
    assert _rel(g, O2.loglik_grad(p)[1]) <= 1e-9


@pytest.mark.parametrize("d, s", [(9, 77), (3, 128)])
def test_mixed_gradient_products_at_tile_edges(L, d, s):
    """N x s products of the adjoint on 64-wide tiles with ragged edges, input dimensions padded to 8 and to 24 (the
    128-wide tiles run in the full-size gradient test).  Bound: the mixed gradient's 5e-4."""
    n = 333
    p = make_random_problem(5, [n // 9] * 8 + [n - 8 * (n // 9)], d=d, s=s, B=1, ell=0.06 + 0.08 * d, sigma_n=0.2)
    _, g = L.lma_loglik_grad(precision=L.MIXED, **L.problem_args(p))
    assert _rel(g, O2.loglik_grad(p)[1]) <= 5e-4


@pytest.mark.parametrize("s", [1001, 900])
def test_adjoint_128_wide_tiles_equal_64_wide_ones(L, s):
    """The gradient of a whole fit (128-wide tiles: 4,871 points, rows of s values aligned or not) against the sum of
    the gradients of two shards of its blocks (64-wide ones).  The terms are the same, each shard's Vt-bar is rounded to
    FP32 by itself and its K-sums run over its own points: 2^-24 per operation over sums whose terms cancel by up to
    about 1e3 leaves 1e-4 of the gradient."""
    n, nb = 4871, 9
    p = make_random_problem(5, [n // nb] * (nb - 1) + [n - (nb - 1) * (n // nb)], d=8, s=s, B=0, ell=0.7, sigma_n=0.2)
    args = L.problem_args(p)
    _, g = L.lma_loglik_grad(precision=L.MIXED, **args)
    ptr, parts = p.block_ptr, []
    for b0, b1 in ((0, 2), (2, 4), (4, 6), (6, 8), (8, 9)):
        rows = slice(ptr[b0], ptr[b1])
        sub = dict(args, X=p.X[rows], y=p.y[rows], block_ptr=ptr[b0:b1 + 1] - ptr[b0])
        m = L.lma_fit_local(win_begin=0, own_begin=0, own_end=b1 - b0, precision=L.MIXED, **sub)
        parts.append((m, *L.lma_model_local_summary(m)))
    G, ld = sum(x[1] for x in parts), sum(x[2] for x in parts)
    total = 0.0
    for m, _, _ in parts:
        L.lma_model_set_global(m, G, ld, n)
        total = total + L.lma_model_loglik_grad(m)
    # the support-set term's partial sums are per shard: everything after the window terms is linear in them
    assert _rel(total, g) <= 1e-4
