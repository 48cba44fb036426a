"""The 128-wide N x s products of the mixed gradient at ragged edges, against the oracle's adjoint.

N follows from the device: the wide tiles run where there are at least two for every SM (at N x s of this test three).
Short length-scales in 8 and 9 dimensions and a noise of 0.3 keep the covariances near their diagonal, so that the bound
of the mixed gradient, 5e-4, is what FP32 leaves."""
import numpy as np
import pytest

from workloads import make_random_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d, s", [(8, 901), (9, 900)])
def test_wide_adjoint_matches_oracle(d, s):
    import torch
    import paper_1411_4510_gb300 as L
    from oracle import lma_oracle as O2
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 128 * -(-3 * sms // -(-s // 128)) + 71
    blocks = 17
    p = make_random_problem(8, [n // blocks] * (blocks - 1) + [n - (blocks - 1) * (n // blocks)], d=d, s=s, B=1, ell=0.35,
                            sigma_n=0.3, test_sizes=np.zeros(blocks, dtype=np.int64))
    assert -(-n // 128) * -(-s // 128) >= 2 * sms
    ll_ref, g_ref = O2.loglik_grad(p)
    ll, g = L.lma_loglik_grad(precision=L.MIXED, **L.problem_args(p))
    assert abs(ll - ll_ref) <= 1.5e-4 * abs(ll_ref)
    assert np.linalg.norm(g - g_ref) <= 5e-4 * np.linalg.norm(g_ref)
