"""A fit in the FP64 form keeps no page-locked host memory that grows with the factorisation's work."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _resident_mb():
    with open("/proc/self/status") as fh:
        return next(int(ln.split()[1]) for ln in fh if ln.startswith("VmRSS")) / 1024


def test_fp64_fit_uploads_little(capsys):
    """16,384 windows of 64 points with 513 extra rows: 2.3 million 16 x 16 tiles, 36 MB as a list of them.  What has to
    be uploaded is a descriptor of each window (about 100 bytes, 2 MB, in a buffer that doubles)."""
    import torch
    import paper_1411_4510_gb300 as L
    dev = torch.device("cuda")
    g = torch.Generator(device="cuda")
    g.manual_seed(1)

    def fit(blocks):
        X = torch.rand(64 * blocks, 2, dtype=torch.float64, device=dev, generator=g)
        y = torch.sin(6 * X[:, 0])
        S = X[torch.randperm(len(X), device=dev, generator=g)[:512]].contiguous()
        L.lma_fit(X, y, 64 * np.arange(blocks + 1), S, 0, [-1.5, -1.5], 0.0, -1.0, jitter=1e-4, precision=L.FP64)
        torch.cuda.synchronize()

    L.lma_autotune(False)
    fit(128)  # everything that a first call loads
    before = _resident_mb()
    fit(16384)
    grown = _resident_mb() - before
    L.lma_autotune(True)
    L.lma_workspace_release()
    assert grown <= 16, f"{grown:.1f} MB more resident host memory after the fit"
