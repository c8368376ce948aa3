"""The one-pass residual norms of the allocation-free entry point: every number of right-hand sides, sizes
around a block of rows, rows longer than one batch of entries, against numpy (FP64, rtol 1e-12: sums of
at most 1e5 terms of one sign).
"""
import numpy as np
import pytest

from paper_0807_1949_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("nrhs", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("n,degree", [(2, 1.0), (255, 6.0), (257, 30.0), (70001, 5.0)])
def test_norms(vtmlib, n, degree, nrhs):
    A = inputs.random_dd_spd(n, avg_degree=degree, seed=n)
    rng = np.random.default_rng(nrhs)
    b, x = rng.uniform(-1, 1, (nrhs, n)), rng.uniform(-1, 1, (nrhs, n))
    dev = [torch.tensor(a, device="cuda") for a in (A.rowptr, A.col, A.val, b, x)]
    rel = torch.full((nrhs,), float("nan"), dtype=torch.float64, device="cuda")
    vtmlib.relative_residual_noalloc(*dev, rel)
    torch.cuda.synchronize()
    ref = np.linalg.norm(b - (A.to_scipy() @ x.T).T, axis=1) / np.linalg.norm(b, axis=1)
    assert np.allclose(rel.cpu().numpy(), ref, rtol=1e-12, atol=0)
