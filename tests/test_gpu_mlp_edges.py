"""The perceptron's tensor-core kernels at the edges of their tiles (16 samples per warp, 64 per CTA of
the gradient) and with inputs that are not 8-byte aligned, against the FP64 oracle.

Tolerance 1e-5 of the largest value: FP32 sums of at most 64 terms (outputs) or of exact bf16-term
products over the samples (gradients) stay below 64 x 2^-24 x the sum of magnitudes, a few times the
largest value here.
"""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("n", [1, 7, 16, 17, 63, 64, 65, 129, 20011])
@pytest.mark.parametrize("shift", [0, 1])
def test_tile_edges(vtmlib, n, shift):
    rng = np.random.default_rng(n)
    X = rng.normal(0, 1.5, (n, 8)).astype(np.float32)
    t = rng.normal(0, 1, n).astype(np.float32)
    m = vtmlib.MLP(seed=2)
    flat = torch.zeros(8 * n + 1, device="cuda")
    Xd = flat[shift:shift + 8 * n].view(n, 8)
    Xd.copy_(torch.tensor(X))
    td = torch.tensor(t, device="cuda")
    y = torch.full((n + 1,), 7.0, device="cuda")
    m.forward(Xd, y[:n])
    torch.cuda.synchronize()
    pb = omlp.bf16_round(m.get_params())
    yref, _ = omlp.forward(pb, X)
    got = y.cpu().numpy()
    assert np.max(np.abs(got[:n] - yref)) <= 1e-5 * np.max(np.abs(yref)) and got[n] == 7.0
    loss = m.loss_grad(Xd, td)
    lref, gref = omlp.loss_and_grad(pb, X, t)
    g = m.get_grads()
    assert abs(loss - lref) <= 1e-5 * lref
    assert np.max(np.abs(g - gref)) <= 1e-5 * np.max(np.abs(gref))
    assert m.loss_grad(Xd, td) == loss and np.array_equal(g, m.get_grads())
