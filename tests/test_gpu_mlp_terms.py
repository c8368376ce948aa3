"""The gradient kernel's sums over samples, which multiply operands split into three bf16 terms, at the
values where a lost term product or a cut-off sum shows.

* One sample: dW1[j][k] = d1[j] x[k] is one product, and db1[j] = d1[j] comes back exactly (its three
  terms add up to it in 24 bits).  x has every mantissa bit below its first bf16 term set, so that the
  terms of the products are as large as they get.  FP32 rounds a product by 2^-24; the products of terms
  that are left out are at most 2^-24 more: 2^-23 in all.
* 64 equal samples: each sum is 64 times a sample's share of 1/64, so the biases' gradients are one
  sample's.  Sums of 16 equal values are exact, and of the additions of four such sums only 48 d rounds:
  at most half a unit there and half a unit of the result, 2^-23 in all, of either sign (in the mean
  over 128 units below 2^-25).  A sum that cuts off errs towards zero every time.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

B1, W2, B2, W3 = 512, 576, 4672, 4736  # offsets of the parameter blocks


def _grad(vtmlib, seed, n):
    x = np.array([0x3F80FFFF, 0x3F81FFFF, 0xBF80FFFF, 0x3F82FFFD, 0x3F80FFF7, 0xBF85FFFF, 0x3F87FFFF, 0x3F80FFFF],
                 np.uint32).view(np.float32)
    m = vtmlib.MLP(seed=seed)
    X = torch.tensor(np.tile(x, (n, 1)), device="cuda")
    m.loss_grad(X, torch.full((n,), 0.3137, device="cuda"))
    return x.astype(np.float64), m.get_grads().astype(np.float64)


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_one_sample_products(vtmlib, seed):
    x, g = _grad(vtmlib, seed, 1)
    d1 = g[B1:W2]
    live = d1 != 0
    assert live.sum() >= 16
    err = g[:B1].reshape(64, 8)[live] / (d1[live, None] * x[None, :]) - 1.0
    assert np.max(np.abs(err)) <= 2.0 ** -23


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_equal_samples_bias_sums(vtmlib, seed):
    _, one = _grad(vtmlib, seed, 1)
    _, many = _grad(vtmlib, seed, 64)
    one = np.concatenate([one[B1:W2], one[B2:W3]])
    many = np.concatenate([many[B1:W2], many[B2:W3]])
    assert np.array_equal(one == 0, many == 0)
    err = many[one != 0] / one[one != 0] - 1.0
    assert np.max(np.abs(err)) <= 2.0 ** -23 and abs(np.mean(err)) <= 2.0 ** -25
