"""Products of the port sweep whose operands are split into 16-bit terms, port by port.

The system is diagonal: every vertex is shared by the two subgraphs and joined by one line (Z = 1), so a
subgraph's S_j is diagonal and a port's next wave is one product: w_out = 2 S_pp w_in - w_in with
S_pp = 1 / (a / 2 + 1), the same for both ends of the line.  vtm_iterate(2) is one port sweep and one band
sweep; sums play no part, so nothing hides a product that lost its operand's lower bits.
"""
import numpy as np
import pytest

from paper_0807_1949_gb300 import inputs
from test_precision_bounds import TOL_FP16

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

N = 1500  # S_j of 9 MB as a dense matrix: the tiled sweeps of port.cu, not the resident one


def _two_sweeps(vtmlib, a, w, storage):
    """Waves after two sweeps from w (nrhs, N), the same at both ends of a line; and those of FP64."""
    nrhs = len(w)
    A = inputs.CSR(n=N, rowptr=np.arange(N + 1, dtype=np.int64), col=np.arange(N, dtype=np.int32), val=a)
    part = vtmlib.partition_evs(A, "owners", owners=[(0, 1)] * N, lines=[(i, 0, 1) for i in range(N)])
    vertex = part.lines()[:, 1]
    assert np.array_equal(vertex, part.lines()[:, 3])  # both subgraphs hold every vertex, in order
    s = vtmlib.Solver(part, z=1.0, precision="fp32", nrhs=nrhs, form="port", port_storage=storage)
    s.set_rhs(np.zeros((nrhs, N)))
    s.reset()
    s.set_state(np.repeat(w[:, vertex], 2, axis=1))
    s.iterate(2)
    got = s.get_state()
    assert np.array_equal(got[:, 0::2], got[:, 1::2])
    out = np.empty_like(w)
    out[:, vertex] = got[:, 0::2]
    return out, (2.0 / (a / 2 + 1.0) - 1.0) ** 2 * w


@pytest.mark.parametrize("nrhs", [1, 2, 4, 8])
def test_fp16_storage_keeps_small_waves(vtmlib, nrhs):
    """Waves of a subgraph that differ by up to 2^34: every port's next wave within the rounding of the
    FP16 storage (S_pp within 0.9 .. 0.99 of its tile's largest entry: 2^-12 / 0.9 of S_pp, times
    2 S_pp / (2 S_pp - 1) <= 2.25 in the wave: 6.1e-4, below TOL_FP16), the smallest included."""
    rng = np.random.default_rng(nrhs)
    a = rng.uniform(0.02, 0.2, N)
    w = rng.uniform(0.5, 1.0, (nrhs, N)) * rng.choice([-1.0, 1.0], (nrhs, N))
    w *= 2.0 ** -rng.choice([0, 7, 13, 20, 26, 34], (nrhs, N))
    w = w.astype(np.float32).astype(np.float64)
    got, ref = _two_sweeps(vtmlib, a, w, "fp16")
    assert np.max(np.abs(got / ref - 1.0)) <= TOL_FP16


@pytest.mark.parametrize("nrhs", [2, 4, 8])
def test_fp32_products_have_no_bias(vtmlib, nrhs):
    """The first column's waves are 1 (its products are exact), the others' have every bit below their
    first bf16 term set, so that left-out term products are as large as they get.  FP32 roundings
    (2^-24 each, of either sign) cancel in the mean over the ports; a loss towards zero does not."""
    rng = np.random.default_rng(nrhs)
    a = rng.uniform(0.02, 0.2, N)
    x = np.array([0x3F800000, 0x3F80FFFF, 0x3F81FFFF, 0x3F80FFFD, 0x3F83FFFF, 0x3F80FFFB, 0x3F80FFFF, 0x3F81FFFD],
                 np.uint32).view(np.float32).astype(np.float64)[:nrhs]
    got, _ = _two_sweeps(vtmlib, a, np.repeat(x[:, None], N, axis=1), "native")
    err = got[1:] / (got[0] * x[1:, None]) - 1.0
    assert np.max(np.abs(np.mean(err, axis=1))) <= 2.0 ** -24
