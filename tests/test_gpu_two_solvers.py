"""A solver keeps working after another one with smaller subgraphs was set up: the shared memory that a kernel
may take belongs to the kernel, not to the solver that came last.
"""
import numpy as np
import pytest

from paper_0807_1949_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


CUBE, SQUARE = ((33, 17, 17), (16, 16, 16)), ((80, 40), (40, 40))


@pytest.mark.parametrize("precision,nrhs,variant,case", [
    ("fp64", 1, "single", CUBE), ("fp32", 1, "single", CUBE), ("fp32", 2, "pipelined", CUBE), ("fp64", 8, "single", SQUARE),
    ("fp64", 16, "auto", SQUARE), ("fp32", 16, "simt", CUBE)])
def test_smaller_solver_set_up_later(vtmlib, precision, nrhs, variant, case):
    def make(dims, block):
        A = inputs.grid_poisson(dims, sigma=0.5, seed=2)
        part = vtmlib.partition_evs(A, "grid", dims=dims, block=block)
        return A, vtmlib.Solver(part, z=1.0, precision=precision, nrhs=nrhs, form="band", sweep_variant=variant)

    def sweeps(A, s):
        s.set_rhs(inputs.rhs_uniform(A.n, nrhs, seed=2))
        s.reset()
        s.iterate(3)
        return s.get_state()
    ref = sweeps(*make(*case))
    A, big = make(*case)
    B, small = make((9, 8), (4, 4))
    assert np.array_equal(ref, sweeps(A, big))  # its first sweeps: nothing recorded before the other's setup
    assert np.all(np.isfinite(sweeps(B, small)))
