"""The resident port sweep's bounded waits: a wave that nothing publishes makes its reader's wait run out.

Nothing faults or hangs: the reader gives up after `wait_polls` loads and goes on without waiting, as does every
thread that then waits in vain, the launch ends, the solve reports VTM_ERR_TIMEOUT and the context stays
usable.
"""
import numpy as np
import pytest

from paper_0807_1949_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("precision,nrhs,coupling", [("fp64", 1, None), ("fp32", 1, 1.0), ("fp64", 8, None), ("fp32", 16, None),
                                                     ("fp32", 32, 1.0)])
def test_withheld_wave(vtmlib, precision, nrhs, coupling):
    dims, block = (40, 36), (16, 12)
    A = inputs.grid_poisson(dims, sigma=0.5, seed=1)
    part = vtmlib.partition_evs(A, "grid", dims=dims, block=block)
    b = inputs.rhs_uniform(A.n, nrhs, seed=1)
    x = np.zeros_like(b)
    s = vtmlib.Solver(part, z=1.0, precision=precision, nrhs=nrhs, form="port", coupling=coupling, wait_polls=2000,
                      withhold_wave=True)
    assert s.info().port_kernel == vtmlib.PORT_RESIDENT
    for _ in range(2):
        with pytest.raises(vtmlib.VTMError) as e:
            s.solve(b, x, rtol=1e-8, maxit=100)
        assert e.value.code == 7
    del s
    ok = vtmlib.Solver(part, z=1.0, precision=precision, nrhs=nrhs, form="port", coupling=coupling, wait_polls=2000)
    assert ok.solve(b, x, rtol=1e-8, maxit=20000).rel_residual <= 1e-8
