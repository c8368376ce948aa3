"""The tiled port sweep of subgraphs with very many ports, where its vectors leave no room for the usual
shape: no accumulator per warp (one or two right-hand sides), the SIMT products with and without gaps in the
vectors, no shared-memory slots for the tiles.

Every vertex of an nx x ny grid is shared by both subgraphs, so all are ports and the half-bandwidth is nx;
Z = 30 lets the port responses reach over several rows of tiles.  Tolerances as in test_gpu_port.
"""
import numpy as np
import pytest

from oracle import evs
from paper_0807_1949_gb300 import inputs
from test_precision_bounds import TOL_FP16, TOL_FP32  # noqa: F401
from test_gpu_parity import _line_map, _oracle_after, _rel

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

TOL = {"fp64": 1e-12, "fp32": TOL_FP32, "fp16": TOL_FP16}


@pytest.mark.parametrize("kind,nrhs,nx,ny", [
    ("fp32", 1, 40, 60), ("fp64", 1, 40, 60), ("fp16", 1, 40, 46),   # one accumulator for all warps
    ("fp32", 2, 30, 41), ("fp64", 2, 30, 41), ("fp16", 2, 30, 31),
    ("fp32", 8, 40, 61), ("fp32", 8, 40, 68), ("fp32", 8, 50, 63),   # SIMT: gaps, no gaps, no slots
    ("fp32", 4, 50, 100), ("fp32", 4, 60, 104), ("fp32", 2, 12, 1033),  # no gaps, no slots, no slots
    ("fp16", 8, 45, 72), ("fp16", 8, 12, 272), ("fp16", 4, 12, 550), ("fp16", 2, 12, 1105),  # SIMT: slots, none
    ("fp64", 8, 35, 35), ("fp64", 4, 50, 52)])                       # no slots
def test_many_ports(vtmlib, kind, nrhs, nx, ny):
    A = inputs.grid_poisson((nx, ny), sigma=0.5, seed=nx)
    owners = [(0, 1)] * A.n
    lines = [(i, 0, 1) for i in range(A.n)]
    part = vtmlib.partition_evs(A, "owners", owners=owners, lines=lines)
    osplit = evs.split_by_owners(A.to_scipy(), owners, lines)
    b = inputs.rhs_uniform(A.n, nrhs, seed=3)
    s = vtmlib.Solver(part, z=30.0, precision="fp64" if kind == "fp64" else "fp32", nrhs=nrhs, form="port",
                      port_storage="fp16" if kind == "fp16" else "native")
    assert s.info().port_kernel == vtmlib.PORT_TILES and s.info().nports == 2 * nx * ny
    assert s.info().flagged_pieces == 0
    s.set_rhs(b)
    s.reset()
    s.iterate(4)
    copies, waves = _oracle_after(osplit, b, 30.0, 4)
    assert _rel(s.copies(), copies) <= TOL[kind]
    assert _rel(s.get_state(), waves[:, _line_map(part, osplit)]) <= TOL[kind]
    first = s.get_state()
    s.reset()
    s.iterate(4)
    assert np.array_equal(first, s.get_state())
