"""The divided and the resident port sweeps at the sizes where they can go wrong, against the oracle.

Tolerances are those of the sweeps' precision (test_precision_bounds): FP64 1e-12, FP32 TOL_FP32, FP16
storage TOL_FP16 (max norm of copies and waves after k sweeps, relative to the largest entry).
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


def _check(vtmlib, dims, block, nrhs, precision, storage, sweeps, tol):
    A = inputs.grid_poisson(dims, sigma=0.8, seed=5)
    b = inputs.rhs_uniform(A.n, nrhs, seed=5)
    part = vtmlib.partition_evs(A, "grid", dims=dims, block=block)
    osplit = evs.split_grid(A, dims, block)
    s = vtmlib.Solver(part, z=0.9, precision=precision, nrhs=nrhs, form="port", port_storage=storage)
    assert s.info().sweep_form == 2
    s.set_rhs(b)
    s.reset()
    s.iterate(sweeps)
    copies, waves = _oracle_after(osplit, b, 0.9, sweeps)
    assert _rel(s.copies(), copies) <= tol
    assert _rel(s.get_state(), waves[:, _line_map(part, osplit)]) <= tol
    first = s.get_state()
    s.reset()
    s.iterate(sweeps)
    assert np.array_equal(first, s.get_state())  # fixed order of sums


# 27 ragged subgraphs of up to 13 rows of tiles, divided among all CTAs; two subgraphs of a few tiles
@pytest.mark.parametrize("nrhs", [1, 2, 4, 8])
@pytest.mark.parametrize("kind", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("dims,block", [((21, 19, 18), (8, 8, 8)), ((9, 8, 15), (9, 8, 7))])
def test_divided_sweep(vtmlib, dims, block, nrhs, kind):
    _check(vtmlib, dims, block, nrhs, "fp64" if kind == "fp64" else "fp32", "fp16" if kind == "fp16" else "native", 6,
           TOL[kind])


# subgraphs of up to 1000 ports with eight right-hand sides: one CTA of 16 warps per SM
def test_divided_sweep_large(vtmlib):
    _check(vtmlib, (40, 34, 47), (13, 11, 16), 8, "fp32", "native", 4, TOL["fp32"])


# one CTA per subgraph and several subgraphs per CTA, every number of right-hand sides; two sweeps
# (one resident sweep), three, and enough for both exchange buffers to be used again
@pytest.mark.parametrize("nrhs,kind", [(1, "fp64"), (2, "fp64"), (4, "fp64"), (8, "fp64"), (1, "fp32"), (2, "fp32"),
                                       (4, "fp32"), (8, "fp32"), (16, "fp32"), (32, "fp32")])
@pytest.mark.parametrize("dims,block,sweeps", [((40, 33), (13, 11), 7), ((40, 33), (13, 11), 2), ((23, 5), (3, 4), 3),
                                               ((97, 83), (5, 6), 5)])
def test_resident_sweep(vtmlib, dims, block, sweeps, nrhs, kind):
    _check(vtmlib, dims, block, nrhs, kind, "native", sweeps, TOL[kind])


# the pipelined band sweep with several chain warps: half-bandwidths below 32, around 64 and above,
# last blocks cut short, one block only, one subgraph without lines
@pytest.mark.parametrize("nrhs", [1, 2, 4, 8])
@pytest.mark.parametrize("dims,block", [((21, 19, 18), (8, 8, 8)), ((23, 17), (6, 5)), ((70, 9), (70, 9)),
                                        ((64, 31), (63, 31)), ((67, 40), (33, 20))])
def test_pipelined_band_sweep(vtmlib, dims, block, nrhs):
    A = inputs.grid_poisson(dims, sigma=0.7, seed=8)
    b = inputs.rhs_uniform(A.n, nrhs, seed=8)
    part = vtmlib.partition_evs(A, "grid", dims=dims, block=block)
    osplit = evs.split_grid(A, dims, block)
    s = vtmlib.Solver(part, z=0.9, precision="fp32", nrhs=nrhs, form="band")
    assert s.info().sweep_variant == 1
    s.set_rhs(b)
    s.reset()
    s.iterate(4)
    copies, waves = _oracle_after(osplit, b, 0.9, 4)
    assert _rel(s.copies(), copies) <= TOL_FP32
    if len(osplit.vtl):
        assert _rel(s.get_state(), waves[:, _line_map(part, osplit)]) <= TOL_FP32


# tensor-core port sweep, port vectors in a launch of their own: 75 subgraphs of up to four super-rows cut
# in two, 8 of six cut into more (FP16; their FP32 responses stay resident); fused: 504 of one to three
@pytest.mark.parametrize("nrhs", [16, 32])
@pytest.mark.parametrize("kind", ["fp32", "fp16"])
@pytest.mark.parametrize("dims,block", [((40, 37, 21), (8, 8, 8)), ((26, 26, 26), (13, 13, 13)),
                                        ((52, 47, 41), (6, 6, 6))])
def test_tensor_core_sweep(vtmlib, dims, block, nrhs, kind):
    _check(vtmlib, dims, block, nrhs, "fp32", "fp16" if kind == "fp16" else "native", 6, TOL[kind])


# port responses from the band kernels without the tensor cores (half-bandwidth above 384) and with them
# (385 > w): the batches start at the first row they need, here deep inside the subgraph
@pytest.mark.parametrize("dims,block,nrhs,kind", [((41, 20, 21), (20, 20, 21), 1, "fp32"),
                                                  ((41, 20, 21), (20, 20, 21), 16, "fp32"),
                                                  ((37, 19, 18), (18, 19, 18), 1, "fp32"),
                                                  ((37, 19, 18), (18, 19, 18), 16, "fp32"),
                                                  ((27, 13, 12), (13, 13, 12), 1, "fp64")])
def test_port_response(vtmlib, dims, block, nrhs, kind):
    _check(vtmlib, dims, block, nrhs, kind, "native", 4, TOL[kind])
