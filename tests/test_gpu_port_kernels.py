"""Which kernel runs the port sweeps (vtm_solver_info.port_kernel), and the ones that only systems of many
subgraphs reach, against the oracle.

Systems whose S_j fit into the SMs' shared memory run k_port_resident.  Beyond, nrhs <= 8 takes the tiled
sweep; nrhs 16 / 32 the tensor cores, with the port vectors in a launch of their own up to five items per SM
and fused into the sweep beyond.  Tolerances are those of the sweeps' precision (test_precision_bounds).
"""
import functools

import numpy as np
import pytest

from oracle import coupled, evs
from paper_0807_1949_gb300 import inputs
from test_precision_bounds import TOL_FP16, TOL_FP32  # noqa: F401
from test_gpu_parity import _line_map, _oracle_after, _rel

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

TOL = {"fp64": 1e-12, "fp32": TOL_FP32, "fp16": TOL_FP16}
NSM = torch.cuda.get_device_properties(0).multi_processor_count


@functools.lru_cache(maxsize=1)
def _split(dims, block):
    A = inputs.grid_poisson(dims, sigma=0.8, seed=5)
    return A, evs.split_grid(A, dims, block)


def _solver(vtmlib, dims, block, nrhs, kind, coupling=None):
    A, osplit = _split(dims, block)
    part = vtmlib.partition_evs(A, "grid", dims=dims, block=block)
    s = vtmlib.Solver(part, z=0.9, precision="fp64" if kind == "fp64" else "fp32", nrhs=nrhs, form="port",
                      port_storage="fp16" if kind == "fp16" else "native", coupling=coupling)
    return A, osplit, part, s


def _check(s, b, sweeps, copies, waves, tol):
    s.set_rhs(b)
    s.reset()
    s.iterate(sweeps)
    assert _rel(s.copies(), copies) <= tol
    assert _rel(s.get_state(), waves) <= tol
    first = s.get_state()
    s.reset()
    s.iterate(sweeps)
    assert np.array_equal(first, s.get_state())


# the cases of the other files' port tests, so that a change of the rules cannot move them unseen
@pytest.mark.parametrize("dims,block,nrhs,kind,kernel", [
    ((40, 33), (13, 11), 1, "fp64", "PORT_RESIDENT"), ((40, 33), (13, 11), 16, "fp32", "PORT_RESIDENT"),
    ((40, 33), (13, 11), 2, "fp16", "PORT_TILES"), ((40, 33), (13, 11), 16, "fp16", "PORT_TC_SEPARATE"),
    ((9, 8, 15), (9, 8, 7), 4, "fp32", "PORT_RESIDENT"), ((9, 8, 15), (9, 8, 7), 4, "fp16", "PORT_TILES"),
    ((34, 34, 34), (16, 16, 16), 1, "fp64", "PORT_TILES"), ((34, 34, 34), (16, 16, 16), 32, "fp32", "PORT_TC_SEPARATE"),
    ((52, 47, 41), (6, 6, 6), 16, "fp16", "PORT_TC_SEPARATE")])
def test_kernel_choice(vtmlib, dims, block, nrhs, kind, kernel):
    A, _, _, s = _solver(vtmlib, dims, block, nrhs, kind)
    i = s.info()
    assert i.port_kernel == getattr(vtmlib, kernel)
    if kernel == "PORT_RESIDENT":  # the dense S_j that a sweep reads from shared memory
        assert 0 < i.port_bytes <= NSM * 227 * 1024
    part = vtmlib.partition_evs(A, "grid", dims=dims, block=block)
    assert vtmlib.Solver(part, z=0.9, precision="fp32", form="band").info().port_kernel == vtmlib.PORT_NONE


# fused: more than five items per SM, so that both slots of the port vectors are used again; subgraphs of 91 to
# 152 ports, one and two super-rows.  Coupled lines: entries past the
# fourth of a port's list (a gather record holds four)
@pytest.mark.parametrize("nrhs,kind,gamma", [(16, "fp32", None), (32, "fp32", None), (16, "fp16", None),
                                             (32, "fp16", None), (32, "fp32", 1.0)])
def test_fused_port_vectors(vtmlib, nrhs, kind, gamma):
    nz = 5 * NSM // 100 + 1
    dims, block = (51, 51, 5 * nz + 1), (5, 5, 5)
    A, osplit, part, s = _solver(vtmlib, dims, block, nrhs, kind, gamma)
    assert s.info().port_kernel == vtmlib.PORT_TC_FUSED and s.info().npieces > 5 * NSM
    b = inputs.rhs_uniform(A.n, nrhs, seed=5)
    lm = _line_map(part, osplit)
    if gamma is None:
        copies, waves = _oracle_after(osplit, b, 0.9, 4)
    else:
        pr, w = part.line_pairs()
        Y = coupled.laplacian_admittance(osplit, 0.9, (lm[0::2] // 2)[pr], gamma * w)
        m = coupled.CoupledVTM(osplit, Y)
        st = m.initial_state(nrhs)
        for _ in range(4):
            st = m.sweep(st, b)
        copies, waves = np.concatenate(st.x_local, axis=1), m.waves_out(st)
    _check(s, b, 4, copies, waves[:, lm], TOL[kind])


# fused, with a subgraph that is cut between super-rows: 1512 cells of 2^3 vertices around one of 12^3 (1592 ports,
# 91 blocks, where a CTA's share of all is 40), whose items leave partial sums
@pytest.mark.parametrize("nrhs,kind", [(16, "fp32"), (32, "fp16")])
def test_fused_with_a_cut_subgraph(vtmlib, nrhs, kind):
    n, lo, hi = 24, 6, 18
    A = inputs.grid_poisson((n, n, n), sigma=0.8, seed=7)
    As = A.to_scipy()
    z, y, x = np.meshgrid(*(np.arange(n),) * 3, indexing="ij")
    cell = ((z // 2) * (n // 2) + y // 2) * (n // 2) + x // 2
    core = (x >= lo) & (x < hi) & (y >= lo) & (y < hi) & (z >= lo) & (z < hi)
    home = np.unique(np.where(core, -1, cell).ravel(), return_inverse=True)[1]
    owners = [tuple(sorted({int(home[i])} | {int(h) for h in home[As.indices[As.indptr[i]:As.indptr[i + 1]]]}))
              for i in range(A.n)]
    lines = [(i, p, q) for i, o in enumerate(owners) for a, p in enumerate(o) for q in o[a + 1:]]
    part = vtmlib.partition_evs(A, "owners", owners=owners, lines=lines)
    osplit = evs.split_by_owners(As, owners, lines)
    s = vtmlib.Solver(part, z=0.9, precision="fp32", nrhs=nrhs, form="port",
                      port_storage="fp16" if kind == "fp16" else "native")
    assert s.info().port_kernel == vtmlib.PORT_TC_FUSED and s.info().npieces == 1513 > 5 * NSM
    b = inputs.rhs_uniform(A.n, nrhs, seed=7)
    copies, waves = _oracle_after(osplit, b, 0.9, 4)
    _check(s, b, 4, copies, waves[:, _line_map(part, osplit)], TOL[kind])


# FP32 responses of single partial super-rows (up to 88 ports) that do not fit into shared memory: 750 subgraphs
@pytest.mark.parametrize("nrhs", [16, 32])
def test_tensor_core_single_super_row(vtmlib, nrhs):
    dims, block = (30 * 22 + 1, 25 * 22 + 1), (22, 22)
    A, osplit, part, s = _solver(vtmlib, dims, block, nrhs, "fp32")
    assert s.info().port_kernel == vtmlib.PORT_TC_SEPARATE
    b = inputs.rhs_uniform(A.n, nrhs, seed=5)
    copies, waves = _oracle_after(osplit, b, 0.9, 3)
    _check(s, b, 3, copies, waves[:, _line_map(part, osplit)], TOL_FP32)


# the tiled sweep's shortest segments, whole subgraphs of up to 72 ports (six tiles), several per CTA
@pytest.mark.parametrize("nrhs,kind", [(1, "fp64"), (8, "fp64"), (1, "fp32"), (4, "fp32"), (8, "fp32")])
def test_small_subgraphs_in_tiles(vtmlib, nrhs, kind):
    dims, block = (36 * 18 + 1, 36 * 18 + 1), (18, 18)
    A, osplit, part, s = _solver(vtmlib, dims, block, nrhs, kind)
    assert s.info().port_kernel == vtmlib.PORT_TILES
    b = inputs.rhs_uniform(A.n, nrhs, seed=5)
    copies, waves = _oracle_after(osplit, b, 0.9, 3)
    _check(s, b, 3, copies, waves[:, _line_map(part, osplit)], TOL[kind])
