"""The calls that the performance of this library is measured on.

Nearly everything a user asks of the library is ``Solver.solve``: a system is split and factored
once, and then solved for the right-hand sides that come.  Most cases are therefore whole solves,
to a tolerance, of the problem families that the repository's benchmark, models and tests use:
variable-coefficient Poisson grids in 2D and 3D and P1 finite elements, with one to 32 right-hand
sides, FP64 or FP32 sweeps, coupled or plain lines.  One case sets up the solver as well (a new
matrix every time).  The others are the entry points that stand on their own: the learned
impedance model forward and backward, and the residual without allocation.

Every solve starts from zero waves and returns the whole solution.  The tolerance is tight enough
that two correct solvers give the same solution to about 1e-10, whatever the order of their sums.
"""
import json
import math
import os

import numpy as np
import torch

import paper_0807_1949_gb300
from paper_0807_1949_gb300 import inputs, vtm

MODELS = os.path.join(os.path.dirname(os.path.abspath(paper_0807_1949_gb300.__file__)), "models")

#: family -> learned impedance model of the repository
MODEL_2D, MODEL_3D, MODEL_3D_WIDE = "z_poisson2d-256", "z_poisson3d", "z_poisson3d-wide"


def _grid(name, dims, block, sigma, nrhs, precision, model, coupled, storage="native", form="auto", what="solve",
          rtol=1e-12, check_every=20):
    d, b = list(dims) + [1] * (3 - len(dims)), list(block) + [1] * (3 - len(block))
    c = dict(what=what, nx=d[0], ny=d[1], nz=d[2], bx=b[0], by=b[1], bz=b[2], sigma=sigma, nrhs=nrhs,
             precision=precision, model=model, coupled=coupled, storage=storage, form=form, rtol=rtol,
             check_every=check_every)
    if name:
        c["name"] = name
    return c


def _fem(name, npoints, pieces, nrhs, precision, contrast, zc, rtol=1e-12):
    c = dict(what="fem", npoints=npoints, pieces=pieces, nrhs=nrhs, precision=precision, contrast=contrast, zc=zc,
             rtol=rtol, check_every=20)
    if name:
        c["name"] = name
    return c


def _mlp(name, what, n, model):
    c = dict(what=what, n=n, model=model)
    if name:
        c["name"] = name
    return c


def _resid(name, dims, nrhs):
    d = list(dims) + [1] * (3 - len(dims))
    c = dict(what="residual", nx=d[0], ny=d[1], nz=d[2], sigma=1.0, nrhs=nrhs)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest system of the benchmark and the smoke test: 32^2 in four subgraphs, FP64, plain
        # lines.  Nothing but latency: launches, checks, host work.
        _grid("solve-2d-32-fp64", (32, 32), (16, 16), 0.0, 1, "fp64", "", False, check_every=10),
        # the 2D benchmark: 256^2 in 64 subgraphs, learned impedances, coupled lines, one right-hand side
        _grid("solve-2d-256-fp32", (256, 256), (32, 32), 1.25, 1, "fp32", MODEL_2D, True, storage="fp16-auto"),
        # full precision in 3D: 64^3 in 64 subgraphs, FP64 factors and sweeps, learned impedances
        _grid("solve-3d-64-fp64", (64, 64, 64), (16, 16, 16), 1.0, 1, "fp64", MODEL_3D, True),
        # the 3D benchmark with one right-hand side: 128^3 in 512 subgraphs, FP16 responses where they pay
        _grid("solve-3d-128-fp32", (128, 128, 128), (16, 16, 16), 1.0, 1, "fp32", MODEL_3D, True, storage="fp16-auto"),
        # a few right-hand sides on a ragged grid with odd blocks
        _grid("solve-3d-ragged-r8", (101, 67, 83), (13, 11, 16), 0.8, 8, "fp32", MODEL_3D, True),
        # 32 right-hand sides on the tensor cores: few subgraphs, and the mid-size benchmark
        _grid("solve-3d-64-r32", (64, 64, 64), (16, 16, 16), 1.0, 32, "fp32", MODEL_3D_WIDE, True),
        _grid("solve-3d-128-r32", (128, 128, 128), (16, 16, 16), 1.5, 32, "fp32", MODEL_3D_WIDE, True),
        # finite elements: uneven subgraphs with thin bands, 16 right-hand sides
        _fem("solve-fem-r16", 50000, 100, 16, "fp32", 10.0, 20.0),
        # a new matrix every time (time stepping, Newton): setup and one solve
        _grid("setup-3d-64-fp32", (64, 64, 64), (16, 16, 16), 1.0, 1, "fp32", MODEL_3D, True, what="setup"),
        # the learned impedance model on all line ends of a 128^3 problem (setup), and one gradient of
        # its training on the training loop's batch
        _mlp("model-forward", "forward", 760000, MODEL_3D),
        _mlp("model-gradient", "gradient", 16384, MODEL_3D),
        # a monitor's residual of a 3D solution, eight right-hand sides, no allocation
        _resid("residual-3d-128-r8", (128, 128, 128), 8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["2d", "2d", "3d", "3d", "3d", "3d-wide", "3d-wide", "fem", "setup", "forward", "gradient",
                       "residual"])
    if kind == "2d":
        dims = (_log_int(rng, 30, 400), _log_int(rng, 30, 400))
        block = (rng.randint(13, 36), rng.randint(13, 36))
        precision = rng.choice(["fp64", "fp32", "fp32"])
        return _grid(None, dims, block, round(rng.uniform(0.0, 1.25), 3), rng.choice([1, 1, 2, 4, 8]), precision,
                     MODEL_2D, rng.random() < 0.7, storage=rng.choice(["native", "fp16-auto"]))
    if kind in ("3d", "setup"):
        precision = rng.choice(["fp64", "fp32", "fp32", "fp32"])
        nrhs = 1 if precision == "fp64" else rng.choice([1, 1, 2, 4, 8])
        top = 56 if precision == "fp64" or kind == "setup" else 110 if nrhs == 1 else 72
        dims = tuple(_log_int(rng, 24, top) for _ in range(3))
        block = tuple(rng.randint(10, 16) for _ in range(3))
        return _grid(None, dims, block, round(rng.uniform(0.5, 1.25), 3), nrhs, precision, MODEL_3D,
                     rng.random() < 0.7, storage=rng.choice(["native", "fp16-auto"]),
                     what="setup" if kind == "setup" else "solve")
    if kind == "3d-wide":
        dims = tuple(_log_int(rng, 33, 110) for _ in range(3))
        block = tuple(rng.randint(10, 16) for _ in range(3))
        return _grid(None, dims, block, round(rng.uniform(0.75, 1.5), 3), rng.choice([16, 32]), "fp32", MODEL_3D_WIDE,
                     True)
    if kind == "fem":
        n = _log_int(rng, 4000, 60000)
        return _fem(None, n, max(8, n // rng.randint(300, 550)), rng.choice([1, 8, 16, 32]), "fp32", 10.0, 20.0)
    if kind == "residual":
        return _resid(None, [_log_int(rng, 20, 128) for _ in range(3)], rng.randint(1, 8))
    if kind == "forward":
        return _mlp(None, kind, _log_int(rng, 100, 760000), rng.choice([MODEL_2D, MODEL_3D, MODEL_3D_WIDE]))
    return _mlp(None, kind, _log_int(rng, 100, 65536), rng.choice([MODEL_2D, MODEL_3D, MODEL_3D_WIDE]))


# ------------------------------------------------------------------------------------------ inputs

def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * (salt + 1) + seed)
    return g


def _grid_matrix(case, seed):
    """A matrix of ``inputs.grid_poisson``'s family (log-normal node coefficients, harmonic edge
    weights, Dirichlet boundary), made on the GPU; returns the CSR (host) and its device arrays."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    k = torch.exp(case["sigma"] * torch.randn((nz, ny, nx), generator=_gen(seed), device="cuda", dtype=torch.float64))
    n = nx * ny * nz
    idx = torch.arange(n, device="cuda").reshape(nz, ny, nx)
    diag = torch.zeros_like(k)
    below, above = [], []
    for ax, ext in ((0, nz), (1, ny), (2, nx)):
        if ext == 1:
            continue
        w = torch.zeros_like(k)       # weight of the edge to the next vertex along the axis
        a, b = k.narrow(ax, 0, ext - 1), k.narrow(ax, 1, ext - 1)
        w.narrow(ax, 0, ext - 1).copy_(2.0 * a * b / (a + b))
        step = {0: nx * ny, 1: nx, 2: 1}[ax]
        wb = torch.zeros_like(k)
        wb.narrow(ax, 1, ext - 1).copy_(w.narrow(ax, 0, ext - 1))
        diag += w + wb
        diag.narrow(ax, 0, 1).add_(k.narrow(ax, 0, 1))
        diag.narrow(ax, ext - 1, 1).add_(k.narrow(ax, ext - 1, 1))
        below.append((idx - step, -wb))
        above.insert(0, (idx + step, -w))
    entries = below + [(idx, diag)] + above
    cols = torch.stack([c for c, _ in entries], dim=-1).reshape(n, -1)
    vals = torch.stack([v for _, v in entries], dim=-1).reshape(n, -1)
    keep = vals != 0
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = torch.cumsum(keep.sum(dim=1), 0)
    col, val = cols[keep].to(torch.int32), vals[keep]
    A = inputs.CSR(n=n, rowptr=rowptr.cpu().numpy(), col=col.cpu().numpy(), val=val.cpu().numpy())
    return A, (rowptr, col, val)


def _rhs(n, nrhs, seed):
    return 2.0 * torch.rand((nrhs, n), generator=_gen(seed, 1), device="cuda", dtype=torch.float64) - 1.0


def _load_model(name):
    with open(os.path.join(MODELS, name + ".json")) as f:
        d = json.load(f)
    m = vtm.MLP(seed=0)
    m.set_params(np.asarray(d["params"], np.float32))
    return m, np.asarray(d["params"], np.float32), d.get("coupling")


def _model_impedances(part, model):
    """Line impedances of the learned model: the geometric mean of what it says for the two ends."""
    X = torch.from_numpy(part.line_features()).cuda()
    y = torch.empty(len(X), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    model.forward(X, y)
    torch.cuda.synchronize()
    lz = y.double().cpu().numpy()
    return np.exp(0.5 * (lz[0::2] + lz[1::2]))


def _solver_options(case, part):
    z, coupling = 1.0, None
    if case["what"] == "fem":
        # the split-weight rule of the finite-element tests
        d = np.exp(part.line_features()[:, 1].astype(np.float64))
        z = case["zc"] / (d[0::2] + d[1::2])
    elif case["model"]:
        model, _, rule = _load_model(case["model"])
        z = _model_impedances(part, model)
        if case["coupled"]:
            z, coupling = rule["z_scale"] * z, rule["gamma"]
    o = dict(z=z, coupling=coupling, precision=case["precision"], nrhs=case["nrhs"], check_every=case["check_every"])
    if case["what"] != "fem":
        o.update(port_storage=case["storage"], form=case["form"])
    return o


def _system(case, seed):
    """(A, partition) of a case's linear system."""
    if case["what"] == "fem":
        c = math.sqrt(case["contrast"])
        # one mesh for a number of points (its hull, and so the number of unknowns, is the mesh's own)
        fem = inputs.fem_delaunay(case["npoints"], k_lo=1.0 / c, k_hi=c, seed=case["npoints"])
        part = vtm.partition_evs(fem.A, "elements", npieces=case["pieces"], elements=dict(
            elem_nodes=fem.elem_nodes, elem_mats=fem.elem_mats, node_unknown=fem.node_unknown,
            elem_coords=fem.centroids))
        return fem.A, part
    A, _ = _grid_matrix(case, seed)
    nd = 3 if case["nz"] > 1 else 2
    part = vtm.partition_evs(A, "grid", dims=(case["nx"], case["ny"], case["nz"])[:nd],
                             block=(case["bx"], case["by"], case["bz"])[:nd])
    return A, part


def prepare(case, seed):
    what = case["what"]
    if what in ("forward", "gradient"):
        model, params, _ = _load_model(case["model"])
        X, t = _ends(case["n"], seed)
        torch.cuda.synchronize()
        return dict(what=what, model=model, X=X, t=t, y=torch.empty_like(t))
    if what == "residual":
        _, (rowptr, col, val) = _grid_matrix(case, seed)
        n = len(rowptr) - 1
        b = _rhs(n, case["nrhs"], seed)
        x = torch.randn(b.shape, generator=_gen(seed, 2), device="cuda", dtype=torch.float64)
        rel = torch.zeros(case["nrhs"], dtype=torch.float64, device="cuda")
        return dict(what=what, rowptr=rowptr, col=col, val=val, b=b, x=x, rel=rel)
    A, part = _system(case, seed)
    options = _solver_options(case, part)
    b = _rhs(A.n, case["nrhs"], seed)
    x = torch.zeros_like(b)
    torch.cuda.synchronize()
    state = dict(what=what, part=part, options=options, b=b, x=x, rtol=case["rtol"])
    if what != "setup":
        state["solver"] = vtm.Solver(part, **options)
    return state


def _ends(n, seed):
    """Features of n line ends with the spread that vtm_line_features gives on the model's family,
    and target impedances near what such ends get."""
    g = _gen(seed, 3)

    def normal():
        return torch.randn(n, generator=g, device="cuda")

    base = 1.5 + 0.8 * normal()
    copies = 2 * torch.randint(1, 3, (n,), generator=g, device="cuda").float()
    X = torch.stack([base, base - 0.7 + 0.3 * normal(), torch.log(copies), torch.ceil(copies / 2),
                     base - 0.9 + 0.3 * normal(), base - 0.7 + 0.3 * normal(), (1.2 * normal()).abs() + 0.5,
                     6.0 + 0.2 * normal()], dim=1).contiguous()
    t = (0.6 - 0.7 * (X[:, 1] + X[:, 5]) / 2 + 0.2 * normal()).contiguous()
    return X, t


# --------------------------------------------------------------------------------------------- run

def run(state):
    what = state["what"]
    if what == "forward":
        state["model"].forward(state["X"], state["y"], stream=torch.cuda.current_stream())
        return state["y"]
    if what == "gradient":
        loss = state["model"].loss_grad(state["X"], state["t"], stream=torch.cuda.current_stream())
        return {"loss": np.float32(loss), "grads": state["model"].get_grads()}
    if what == "residual":
        vtm.relative_residual_noalloc(state["rowptr"], state["col"], state["val"], state["b"], state["x"],
                                      state["rel"], stream=torch.cuda.current_stream())
        return state["rel"]
    solver = state.get("solver") or vtm.Solver(state["part"], **state["options"])
    solver.solve(state["b"], state["x"], rtol=state["rtol"], maxit=100000)
    return state["x"]


# -------------------------------------------------------------------------------------------- work

def _counts(case):
    """(unknowns, entries of A) of a case's system."""
    if case["what"] == "fem":
        return case["npoints"], 7 * case["npoints"]
    d = (case["nx"], case["ny"], case["nz"])
    n = d[0] * d[1] * d[2]
    return n, n + 2 * sum(n - n // e for e in d if e > 1)


def work(case):
    """One pass's inputs and outputs; the operations of a solve are those of its result's residual,
    the least that any method of solving spends on showing it."""
    if case["what"] in ("forward", "gradient"):
        f = 2 * (8 * 64 + 64 * 64 + 64) * case["n"]
        return {"bytes": 36 * case["n"] + 2 * 4801, "flops": f if case["what"] == "forward" else 3 * f}
    n, nnz = _counts(case)
    R = case["nrhs"]
    return {"bytes": 12 * nnz + 8 * (n + 1) + 16 * n * R, "flops": 2 * nnz * R}


# ------------------------------------------------------------------------------------------- exact

def _solution(A, b):
    """A^-1 b in 64 bits: Jacobi-preconditioned conjugate gradients, restarted on the true residual."""
    M = torch.sparse_csr_tensor(torch.from_numpy(np.asarray(A.rowptr)), torch.from_numpy(np.asarray(A.col).astype(np.int64)),
                                torch.from_numpy(np.asarray(A.val)), size=(A.n, A.n)).cuda()
    rows = torch.repeat_interleave(torch.arange(A.n, device="cuda"), M.crow_indices().diff())
    diag = torch.zeros(A.n, dtype=torch.float64, device="cuda")
    on = rows == M.col_indices()
    diag[rows[on]] = M.values()[on]
    inv = (1.0 / diag)[:, None]
    B = b.T.contiguous()
    x = torch.zeros_like(B)
    for _ in range(3):
        r = B - M @ x
        zed = inv * r
        p = zed.clone()
        rz = (r * zed).sum(0)
        first = rz.clamp_min(1e-300)
        for it in range(20000):
            q = M @ p
            alpha = rz / (p * q).sum(0).clamp_min(1e-300)
            x += alpha * p
            r -= alpha * q
            zed = inv * r
            new = (r * zed).sum(0)
            if it % 50 == 49 and bool(((new / first) < 1e-26).all()):
                break
            p = zed + (new / rz.clamp_min(1e-300)) * p
            rz = new
    return x.T.contiguous()


def _layers(params):
    w = torch.from_numpy(params).cuda().to(torch.bfloat16).double()
    return w[:512].reshape(64, 8), w[512:576], w[576:4672].reshape(64, 64), w[4672:4736], w[4736:4800], w[4800]


def exact(case, seed):
    what = case["what"]
    if what in ("forward", "gradient"):
        model, params, _ = _load_model(case["model"])
        X, t = _ends(case["n"], seed)
        W1, b1, W2, b2, W3, b3 = _layers(params)
        X = X.double()
        a1 = X @ W1.T + b1
        h1 = a1.clamp_min(0)
        a2 = h1 @ W2.T + b2
        h2 = a2.clamp_min(0)
        y = h2 @ W3 + b3
        if what == "forward":
            return y
        err = y - t.double()
        dy = 2.0 * err / case["n"]
        d2 = dy[:, None] * W3 * (a2 > 0)
        d1 = (d2 @ W2) * (a1 > 0)
        grads = torch.cat([(d1.T @ X).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0), h2.T @ dy,
                           dy.sum()[None]])
        return {"loss": (err * err).mean().cpu().numpy(), "grads": grads.cpu().numpy()}
    if what == "residual":
        A, (rowptr, col, val) = _grid_matrix(case, seed)
        b = _rhs(A.n, case["nrhs"], seed)
        x = torch.randn(b.shape, generator=_gen(seed, 2), device="cuda", dtype=torch.float64)
        M = torch.sparse_csr_tensor(rowptr, col.to(torch.int64), val, size=(A.n, A.n))
        r = b.T - M @ x.T.contiguous()
        return r.norm(dim=0) / b.norm(dim=1)
    A, _ = _system(case, seed)
    return _solution(A, _rhs(A.n, case["nrhs"], seed))
