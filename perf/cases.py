"""The calls that users of this library make most, for timing and comparing its results.

A simulator keeps one mesh for a whole run: its sparsity pattern and the
symbolic analysis of it (``opm.Analysis``) are made once, and so are the
solver handles.  What changes from call to call is the matrix values (one
Newton step's Jacobian), the right-hand side and the vectors.  So a case's
mesh depends on the case alone and is kept for the process; ``prepare`` draws
the values, x_true and b = A x_true from the seed, on the GPU, and makes the
handles of that state from the kept analysis.

Meshes: ``full`` (all cells of a box active), ``faulted`` (n^3 cells, 5% of
them inactive, 1% fault connections) and ``region`` (the connected region of
44,431 cells of a 46 x 112 x 22 grid).
"""
import functools
import math

import numpy as np
import torch

from paper_2309_11488_gb300 import opm, synth

DEV = "cuda"


def listed():
    return [
        # the smallest model: one Newton step's linear system (new values: refactor, solve), Dune's default tolerance
        {"name": "step_500_fp64", "kind": "step", "mesh": "full", "nx": 10, "ny": 10, "nz": 5,
         "precision": "fp64", "rtol": 1e-2},
        # a field-sized model (44,431 cells): a Newton step at the default tolerance
        {"name": "step_44k_fp64", "kind": "step", "mesh": "region", "nx": 46, "ny": 112, "nz": 22,
         "precision": "fp64", "rtol": 1e-2},
        # the same model solved tightly on the factors it has: many Krylov iterations per factorisation
        {"name": "solve_44k_fp64_tight", "kind": "solve", "mesh": "region", "nx": 46, "ny": 112, "nz": 22,
         "precision": "fp64", "rtol": 1e-6},
        # one request of the serving workload: refactor + solve, FP32 factors
        {"name": "step_22k_fp32", "kind": "step", "mesh": "full", "nx": 37, "ny": 31, "nz": 19,
         "precision": "fp32", "rtol": 1e-2},
        # the largest model (949,871 cells), both factor precisions
        {"name": "step_950k_fp64", "kind": "step", "mesh": "faulted", "nx": 100, "ny": 100, "nz": 100,
         "precision": "fp64", "rtol": 1e-3},
        {"name": "step_950k_fp32", "kind": "step", "mesh": "faulted", "nx": 100, "ny": 100, "nz": 100,
         "precision": "fp32", "rtol": 1e-3},
        # an ensemble: 256 models of 500 to 20,000 cells refactored and solved in one launch
        {"name": "batch_256_fp32", "kind": "batch", "nsys": 256, "precision": "fp32", "rtol": 1e-2},
        # block-Jacobi ILU0 over 8 partitions with standard wells kept separate
        {"name": "step_61k_jacobi_wells", "kind": "step", "mesh": "faulted", "nx": 40, "ny": 40, "nz": 40,
         "precision": "fp64", "rtol": 1e-2, "parts": 8, "wells": 24},
        # the other Krylov solver, restarted GMRES(30)
        {"name": "gmres_249k_fp64", "kind": "gmres", "mesh": "faulted", "nx": 64, "ny": 64, "nz": 64,
         "precision": "fp64", "rtol": 1e-3},
        # the operators alone, for a caller's own Krylov method
        {"name": "spmv_249k", "kind": "spmv", "mesh": "faulted", "nx": 64, "ny": 64, "nz": 64, "precision": "fp64"},
        {"name": "ilu_apply_44k_fp64", "kind": "apply", "mesh": "region", "nx": 46, "ny": 112, "nz": 22,
         "precision": "fp64"},
        # a convergence check on the caller's own arrays: r = b - A x and its norm
        {"name": "residual_249k", "kind": "residual", "mesh": "faulted", "nx": 64, "ny": 64, "nz": 64},
    ]


def _loguniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _mesh_of(rng, cells):
    """A mesh of about that many cells; odd and uneven sides."""
    u = rng.random()
    if u < 0.15 and 20_000 <= cells:
        return {"mesh": "region", "nx": 46, "ny": 112, "nz": 22}
    if u < 0.6:
        n = max(8, min(99, round(cells ** (1 / 3))))
        return {"mesh": "faulted", "nx": n, "ny": n, "nz": n}
    nz = max(2, round(cells ** (1 / 3) * rng.uniform(0.3, 1.0)))
    nx = max(2, round(math.sqrt(cells / nz) * rng.uniform(0.7, 1.4)))
    ny = max(2, round(cells / nz / nx))
    return {"mesh": "full", "nx": nx, "ny": ny, "nz": nz}


def draw(rng):
    kind = rng.choices(["step", "solve", "spmv", "apply", "gmres", "batch", "residual"], [45, 12, 9, 9, 9, 8, 8])[0]
    precision = rng.choice(["fp64", "fp32"])
    if kind == "batch":
        return {"kind": "batch", "nsys": round(_loguniform(rng, 4, 200)), "precision": precision, "rtol": 1e-2}
    cells = _loguniform(rng, 500, 900_000 if kind in ("step", "spmv", "residual") else 250_000)
    case = {"kind": kind, **_mesh_of(rng, cells)}
    if kind == "residual":
        return case
    case["precision"] = "fp64" if kind in ("spmv", "gmres") else precision
    if kind in ("step", "solve", "gmres"):
        case["rtol"] = rng.choice([1e-2, 1e-2, 1e-3, 1e-6] if kind != "gmres" else [1e-2, 1e-3])
    if kind == "step" and case["mesh"] != "region" and case["nx"] >= 12 and rng.random() < 0.2:
        case["parts"] = rng.choice([2, 3, 8])
        case["wells"] = rng.randint(2, 40)
    return case


# ------------------------------------------------------------------ meshes


@functools.lru_cache(maxsize=4)
def _system(mesh, nx, ny, nz):
    if mesh == "region":
        return synth.config2()
    if mesh == "faulted":
        return synth.config3(nx)
    logk = np.random.default_rng([nx, ny, nz]).normal(size=(nz, ny, nx))
    return synth.grid_system(nx, ny, nz, logk, seed=synth.SEED_BASE + nx + 100 * ny + 10_000 * nz)


@functools.lru_cache(maxsize=4)
def _ensemble(nsys):
    return synth.config4(nsys)


class _Mesh:
    """A pattern, the base values on it (GPU), its analysis, and rows as index lists."""

    def __init__(self, system, parts=0, nwells=0):
        self.nb, self.nnzb = system.nb, system.nnzb
        self.rowptr, self.colidx = system.rowptr, system.colidx
        self.base = torch.from_numpy(system.vals).to(DEV)
        self.rp = torch.from_numpy(system.rowptr).to(DEV)
        self.ci = torch.from_numpy(system.colidx).to(DEV)
        self.maxlen = int(np.diff(system.rowptr).max())
        part = np.ascontiguousarray(synth.partition_grid(system, parts), dtype=np.int32) if parts else None
        rows = np.repeat(np.arange(system.nb), np.diff(system.rowptr))
        self.diag = torch.from_numpy(np.flatnonzero(rows == system.colidx)).to(DEV)
        self.base_sums = self.abs_sums(self.base)
        self.analysis = opm.Analysis(system.nb, system.rowptr, system.colidx, part=part)
        self.wells = synth.wells(system, nwells, 6) if nwells else None

    def abs_sums(self, vals):
        """Per row of the matrix, the sum of its absolute entries outside the diagonal block [nb, 3]."""
        a = vals.abs().view(-1, 3, 3).sum(2)
        a[self.diag] = 0.0
        total = torch.zeros(self.nb, 3, dtype=torch.float64, device=DEV)
        start, end = self.rp[:-1].long(), self.rp[1:].long()
        for k in range(self.maxlen):
            has = (start + k < end).nonzero().view(-1)
            total[has] += a[start[has] + k]
        return total

    def times(self, vals, x):
        """A x, plain torch, 64 bits, the same bits every time."""
        x3 = x.view(-1, 3)
        y = torch.zeros_like(x3)
        start, end = self.rp[:-1].long(), self.rp[1:].long()
        blocks = vals.view(-1, 3, 3)
        for k in range(self.maxlen):
            has = (start + k < end).nonzero().view(-1)
            m = start[has] + k
            y[has] += (blocks[m] * x3[self.ci[m].long()].unsqueeze(1)).sum(2)
        return y.view(-1)


@functools.lru_cache(maxsize=4)
def _mesh(mesh, nx, ny, nz, parts, nwells):
    return _Mesh(_system(mesh, nx, ny, nz), parts, nwells)


@functools.lru_cache(maxsize=2)
def _meshes(nsys):
    return [_Mesh(s) for s in _ensemble(nsys)]


def _mesh_for(case):
    return _mesh(case["mesh"], case["nx"], case["ny"], case["nz"], case.get("parts", 0), case.get("wells", 0))


def _draws(mesh, gen):
    """One Newton step's values and x_true in U(-1, 1).  Every coupling block is scaled by U(0.9, 1.1); the diagonal
    block keeps its accumulation term and carries the new couplings' sums, as a flow Jacobian's does."""
    f = torch.rand(mesh.nnzb, 1, generator=gen, device=DEV, dtype=torch.float64)
    f[mesh.diag] = 0.5
    vals = mesh.base * (0.9 + 0.2 * f)
    vals[mesh.diag[:, None], torch.tensor([[0, 4, 8]], device=DEV)] += mesh.abs_sums(vals) - mesh.base_sums
    x_true = 2 * torch.rand(3 * mesh.nb, generator=gen, device=DEV, dtype=torch.float64) - 1
    return vals, x_true


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


# ------------------------------------------------------------------ the cases


def prepare(case, seed):
    gen = _gen(seed)
    kind = case["kind"]
    if kind == "batch":
        meshes = _meshes(case["nsys"])
        ends = np.cumsum([0] + [3 * m.nb for m in meshes])
        x = torch.empty(int(ends[-1]), dtype=torch.float64, device=DEV)
        vals, bs = [], []
        for m in meshes:
            v, x_true = _draws(m, gen)
            vals.append(v)
            bs.append(m.times(v, x_true))
        solvers = [opm.Solver.from_analysis(m.analysis, v, precision=case["precision"]) for m, v in zip(meshes, vals)]
        return {"kind": kind, "rtol": case["rtol"], "solvers": solvers, "batch": opm.Batch([s.h for s in solvers]),
                "vals": vals, "b": bs, "x": x, "xs": [x[a:e] for a, e in zip(ends[:-1], ends[1:])]}
    m = _mesh_for(case)
    vals, x_true = _draws(m, gen)
    state = {"kind": kind, "mesh": m, "vals": vals, "rtol": case.get("rtol")}
    if kind == "residual":
        # an iterate as a solver leaves it: close to the solution
        state["b"] = m.times(vals, x_true)
        state["x"] = x_true + 1e-3 * (torch.rand(3 * m.nb, generator=gen, device=DEV, dtype=torch.float64) - 0.5)
        state["r"] = torch.empty_like(x_true)
        state["norms"] = torch.empty(2, dtype=torch.float64, device=DEV)
        return state
    state["solver"] = opm.Solver.from_analysis(m.analysis, vals, precision=case["precision"])
    if m.wells is not None:
        state["solver"].set_wells(m.wells)
    state["b"] = x_true if kind in ("spmv", "apply") else m.times(vals, x_true)
    state["x"] = torch.empty_like(x_true)
    return state


def run(state):
    kind = state["kind"]
    if kind == "step":
        sv = state["solver"]
        sv.launch(state["vals"], state["b"], state["x"], rtol=state["rtol"])
        status, iters, relres = sv.wait()
        return {"x": state["x"], "status": status, "iters": iters, "relres": relres}
    if kind == "solve":
        x, status, iters, relres = state["solver"].solve(state["b"], state["x"], rtol=state["rtol"])
        return {"x": x, "status": status, "iters": iters, "relres": relres}
    if kind == "gmres":
        x, status, iters, relres = state["solver"].gmres(state["b"], state["x"], rtol=state["rtol"])
        return {"x": x, "status": status, "iters": iters, "relres": relres}
    if kind == "batch":
        state["batch"].launch(state["vals"], state["b"], state["xs"], rtol=state["rtol"])
        status, each, iters, relres = state["batch"].wait()
        return {"x": state["x"], "status": np.array([status] + each), "iters": np.array(iters),
                "relres": np.array(relres)}
    if kind == "spmv":
        return {"y": state["solver"].spmv(state["b"], state["x"])}
    if kind == "apply":
        return {"z": state["solver"].ilu_apply(state["b"], state["x"])}
    m = state["mesh"]
    status = opm.opm_bsr_residual_noalloc(m.nb, m.rp, m.ci, state["vals"], state["x"], state["b"], state["r"],
                                          state["norms"])
    return {"r": state["r"], "norms": state["norms"], "status": status}


def work(case):
    """Bytes: values, indices and vectors of the call once.  FP64 operations: 18 per block of a product or a
    triangular solve, about 50 per lower block of a factorisation, for the iterations such a tolerance takes."""
    if case["kind"] == "batch":
        sizes = [(s.nb, s.nnzb) for s in _ensemble(case["nsys"])]
    else:
        s = _system(case["mesh"], case["nx"], case["ny"], case["nz"])
        sizes = [(s.nb, s.nnzb)]
    n, nnzb = sum(a for a, _ in sizes), sum(b for _, b in sizes)
    its = {None: 0, 1e-2: 2, 1e-3: 5, 1e-6: 25}[case.get("rtol")]
    factors = 4.0 if case.get("precision") == "fp32" else 8.0
    pattern = 4.0 * nnzb + 4.0 * n
    kind = case["kind"]
    if kind in ("step", "batch"):
        return {"bytes": 72.0 * nnzb + pattern + 48.0 * n, "flops": 50.0 * nnzb + its * (72.0 * nnzb + 120.0 * n)}
    if kind == "apply":
        return {"bytes": 9.0 * factors * nnzb + pattern + 48.0 * n, "flops": 18.0 * nnzb}
    if kind in ("spmv", "residual"):
        return {"bytes": 72.0 * nnzb + pattern + (48.0 if kind == "spmv" else 72.0) * n, "flops": 18.0 * nnzb}
    return {"bytes": (72.0 + 9.0 * factors) * nnzb + pattern + 48.0 * n,
            "flops": its * (72.0 * nnzb + 120.0 * n)}


def exact(case, seed):
    """Products and residuals as plain torch gives them in 64 bits; a tight solve's x is the x_true that b was
    made from.  What a loose solve returns after its few iterations has no such value."""
    kind = case["kind"]
    if kind not in ("spmv", "residual") and not (kind in ("step", "solve") and case["rtol"] <= 1e-6):
        return None
    if case.get("wells"):
        return None
    m = _mesh_for(case)
    gen = _gen(seed)
    vals, x_true = _draws(m, gen)
    if kind == "spmv":
        return {"y": m.times(vals, x_true)}
    if kind in ("step", "solve"):
        return {"x": x_true, "status": None, "iters": None, "relres": None}
    b = m.times(vals, x_true)
    x = x_true + 1e-3 * (torch.rand(3 * m.nb, generator=gen, device=DEV, dtype=torch.float64) - 0.5)
    r = b - m.times(vals, x)
    return {"r": r, "norms": torch.stack([r.norm(), b.norm()]), "status": None}
