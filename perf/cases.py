"""Performance cases of the sparse Cholesky library: the work its users have it do, at the
sizes of its own workloads, through its Python entry points.

  listed()            the cases
  draw(rng)           one more case of the same ranges
  prepare(case, seed) a user's program before the call: values, right-hand sides, handles
  run(state)          one pass
  work(case)          bytes and operations of one pass
  exact(case, seed)   what run() returns, in 64 bits

Kinds of work:
  step    new values on a known pattern: re-factorization, then the solve of the right-hand
          sides (iterative refinement for a mixed-precision factor): a Newton or implicit
          time step
  solve   new right-hand sides on a kept FP64 factor
  refine  the same on a kept mixed-precision factor
  batch   one batched re-factorization of several matrices, then a solve of each
  serve   a burst of requests of uneven size to the request server, host arrays in and out

Every value lies on a binary grid coarse enough that b = A x holds exactly in 64 bits in any
order of summation, so the x that b was made from IS the solution of A x = b.
"""
import functools
import math

import numpy as np
import torch

import paper_2202_09288_gb300 as chol
from paper_2202_09288_gb300 import inputs

X_GRID = 2.0 ** -16  # grid of the solutions' entries in [-1, 1)


def listed():
    return [
        # the smallest workload: a 2D 5-point Laplacian, where launches and latency count
        dict(name="step_lap2d_64", kind="step", family="lap2d", k=64, nrhs=1),
        # a ragged 2D grid of the size of a larger served request
        dict(name="step_lap2d_211_3rhs", kind="step", family="lap2d", k=211, nrhs=3),
        # an odd 3D grid with values, right-hand sides and solutions in host memory
        dict(name="step_lap3d_39_host", kind="step", family="lap3d", k=39, nrhs=8, host=True),
        # the reproducible (owner-ordered) assembly, with the factor read back on the device
        dict(name="step_owner_27pt_24", kind="step", family="st27x3", k=24, nrhs=1, owner=True),
        # the 3D elasticity-like workload: factor and one right-hand side
        dict(name="step_27pt_48", kind="step", family="st27x3", k=48, nrhs=1),
        # more right-hand sides on a kept factor: one, and a block of 16
        dict(name="solve_27pt_48", kind="solve", family="st27x3", k=48, nrhs=1),
        dict(name="solve_27pt_48_16rhs", kind="solve", family="st27x3", k=48, nrhs=16),
        # log-normal diffusion in mixed precision, refined to FP64 accuracy
        dict(name="step_mixed_diff_96", kind="step", family="diff3d7", k=96, nrhs=1, mixed=True),
        dict(name="refine_diff_96_16rhs", kind="refine", family="diff3d7", k=96, nrhs=16,
             mixed=True),
        # many small matrices of one pattern at once (parameter sweeps, ensembles)
        dict(name="batch_8x27pt_24", kind="batch", family="st27x3", k=24, nrhs=1, count=8),
        # the request server: 2D and 3D systems of uneven size, both precisions
        dict(name="serve_36", kind="serve", requests=36, max_n=200000),
        # the largest workload (a 33 GB factor)
        dict(name="step_27pt_80", kind="step", family="st27x3", k=80, nrhs=1),
    ]


# smallest and largest grid edge of each family
RANGES = {"lap2d": (32, 447), "lap3d": (10, 58), "diff3d7": (16, 96), "st27x3": (8, 72)}


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "solve", "refine", "batch", "serve"])
    if kind == "serve":
        return dict(kind=kind, requests=rng.randint(8, 36), max_n=_log_int(rng, 5000, 200000))
    mixed = kind == "refine" or (kind == "step" and rng.random() < 0.35)
    family = rng.choice(["diff3d7", "st27x3"] if mixed else list(RANGES))
    lo, hi = RANGES[family]
    case = dict(kind=kind, family=family, nrhs=_log_int(rng, 1, 32))
    if kind == "batch":
        case["count"] = rng.randint(2, 12)
        hi = max(lo + 1, hi // 3)
    if mixed:
        case["mixed"] = True
    elif kind == "step" and rng.random() < 0.2:
        case["owner"] = True
        hi = max(lo + 1, hi // 3)
    elif kind == "step" and rng.random() < 0.2:
        case["host"] = True
    case["k"] = _log_int(rng, lo, hi)
    return case


# ---- patterns and contexts: what a program makes once and keeps -----------------------------
@functools.lru_cache(maxsize=4)
def _context(owner):
    return chol.Context(assembly=chol.CHOL_ASSEMBLY_OWNER if owner else chol.CHOL_ASSEMBLY_ATOMIC)


@functools.lru_cache(maxsize=24)
def _pattern(family, k):
    """Matrix pattern (with the generator's own values) and ordering of a workload."""
    return inputs.workload(f"{family}_{k}")


@functools.lru_cache(maxsize=16)
def _symbolic(family, k, owner):
    A, perm = _pattern(family, k)
    return chol.Symbolic(_context(owner), A, perm)


@functools.lru_cache(maxsize=2)
def _indices(family, k):
    """Row and column of every stored entry, and the positions of the diagonal (GPU)."""
    A, _ = _pattern(family, k)
    colptr = torch.from_numpy(A.colptr).cuda()
    rows = torch.from_numpy(A.rowind).cuda().long()
    cols = torch.repeat_interleave(torch.arange(A.n, device="cuda"), colptr.diff())
    return rows, cols, colptr[:-1]


# ---- values and right-hand sides, from the seed alone ---------------------------------------
def _grid(t, step):
    return torch.round(t / step) * step


def _values(family, k, gen):
    """Values of the stored lower triangle (GPU, float64): the workload's family with new
    random coefficients."""
    A, _ = _pattern(family, k)
    rows, cols, diag = _indices(family, k)
    if family in ("lap2d", "lap3d"):  # A + sigma diag(A), sigma in (0, 1]
        vals = torch.from_numpy(A.vals).cuda()
        sigma = (1 + int(torch.randint(1024, (1,), generator=gen, device="cuda"))) / 1024
        vals[diag] *= 1 + sigma
        return vals
    if family == "diff3d7":  # log-normal cells, harmonic faces, Dirichlet boundary
        z = torch.randn((k, k, k), generator=gen, device="cuda", dtype=torch.float64)
        kap = _grid(torch.exp(1.5 * z), 2.0 ** -20)
        d = torch.zeros_like(kap)
        faces = []
        for ax in (2, 1, 0):  # x runs fastest
            lo, hi = kap.narrow(ax, 0, k - 1), kap.narrow(ax, 1, k - 1)
            f = _grid(2 * lo * hi / (lo + hi), 2.0 ** -20).clamp_(min=2.0 ** -20)
            d.narrow(ax, 0, k - 1).add_(f)
            d.narrow(ax, 1, k - 1).add_(f)
            d.select(ax, 0).add_(kap.select(ax, 0))
            d.select(ax, k - 1).add_(kap.select(ax, k - 1))
            full = torch.zeros_like(kap)
            full.narrow(ax, 0, k - 1).copy_(-f)
            faces.append(full.reshape(-1))
        slots = torch.stack([d.reshape(-1)] + faces, dim=1)
        return slots[slots != 0]
    # st27x3: random couplings, strictly diagonally dominant
    grid = 2.0 ** -20
    vals = _grid(torch.rand(A.nnz_lower, generator=gen, device="cuda", dtype=torch.float64)
                 * 2 - 1, grid)
    vals[diag] = 0
    size = vals.abs()
    dom = torch.zeros(A.n, device="cuda", dtype=torch.float64)
    dom.index_add_(0, rows, size).index_add_(0, cols, size)
    extra = torch.rand(A.n, generator=gen, device="cuda", dtype=torch.float64)
    vals[diag] = dom + 1 + _grid(extra, grid)
    return vals


def _solution(n, nrhs, gen):
    """nrhs solutions, entries uniform in [-1, 1) on the grid; row c is solution c."""
    i = torch.randint(-(1 << 16), 1 << 16, (nrhs, n), generator=gen, device="cuda")
    return i.double() * X_GRID


def _apply(family, k, vals, x):
    """A x for every row of x, A given by its lower triangle."""
    rows, cols, diag = _indices(family, k)
    off = vals.clone()
    off[diag] = 0
    out = torch.zeros_like(x)
    for c in range(x.shape[0]):
        out[c].index_add_(0, rows, vals * x[c][cols]).index_add_(0, cols, off * x[c][rows])
    return out


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _system(family, k, nrhs, seed):
    gen = _generator(seed)
    x = _solution(_pattern(family, k)[0].n, nrhs, gen)
    vals = _values(family, k, gen)
    return vals, _apply(family, k, vals, x), x


def _requests(case):
    """(family, k, nrhs) of every request: 2D 5-point or 3D 7-point, n log-uniform from 1,000
    to max_n, 1-8 right-hand sides.  The burst's patterns belong to the case, its numbers to
    the seed."""
    rng = np.random.RandomState(7)
    out = []
    for _ in range(case["requests"]):
        n = math.exp(rng.uniform(math.log(1000), math.log(case["max_n"])))
        fam = "lap2d" if rng.rand() < 0.5 else "lap3d"
        out.append((fam, round(n ** (0.5 if fam == "lap2d" else 1 / 3)), int(rng.randint(1, 9))))
    return out


# ---- the cases ------------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        reqs = []
        for i, (fam, k, nrhs) in enumerate(_requests(case)):
            A, perm = _pattern(fam, k)
            vals, b, _ = _system(fam, k, nrhs, seed * 1009 + i)
            M = inputs.SpdMatrix(A.n, A.colptr, A.rowind, vals.cpu().numpy(), A.grid, A.dofs)
            reqs.append((M, perm, np.asfortranarray(b.cpu().numpy().T),
                         chol.CHOL_MIXED if i % 2 else chol.CHOL_FP64))
        return dict(kind=kind, server=chol.Server(), requests=reqs)
    family, k, nrhs = case["family"], case["k"], case["nrhs"]
    owner, mixed = bool(case.get("owner")), bool(case.get("mixed"))
    ctx, sym = _context(owner), _symbolic(family, k, owner)
    precision = chol.CHOL_MIXED if mixed else chol.CHOL_FP64
    systems = [_system(family, k, nrhs, seed * 1013 + i)[:2] for i in range(case.get("count", 1))]
    torch.cuda.synchronize()  # the library works on a stream of its own
    factors = [chol.Factor(ctx, sym, vals, precision) for vals, _ in systems]
    vals, b = systems[0]
    state = dict(kind=kind, factors=factors, mixed=mixed, vals=[v for v, _ in systems],
                 b=[b for _, b in systems], x=[torch.empty_like(b) for _, b in systems])
    if kind == "batch":
        state["batch"] = chol.Batch(ctx, factors)
    if case.get("host"):
        state["vals"] = [vals.cpu().numpy()]
        state["b"] = [np.asfortranarray(b.cpu().numpy().T)]
        state["x"] = [np.zeros_like(state["b"][0], order="F")]
    if owner:
        state["panels"] = torch.empty(sym.info["l_storage"], dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    return state


def run(state):
    kind = state["kind"]
    if kind == "serve":
        server = state["server"]
        tickets = [server.submit(A, perm, b, precision=p) for A, perm, b, p in state["requests"]]
        return [server.wait(t)[0] for t in tickets]
    factors, b, x = state["factors"], state["b"], state["x"]
    if kind == "batch":
        state["batch"].factorize(state["vals"])
        for f, bi, xi in zip(factors, b, x):
            f.solve(bi, xi)
        return x
    f = factors[0]
    if kind == "step":
        f.refactor(state["vals"][0])
    if state["mixed"]:
        f.refine(b[0], x[0])
    else:
        f.solve(b[0], x[0])
    if "panels" in state:
        return {"x": x[0], "factor": chol.chol_factor_panels(
            f.ctx.handle, f.handle, 0, f.sym.info["nsuper"], state["panels"])}
    return x[0]


def work(case):
    """A step reads A's values and b and writes the factor and x; a solve reads the factor and
    b and writes x; refinement also reads A's values."""
    def one(family, k, nrhs, mixed, factor, solve_reads, refine):
        info = _info(family, k, case["kind"] == "serve")
        n, nnz = info["n"], info["nnz_a"]
        factor_bytes = (4 if mixed else 8) * info["nnz_l"]
        by = 16.0 * n * nrhs
        fl = 4.0 * info["nnz_l"] * nrhs
        if factor:
            by += 8.0 * nnz + factor_bytes
            fl += info["flops"]
        if solve_reads:
            by += factor_bytes
        if refine and not factor:
            by += 8.0 * nnz
        return by, fl

    if case["kind"] == "serve":
        parts = [one(f, k, r, i % 2 == 1, True, False, True)
                 for i, (f, k, r) in enumerate(_requests(case))]
    else:
        kept = case["kind"] in ("solve", "refine")
        parts = [one(case["family"], case["k"], case["nrhs"], bool(case.get("mixed")), not kept,
                     kept, bool(case.get("mixed")))] * case.get("count", 1)
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


@functools.lru_cache(maxsize=64)
def _info(family, k, served):
    if not served:
        return _symbolic(family, k, False).info
    A, perm = _pattern(family, k)
    return chol.Symbolic(None, A, perm).info


def exact(case, seed):
    """The solutions that the right-hand sides were made from (see the module's text)."""
    if case["kind"] == "serve":
        return [_solution(_pattern(f, k)[0].n, r, _generator(seed * 1009 + i)).cpu().numpy().T
                for i, (f, k, r) in enumerate(_requests(case))]
    n = _pattern(case["family"], case["k"])[0].n
    xs = [_solution(n, case["nrhs"], _generator(seed * 1013 + i))
          for i in range(case.get("count", 1))]
    if case["kind"] == "batch":
        return xs
    if case.get("host"):
        return xs[0].cpu().numpy().T
    if case.get("owner"):
        return {"x": xs[0], "factor": None}
    return xs[0]
