"""Performance cases of the solver: what its users call, over the sizes they call it at.

A case is one of three programs:

* ``factor_solve``: a matrix whose analysis is in hand is factored and its
  system solved (the headline use: coefficients in, solution out);
* ``solve``: the factorization is in hand and new right-hand sides are
  solved (a time-stepping program, or the serving runtime's batches);
* ``apply``: one application of the factorization as a preconditioner inside
  the caller's own Krylov method.

Systems are solved to a relative residual of 1e-12, where the solution is
determined to better than nine digits whatever route the preconditioner took
to it; ``exact`` gives it in float64 by other means (fast sine transforms for
the constant-coefficient symmetric matrices, long plain Krylov iterations for
the others).  Sizes, cluster sizes and tolerances eps are those of the
repository's workloads (``inputs.workload`` and ``inputs.SERVING_FAMILIES``)
and odd sizes around them.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1712_07297_gb300 import hsolve
from paper_1712_07297_gb300 import inputs

TOL = 1e-12


def listed():
    return [
        # the smallest call: one preconditioner application inside a user's
        # own Krylov loop, all launches and latency
        dict(name="apply_2d64_f64", do="apply", family="poisson", shape="64x64", leaf=64,
             eps=1e-3, precision="fp64", krylov="pcg", top_size=0, nrhs=1),
        # the small workload: 4,096 unknowns in a few colour classes
        dict(name="fs_2d64", do="factor_solve", family="poisson", shape="64x64", leaf=64,
             eps=1e-3, precision="mixed_fp32", krylov="pcg", top_size=0, nrhs=1),
        # ragged: a grid of odd sides, clusters of unequal sizes, both eps and
        # precision on the accurate side
        dict(name="fs_3d_ragged_f64", do="factor_solve", family="poisson", shape="29x37x23",
             leaf=128, eps=1e-4, precision="fp64", krylov="pcg", top_size=0, nrhs=3),
        # the ordinary call: 262,144 unknowns, one right-hand side
        dict(name="fs_3d64", do="factor_solve", family="poisson", shape="64x64x64", leaf=128,
             eps=1e-2, precision="mixed_fp32", krylov="pcg", top_size=8192, nrhs=1),
        # the same with the tensor-core Schur products
        dict(name="fs_3d64_tf32", do="factor_solve", family="poisson", shape="64x64x64",
             leaf=128, eps=1e-2, precision="mixed_tf32", krylov="pcg", top_size=8192, nrhs=1),
        # the plain float64 path
        dict(name="fs_3d64_f64", do="factor_solve", family="poisson", shape="64x64x64",
             leaf=128, eps=1e-2, precision="fp64", krylov="pcg", top_size=8192, nrhs=1),
        # nonsymmetric: LU blocks, two-sided compression, GMRES
        dict(name="fs_convdiff64", do="factor_solve", family="convdiff", shape="64x64x64",
             leaf=128, eps=1e-2, precision="mixed_fp32", krylov="gmres", top_size=4096, nrhs=1),
        # variable coefficients 10^U(-3, 3), diagonally equilibrated: many
        # iterations
        dict(name="fs_vcdiff96", do="factor_solve", family="vcdiff", decades=3.0,
             shape="96x96x96", leaf=128, eps=1e-2, precision="mixed_fp32", krylov="pcg",
             top_size=8192, nrhs=1),
        # the largest: several right-hand sides by block GMRES, as the
        # headline benchmark does
        dict(name="fs_3d96_rhs8", do="factor_solve", family="poisson", shape="96x96x96",
             leaf=128, eps=1e-2, precision="mixed_fp32", krylov="gmres", top_size=8192, nrhs=8),
        # a factorization reused for one new right-hand side
        dict(name="solve_3d64", do="solve", family="poisson", shape="64x64x64", leaf=128,
             eps=1e-2, precision="mixed_fp32", krylov="pcg", top_size=8192, nrhs=1),
        # one batch of a serving stream, three-dimensional family
        dict(name="solve_3d64_rhs32", do="solve", family="poisson", shape="64x64x64", leaf=128,
             eps=1e-2, precision="mixed_fp32", krylov="pcg", top_size=8192, nrhs=32),
        # a large batch of a serving stream (its mean batch holds about 124
        # right-hand sides), two-dimensional family
        dict(name="solve_2d512_rhs124", do="solve", family="poisson", shape="512x512", leaf=64,
             eps=1e-2, precision="mixed_fp32", krylov="pcg", top_size=0, nrhs=124),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_shape(rng, dim, lo, hi):
    """Sides with a product of about n, n log-uniform in [lo, hi], up to 1.6:1."""
    side = _log_uniform(rng, lo, hi) ** (1.0 / dim)
    return "x".join(str(max(6, round(side * rng.uniform(0.8, 1.25)))) for _ in range(dim))


def draw(rng):
    do = rng.choice(["factor_solve", "factor_solve", "factor_solve", "solve", "solve", "apply"])
    c = dict(do=do, family="poisson", krylov="pcg", top_size=0)
    if do == "apply":
        dim = rng.choice([2, 3])
        c.update(shape=_draw_shape(rng, dim, 1000, 8000), leaf=rng.randint(48, 96), eps=1e-3,
                 precision="fp64", nrhs=_log_uniform(rng, 1, 16))
        return c
    dim = rng.choice([2, 3, 3])
    c["leaf"] = rng.randint(48, 80) if dim == 2 else rng.randint(96, 144)
    c["eps"] = rng.choice([1e-2, 1e-2, 1e-3, 1e-4])
    if do == "solve":
        c.update(precision=rng.choice(["mixed_fp32", "mixed_fp32", "fp64"]),
                 nrhs=_log_uniform(rng, 1, 128))
        hi = 30000 if c["precision"] == "fp64" or c["eps"] < 1e-2 else 150000
        c["shape"] = _draw_shape(rng, dim, 2000, hi)
        return c
    c.update(family=rng.choice(["poisson", "poisson", "vcdiff", "convdiff"]),
             precision=rng.choice(["mixed_fp32", "mixed_fp32", "mixed_3xtf32", "fp64"]),
             nrhs=_log_uniform(rng, 1, 16))
    if c["family"] == "vcdiff":
        # a milder field: truncation at an arbitrary size and eps may cost a
        # wider one its definiteness
        dim = 3
        c.update(decades=1.0, leaf=rng.randint(96, 144), eps=min(c["eps"], 1e-3))
    hi = 30000 if c["precision"] == "fp64" or c["eps"] < 1e-2 or c["family"] == "convdiff" \
        else 150000
    c["shape"] = _draw_shape(rng, dim, 2000, hi)
    if c["family"] == "convdiff":
        c["krylov"] = "gmres"
    elif rng.random() < 0.3:
        c["krylov"] = "gmres"
    if rng.random() < 0.5:
        c["top_size"] = rng.choice([1024, 2048, 4096])
    return c


# ---------------------------------------------------------------------------
# What a user's program has in hand
# ---------------------------------------------------------------------------
# The coefficient field of the variable-coefficient matrices belongs to the
# case (the workload's own seed); a pass's seed makes its right-hand sides.
FIELD_SEED = 2002


def _shape(case):
    return tuple(int(x) for x in case["shape"].split("x"))


@functools.lru_cache(maxsize=2)
def _matrix(family, shape, decades):
    if family == "poisson":
        return inputs.poisson(shape)
    if family == "convdiff":
        return inputs.convection_diffusion(shape, 10.0)
    if family == "vcdiff":
        return inputs.vc_diffusion(shape, seed=FIELD_SEED, log10_range=decades)
    raise ValueError(family)


def _rhs(n, nrhs, seed):
    """Entries uniform in [-1, 1]: an (nrhs, n) tensor, column-major n x nrhs."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.rand((nrhs, n), generator=g, dtype=torch.float64, device="cuda") * 2.0 - 1.0


def prepare(case, seed):
    p = _matrix(case["family"], _shape(case), case.get("decades"))
    solver = hsolve.Solver.from_problem(
        p, leaf_size=case["leaf"], symmetric=1 if p.spd else 0, top_size=case["top_size"],
        equilibrate=1 if case["family"] == "vcdiff" else 0)
    if case["do"] != "factor_solve":
        solver.factor(case["eps"], case["precision"])
    return dict(case=case, solver=solver, b=_rhs(p.n, case["nrhs"], seed))


def run(state):
    case, solver = state["case"], state["solver"]
    if case["do"] == "apply":
        return solver.apply(state["b"])
    if case["do"] == "factor_solve":
        solver.factor(case["eps"], case["precision"])
    x, _ = solver.solve(state["b"], krylov=case["krylov"], tol=TOL, maxit=1000)
    return x


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Bytes: the right-hand sides in, the solutions out and, where the pass
    factors or multiplies by it, the matrix (CSR).  Flops: eliminating every
    leaf cluster of m unknowns against its interface of 2 dim faces of
    m^((dim-1)/dim) unknowns (twice for a nonsymmetric matrix), and one
    product with the matrix and one with the leaves' inverse factors per
    right-hand side."""
    shape = _shape(case)
    dim, n, m = len(shape), int(np.prod(shape)), case["leaf"]
    nnz = (2 * dim + 1) * n - 2 * sum(n // s for s in shape)
    vectors = 2 * 8 * n * case["nrhs"]
    per_rhs = 2 * n * m * case["nrhs"]
    if case["do"] == "apply":
        return {"bytes": vectors, "flops": 2 * per_rhs}
    matrix = 12 * nnz + 8 * (n + 1)
    flops = 2 * nnz * case["nrhs"] + 2 * per_rhs
    if case["do"] == "factor_solve":
        face = 2 * dim * m ** ((dim - 1) / dim)
        leaf = m ** 3 / 3 + m ** 2 * face + m * face ** 2
        flops += n / m * leaf * (2 if case["family"] == "convdiff" else 1)
    return {"bytes": matrix + vectors, "flops": flops}


# ---------------------------------------------------------------------------
# The same in float64 by other means
# ---------------------------------------------------------------------------
def _sine_solve(shape, b):
    """A^{-1} b for the unscaled Dirichlet Laplacian: the sine basis of every
    axis diagonalizes it."""
    dim = len(shape)
    x = b.reshape((b.shape[0],) + shape[::-1])  # x fastest
    lam = torch.zeros(shape[::-1], dtype=torch.float64, device=b.device)
    bases = []
    for d, s in enumerate(shape):
        k = torch.arange(1, s + 1, dtype=torch.float64, device=b.device)
        bases.append(torch.sin(torch.outer(k, k) * (math.pi / (s + 1))) *
                     math.sqrt(2.0 / (s + 1)))
        view = [1] * dim
        view[dim - 1 - d] = s
        lam = lam + (4.0 * torch.sin(k * (math.pi / (2 * (s + 1)))) ** 2).reshape(view)

    def transform(v):
        for d in range(dim):
            v = torch.movedim(torch.tensordot(v, bases[d], dims=([dim - d], [0])), -1, dim - d)
        return v

    return transform(transform(x) / lam).reshape(b.shape)


def _csr(p, device):
    return torch.sparse_csr_tensor(torch.from_numpy(p.rowptr).to(device),
                                   torch.from_numpy(p.col.astype(np.int64)).to(device),
                                   torch.from_numpy(p.val).to(device), size=(p.n, p.n))


def _refined(a, b, scale, solve_once):
    """x with A x = b by repeated correction; b is (nrhs, n)."""
    bt = b.T.contiguous()
    x = torch.zeros_like(bt)
    best, keep = math.inf, x
    for _ in range(6):
        r = bt - a @ x
        size = float((r.norm(dim=0) / bt.norm(dim=0)).max())
        if size < best:
            best, keep = size, x
        if not size > 1e-15 or size > 0.5 * best and best < size:
            break
        x = x + solve_once(r, scale)
    return keep.T.contiguous()


def _cg(a, r, dinv, tol=1e-9, maxit=8000):
    """Conjugate gradients preconditioned with the diagonal, column by column."""
    x = torch.zeros_like(r)
    z = dinv * r
    p = z.clone()
    rz = (r * z).sum(0)
    stop = tol * r.norm(dim=0)
    for it in range(maxit):
        q = a @ p
        alpha = rz / (p * q).sum(0).clamp_min(1e-300)
        x += alpha * p
        r = r - alpha * q
        if it % 25 == 24 and bool((r.norm(dim=0) <= stop).all()):
            break
        z = dinv * r
        new = (r * z).sum(0)
        p = z + (new / rz.clamp_min(1e-300)) * p
        rz = new
    return x


def _bicgstab(a, r, tol=1e-6, maxit=2000):
    """BiCGStab without a preconditioner, column by column."""
    x = torch.zeros_like(r)
    r0, p = r.clone(), r.clone()
    rho = (r0 * r).sum(0)
    stop = tol * r.norm(dim=0)
    for it in range(maxit):
        v = a @ p
        alpha = rho / (r0 * v).sum(0)
        s = r - alpha * v
        t = a @ s
        omega = (t * s).sum(0) / (t * t).sum(0).clamp_min(1e-300)
        x += alpha * p + omega * s
        r = s - omega * t
        if it % 5 == 4 and bool((r.norm(dim=0) <= stop).all()):
            break
        new = (r0 * r).sum(0)
        p = r + (new / rho) * (alpha / omega) * (p - omega * v)
        rho = new
    return x


def exact(case, seed):
    if case["do"] == "apply":  # a truncated factorization has no exact value
        return None
    shape = _shape(case)
    p = _matrix(case["family"], shape, case.get("decades"))
    b = _rhs(p.n, case["nrhs"], seed)
    if case["family"] == "poisson":
        return _sine_solve(shape, b)
    a = _csr(p, b.device)
    if case["family"] == "vcdiff":
        rows = np.repeat(np.arange(p.n), np.diff(p.rowptr))
        diag = torch.from_numpy(p.val[rows == p.col]).to(b.device)
        return _refined(a, b, 1.0 / diag[:, None], lambda r, s: _cg(a, r, s))
    return _refined(a, b, None, lambda r, s: _bicgstab(a, r))
