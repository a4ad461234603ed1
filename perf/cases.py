"""The work that programs have this solver do, as cases that can be timed.

A case is a dict of plain values.  `kind` says which calls of the library one
pass makes, through the binding that tests and serving use:

  step    new values on a known pattern: Factor.refactor, then Factor.pcg
          (the benchmark's step; time stepping, parameter sweeps)
  solve   Factor.pcg on a resident factorization (the bulk of the served
          requests, 1 to 16 right-hand sides)
  first   a matrix seen for the first time: Factor(...), one Factor.pcg, close
          (a served factor request, a one-off solve)
  batch   many small systems: refactor_batch, then one Factor.pcg each
  apply   Factor.apply on a resident factorization (the preconditioner inside
          the caller's own outer solver)
  gmres   Factor.gmres on a resident factorization (the outer solver of the
          paper's tables)

Grids are nx x ny (x nz; nz = 0 means two-dimensional).  `s` is the exponent of
the log-normal coefficient field exp(s g) (0: Poisson), `seed` of prepare()
makes the field and the right-hand sides.  Tolerances are the library's and the
benchmark's own: eps 1e-2 (0.1 for the tables), PCG and GMRES to 1e-10 (`rtol`),
and 1e-11 on the unscaled 512 x 512 grid, whose condition number (1e5) would
otherwise show in the digits that a caller compares.
"""
from __future__ import annotations

import math
from functools import lru_cache

import numpy as np
import torch

from paper_1611_03189_gb300 import _lib
from paper_1611_03189_gb300 import problems as P

PREC = {"f64": _lib.HS_PREC_F64, "f32": _lib.HS_PREC_F32, "tf32": _lib.HS_PREC_TF32,
        "tf32x3": _lib.HS_PREC_TF32X3, "bf16": _lib.HS_PREC_BF16}


def _case(kind, nx, ny, nz=0, s=1.0, prec="f32", nrhs=1, leaf=16, scale=False, eps=1e-2, nbr=1, rtol=1e-10,
          name=None):
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "s": s, "prec": prec, "nrhs": nrhs, "leaf": leaf,
         "scale": scale, "eps": eps, "nbr": nbr, "rtol": rtol}
    if name:
        c["name"] = name
    return c


def _batch(count, lo, hi, sides_seed, prec="f32", nrhs=4, name=None):
    c = {"kind": "batch", "count": count, "lo": lo, "hi": hi, "sides_seed": sides_seed, "s": 1.0, "prec": prec,
         "nrhs": nrhs, "leaf": 16, "scale": True, "eps": 1e-2, "nbr": 1, "rtol": 1e-10}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the plain method's configuration: one small FP64 solve, where launches and latency are all there is
        _case("solve", 64, 64, s=0.0, prec="f64", name="solve_poisson_64_f64"),
        # the same problem seen for the first time: planning, first factorization, solve, release
        _case("first", 64, 64, s=0.0, prec="f64", name="first_poisson_64_f64"),
        # the benchmark's step: a new coefficient field on a known 512 x 512 pattern, factored and solved
        _case("step", 512, 512, rtol=1e-11, name="step_diffusion_512_f32"),
        # the same step in plain FP64, on a ragged grid
        _case("step", 331, 198, prec="f64", scale=True, name="step_diffusion_331x198_f64"),
        # a solve alone on the benchmark's resident factor
        _case("solve", 512, 512, rtol=1e-11, name="solve_diffusion_512_f32"),
        # a served solve request: three dimensions, diagonally scaled, 16 right-hand sides
        _case("solve", 40, 40, 40, s=2.0, nrhs=16, leaf=64, scale=True, name="solve_diffusion3d_40_f32_16rhs"),
        # the three-dimensional Poisson configuration, factored on the tensor cores in TF32 and BF16
        _case("step", 40, 40, 40, s=0.0, prec="tf32", leaf=64, name="step_poisson3d_40_tf32"),
        _case("step", 27, 24, 31, s=0.0, prec="bf16", leaf=64, name="step_poisson3d_27x24x31_bf16"),
        # a served factor request with its first solve: a three-dimensional matrix not seen before
        _case("first", 28, 28, 28, s=2.0, leaf=64, scale=True, nrhs=3, name="first_diffusion3d_28_f32_3rhs"),
        # many independent systems of uneven size, four right-hand sides each
        _batch(24, 32, 160, 5, name="batch_24_diffusion_f32_4rhs"),
        # the preconditioner alone, inside somebody else's outer solver
        _case("apply", 300, 217, prec="f64", scale=True, nrhs=5, name="apply_diffusion_300x217_f64_5rhs"),
        # the paper's table 2: GMRES, leaves of 8, neighbours at distance two
        _case("gmres", 256, 256, s=0.0, leaf=8, eps=0.1, nbr=2, name="gmres_poisson_256_f32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "solve", "solve", "first", "batch", "apply", "gmres"])
    if kind == "batch":
        lo = rng.randint(16, 48)
        return _batch(rng.randint(3, 20), lo, _log(rng, 64, 160), rng.randrange(1 << 16),
                      prec=rng.choice(["f32", "f32", "f64"]) if lo < 32 else "f32", nrhs=rng.randint(1, 6))
    if kind == "gmres":
        return _case("gmres", _log(rng, 32, 256), _log(rng, 32, 256), s=0.0, leaf=8, eps=0.1,
                     nbr=2, prec=rng.choice(["f32", "f64"]))
    if kind == "apply":
        # FP64: the application itself is the result, so its own precision is what a caller asks for
        if rng.random() < 0.5:
            return _case("apply", _log(rng, 32, 320), _log(rng, 32, 320), s=rng.choice([0.0, 1.0]), prec="f64",
                         scale=True, nrhs=rng.randint(1, 16))
        return _case("apply", rng.randint(9, 24), rng.randint(9, 24), rng.randint(9, 24),
                     s=rng.choice([0.0, 1.0, 2.0]), prec="f64", leaf=64, scale=True, nrhs=rng.randint(1, 16))
    nrhs = 1 if kind == "step" else rng.randint(1, 16)
    if rng.random() < 0.55:
        prec = rng.choice(["f32", "f32", "f32", "tf32x3", "f64"])
        top = 224 if prec == "f64" else 448
        return _case(kind, _log(rng, 32, top), _log(rng, 32, top), s=rng.choice([0.0, 1.0, 1.0]), prec=prec,
                     scale=True, nrhs=nrhs)
    prec = rng.choice(["f32", "f32", "tf32", "tf32x3", "bf16", "f64"])
    top = 20 if prec == "f64" else 34
    return _case(kind, rng.randint(10, top), rng.randint(10, top), rng.randint(10, top),
                 s=rng.choice([0.0, 1.0, 2.0]), prec=prec, leaf=64, scale=True, nrhs=nrhs)


def _shape(c):
    return (c["nx"], c["ny"]) + ((c["nz"],) if c["nz"] else ())


@lru_cache(maxsize=64)
def _clusters(shape, leaf):
    return P.bisect_clusters(shape, P.levels_for(int(np.prod(shape)), leaf))


def _matrix(shape, s, seed):
    coef = P.coef_lognormal(shape, s, seed) if s > 0.0 else P.coef_constant(shape)
    rp, ci, va = P.stencil_matrix(shape, coef)
    return torch.from_numpy(rp).cuda(), torch.from_numpy(ci).cuda(), torch.from_numpy(va).cuda()


def _rhs(n, nrhs, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    b = torch.randn(nrhs, n, generator=g, device="cuda", dtype=torch.float64)
    return b[0] if nrhs == 1 else b


def _factor(c, A, perm, leaf_ptr):
    return _lib.Factor(*A, perm, leaf_ptr, c["eps"], _lib.HS_GC_CONSTANT, PREC[c["prec"]], nbr_dist=c["nbr"],
                       scale=c["scale"])


def _batch_shapes(c):
    return [(k, k) for k in P.batched_sides(c["count"], c["sides_seed"], c["lo"], c["hi"])]


def prepare(case, seed):
    st = {"case": case}
    if case["kind"] == "batch":
        shapes = _batch_shapes(case)
        cl = [_clusters(sh, case["leaf"]) for sh in shapes]
        # the handles hold another step's factorization; one pass brings the values of `A`
        old = [_matrix(sh, case["s"], seed + 50_000 + i) for i, sh in enumerate(shapes)]
        st["A"] = [_matrix(sh, case["s"], seed + i) for i, sh in enumerate(shapes)]
        st["factors"], status = _lib.factor_batch([(*A, *pl) for A, pl in zip(old, cl)], case["eps"],
                                                  prec=PREC[case["prec"]], nbr_dist=case["nbr"],
                                                  scale=case["scale"])
        assert not status.any(), status
        st["b"] = [_rhs(A[0].numel() - 1, case["nrhs"], seed + i) for i, A in enumerate(st["A"])]
        return st
    shape = _shape(case)
    st["clusters"] = _clusters(shape, case["leaf"])
    st["A"] = _matrix(shape, case["s"], seed)
    st["b"] = _rhs(int(np.prod(shape)), case["nrhs"], seed)
    if case["kind"] == "step":
        # the handle holds the previous step's factorization of the same pattern
        st["factor"] = _factor(case, _matrix(shape, case["s"], seed + 50_000), *st["clusters"])
    elif case["kind"] != "first":
        st["factor"] = _factor(case, st["A"], *st["clusters"])
    return st


def run(st):
    c = st["case"]
    kind = c["kind"]
    if kind == "batch":
        status = _lib.refactor_batch(st["factors"], [A[2] for A in st["A"]])
        assert not status.any(), status
        return [f.pcg(b, rtol=c["rtol"])[0] for f, b in zip(st["factors"], st["b"])]
    if kind == "first":
        f = _factor(c, st["A"], *st["clusters"])
        x = f.pcg(st["b"], rtol=c["rtol"])[0]
        f.close()
        return x
    f = st["factor"]
    if kind == "apply":
        return f.apply(st["b"])
    if kind == "gmres":
        return f.gmres(st["b"], rtol=c["rtol"])[0]
    if kind == "step":
        f.refactor(st["A"][2])
    return f.pcg(st["b"], rtol=c["rtol"])[0]


def _grid_work(c, shape):
    n = float(np.prod(shape))
    d = len(shape)
    nnz = (2 * d + 1) * n
    word = 8 if c["prec"] == "f64" else 4
    # words of the factor records and flops of the factorization per unknown
    # (hs_info.factor_bytes and alg_flops of these recipes, fitted over the grid sizes)
    if d == 3:
        words, flops = 1215.0 * (n / 64000.0) ** 0.24, 5.8e6 * (n / 64000.0) ** 0.85
    elif c["leaf"] == 16:
        words, flops = 150.0 * (n / 4096.0) ** 0.07, 50e3 * (n / 4096.0) ** 0.25
    else:
        words, flops = 107.0, 25e3
    records = words * n * word
    vectors = 16.0 * n * c["nrhs"]                        # right-hand sides in, solutions out
    factor = flops * n if c["kind"] in ("step", "first", "batch") else 0.0
    matrix = 0.0 if c["kind"] == "apply" else 12.0 * nnz   # values and columns
    return matrix + records + vectors, factor + 2.0 * words * n * c["nrhs"]


def work(case):
    shapes = _batch_shapes(case) if case["kind"] == "batch" else [_shape(case)]
    each = [_grid_work(case, sh) for sh in shapes]
    return {"bytes": sum(e[0] for e in each), "flops": sum(e[1] for e in each)}


def _solve_exact(A, b):
    """A^-1 b in FP64 by diagonally preconditioned CG to stagnation, with two restarts on the true residual."""
    rp, ci, va = A
    n = rp.numel() - 1
    M = torch.sparse_csr_tensor(rp, ci, va, size=(n, n))
    rows = torch.repeat_interleave(torch.arange(n, device=va.device), rp[1:] - rp[:-1])
    dinv = torch.zeros(n, dtype=va.dtype, device=va.device)
    at = rows == ci
    dinv[rows[at]] = 1.0 / va[at]
    dinv = dinv[:, None]
    B = b.reshape(-1, n).t().contiguous()
    x = torch.zeros_like(B)
    for _ in range(3):
        r = B - M @ x
        z = dinv * r
        p = z.clone()
        d = torch.zeros_like(B)
        rz = (r * z).sum(0)
        stop = 1e-15 * rz
        for it in range(20000):
            q = M @ p
            pq = (p * q).sum(0)
            a = torch.where(pq > 0, rz / pq, torch.zeros_like(rz))
            d += a * p
            r -= a * q
            z = dinv * r
            new = (r * z).sum(0)
            p = z + torch.where(rz > 0, new / rz, torch.zeros_like(rz)) * p
            rz = new
            if it % 50 == 49 and bool((rz <= stop).all()):
                break
        x = x + d
    return x.t().contiguous().reshape(b.shape)


def exact(case, seed):
    """What run() returns, from A x = b itself.  An application of the preconditioner has no such value."""
    if case["kind"] == "apply":
        return None
    if case["kind"] == "batch":
        out = []
        for i, sh in enumerate(_batch_shapes(case)):
            A = _matrix(sh, case["s"], seed + i)
            out.append(_solve_exact(A, _rhs(A[0].numel() - 1, case["nrhs"], seed + i)))
        return out
    A = _matrix(_shape(case), case["s"], seed)
    return _solve_exact(A, _rhs(A[0].numel() - 1, case["nrhs"], seed))
