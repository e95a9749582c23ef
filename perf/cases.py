"""The eigensolver's work as a user's program gives it, for timing: whole solves and filters and the blocks of
the outer step, on the 1D, 2D and 3D finite-element pencils of this repository from a few hundred unknowns to the
largest named configuration (187 200).

``listed()`` names the cases, ``draw(rng)`` gives further ones of the same ranges, ``prepare(case, seed)`` makes what
a program holds before the call (pencil handle, poles, blocks and output buffers on the GPU), ``run(state)`` is one
call through ``paper_2503_21618_gb300``, ``work(case)`` counts what the call cannot do without and
``exact(case, seed)`` is the same result in plain 64-bit torch.
"""
from __future__ import annotations

import functools
import math
import types

import numpy as np
import torch

import paper_2503_21618_gb300 as slrf
from paper_2503_21618_gb300 import api
from workloads import pencil_1d, pencil_2d_q1, pencil_3d_elasticity, weyl_gamma

MESHES = {"1d": pencil_1d, "2d": pencil_2d_q1, "3d": pencil_3d_elasticity}


def listed():
    # The solver's default is mixed precision: single-precision Krylov blocks (product, cycle below) around a
    # double-precision projection (ritz, eig, gram).  A whole solve or filter in it ends in vectors that one rounding
    # in single precision moves by 1e-5 to 1e-4, and flips the sign of; whole calls are listed in the method's plain
    # double-precision form, whose results can be compared, and the default's blocks each for themselves.
    return [
        # A whole solve of the smallest named configuration: every kernel is a few microseconds, so launches, host
        # polls and the serial small-matrix steps are what a user waits for.
        dict(name="solve_1d_2000", op="solve", mesh="1d", size=2000, nev=20, cols=30, poles=2, double=True),
        # A whole solve of an ordinary member of the batched workload (n = 10 000).
        dict(name="solve_2d_101", op="solve", mesh="2d", size=101, nev=24, cols=36, poles=4, double=True),
        # One application of the filter to a block, all poles and columns solved to 1e-13.
        dict(name="filter_2d_150", op="filter", mesh="2d", size=150, nev=40, cols=60, poles=4, double=True),
        # The shifted block product of the benchmark solve: all 600 (pole, column) systems of the 300 x 300 Q1 mesh
        # (n = 89 401), in single precision.
        dict(name="product_2d_300", op="product", mesh="2d", size=300, nev=100, cols=150, poles=4),
        # The same for the largest named configuration, 3D elasticity (n = 187 200, 1 200 systems), in the
        # node-block form that the solver picks for it.
        dict(name="product_3d_40", op="product", mesh="3d", size=40, nev=200, cols=300, poles=4),
        # A small ragged one (odd column count), as the smaller members of a batch run it.
        dict(name="product_2d_64", op="product", mesh="2d", size=64, nev=20, cols=31, poles=4),
        # One multigrid preconditioner application over all systems: the benchmark's, and a ragged one of a
        # batched problem's size.
        dict(name="cycle_2d_300", op="cycle", mesh="2d", size=300, nev=100, cols=150, poles=4),
        dict(name="cycle_2d_101", op="cycle", mesh="2d", size=101, nev=24, cols=37, poles=4),
        # Rayleigh-Ritz of a filtered block (products, Grams, Cholesky-QR2, small eigenproblem, Ritz vectors,
        # residuals): the benchmark's, and 3D with the 300 columns of the largest configuration and of requests for
        # 200 eigenpairs.
        dict(name="ritz_2d_300", op="ritz", mesh="2d", size=300, nev=100, cols=150, poles=4),
        dict(name="ritz_3d_24", op="ritz", mesh="3d", size=24, nev=200, cols=300, poles=4),
        # The projected eigenproblem alone, at the subspace size of a small request.
        dict(name="eig_45", op="eig", mesh="1d", size=300, nev=30, cols=45, poles=1),
        # The double-precision Gram matrix of two tall blocks, ragged on both sides.
        dict(name="gram_50021x211", op="gram", mesh="1d", size=50021, nev=140, cols=211, poles=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the operation, mesh, size and column count drawn over the ranges the listed ones stand for."""
    op = rng.choice(["solve", "filter", "product", "cycle", "ritz", "eig", "gram", "tall"])
    poles, double = 4, False
    if op == "solve":                      # members of the batched workload
        mesh, double = rng.choice(["1d", "2d"]), True
        size = _log(rng, 300, 2000) if mesh == "1d" else _log(rng, 32, 101)
        nev = rng.randint(10, 20) if mesh == "1d" else rng.randint(10, 24)
        cols = 2 * math.ceil(0.75 * nev)
        poles = rng.choice([2, 4])
    elif op == "filter":
        mesh, double = rng.choice(["1d", "2d"]), True
        size = _log(rng, 300, 20000) if mesh == "1d" else _log(rng, 24, 150)
        nev = rng.randint(8, 20) if mesh == "1d" else rng.randint(8, 40)
        cols = nev + rng.randint(1, nev // 2)
        poles = rng.choice([2, 4, 4])
    elif op == "product":
        mesh = rng.choice(["1d", "2d", "3d"])
        size = _log(rng, *{"1d": (500, 100000), "2d": (24, 300), "3d": (6, 38)}[mesh])
        poles = rng.choice([1, 2, 3, 4, 4, 4, 6])
        nev = rng.randint(5, 100)
        cols = nev + rng.randint(1, 50)
        double = mesh != "3d" and rng.random() < 0.25
    elif op == "cycle":
        mesh = rng.choice(["1d", "2d", "2d"])
        size = _log(rng, 1000, 30000) if mesh == "1d" else _log(rng, 48, 300)
        nev = rng.randint(10, 20) if mesh == "1d" else rng.randint(10, min(100, size // 3))
        cols = nev + rng.randint(1, nev // 2)
        poles = rng.choice([2, 4])
    elif op == "ritz":
        mesh = rng.choice(["2d", "3d"])
        size = _log(rng, 48, 300) if mesh == "2d" else _log(rng, 10, 24)
        cols = rng.randint(15, 150) if mesh == "2d" else rng.randint(15, 300)
        nev = max(5, 2 * cols // 3)
    elif op == "eig":
        mesh, size, poles = "1d", 400, 1
        cols = _log(rng, 8, 300)
        nev = max(5, 2 * cols // 3)
    else:                                  # gram, tall: the pencil only sets the number of rows
        mesh, size, poles = "1d", _log(rng, 1000, 180000), 1
        cols = _log(rng, 12, 300)
        nev = max(5, 2 * cols // 3)
    return dict(op=op, mesh=mesh, size=size, nev=nev, cols=cols, poles=poles, double=double)


# ---------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=3)
def _mesh(mesh, size):
    return MESHES[mesh](size)


@functools.lru_cache(maxsize=None)
def _poles(poles, mesh, nev):
    gamma = weyl_gamma(mesh, nev)
    return gamma, slrf.design_poles("slrf", poles, gamma, 1.0, 0.01)


def _rows(case):
    s = case["size"]
    return {"1d": s, "2d": (s - 1) ** 2, "3d": 3 * (s - 1) * s * s}[case["mesh"]]


def _nnz(case):
    s = case["size"]
    if case["mesh"] == "1d":
        return 3 * s - 2
    if case["mesh"] == "2d":
        return (3 * (s - 1) - 2) ** 2
    return 9 * (3 * (s - 1) - 2) * (3 * s - 2) ** 2


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(g, *shape, dtype=torch.float64):
    return torch.randn(*shape, generator=g, dtype=dtype, device="cuda")


def _state_block(case, seed, dtype):
    """A block over all (pole, column) systems in the solver's state layout: per pole the columns, padded with a
    zero column to an even count."""
    n, m, N = _rows(case), case["cols"], case["poles"]
    ldp = m + (m & 1)
    P = _normal(_generator(seed), n, N, ldp, dtype=dtype)
    P[:, :, m:] = 0
    return P.view(n, N * ldp), ldp


def _filtered_block(case, seed):
    """What an outer step hands to Rayleigh-Ritz: columns near the eigenvectors (here the constant-coefficient modes),
    the ones beyond the interval damped by the filter, and the rest of the spectrum still in them at a per cent."""
    m, s, wanted = case["cols"], case["size"], case["nev"]
    dev = dict(dtype=torch.float64, device="cuda")
    if case["mesh"] == "2d":
        x = torch.arange(1, s, **dev) / s
        k = sorted((a * a + b * b, a, b) for a in range(1, 40) for b in range(1, 40))[:m]
        sx = torch.sin(math.pi * torch.arange(1, 40, **dev)[:, None] * x)
        U = torch.stack([(sx[b - 1][:, None] * sx[a - 1][None, :]).reshape(-1) for _, a, b in k], dim=1)
    else:
        x, y = torch.arange(1, s, **dev) / (s - 1), torch.arange(0, s, **dev) / (s - 1)
        q = torch.arange(0, 12, **dev)[:, None]
        sx, cy = torch.sin(math.pi * (q + 0.5) * x), torch.cos(math.pi * q * y)
        k = sorted(((a + 0.5) ** 2 + b * b + c * c, a, b, c) for a in range(12) for b in range(9) for c in range(9))
        U = torch.zeros(_rows(case), m, **dev)
        for j in range(m):
            _, a, b, c = k[j // 3]
            U[j % 3::3, j] = torch.einsum("z,y,x->zyx", cy[c], cy[b], sx[a]).reshape(-1)
    U /= U.norm(dim=0)
    U += _normal(_generator(seed), *U.shape) * (1e-2 / math.sqrt(U.shape[0]))
    return U * torch.clamp(wanted / torch.arange(1, m + 1, **dev), max=1.0) ** 6


def _projected(case, seed):
    """The projected matrix of an outer step: nearly diagonal, its eigenvalues growing as the pencil's do."""
    m = case["cols"]
    g = _generator(seed)
    lam = 20.0 + 12.0 * (torch.arange(m, dtype=torch.float64, device="cuda")
                         + 0.4 * torch.rand(m, generator=g, dtype=torch.float64, device="cuda"))
    E = _normal(g, m, m) * (1e-2 / math.sqrt(m))
    return torch.diag(lam) + (E + E.T) * torch.sqrt(lam[:, None] * lam[None, :])


def _inputs(case, seed):
    n, m, op = _rows(case), case["cols"], case["op"]
    if op in ("solve", "filter"):
        return (_normal(_generator(seed), n, m),)
    if op == "product":
        return (_state_block(case, seed, torch.complex128 if case.get("double") else torch.complex64)[0],)
    if op == "cycle":
        return (_state_block(case, seed, torch.complex64)[0],)
    if op == "ritz":
        return (_filtered_block(case, seed),)
    if op == "eig":
        return (_projected(case, seed),)
    g = _generator(seed)
    if op == "gram":
        X = _normal(g, n, m)
        return X, X + 0.1 * _normal(g, n, m)
    return _normal(g, n, m) / math.sqrt(n), torch.linalg.qr(_normal(g, m, m))[0].contiguous()


def prepare(case, seed):
    op, m = case["op"], case["cols"]
    s = types.SimpleNamespace(op=op, m=m, x=_inputs(case, seed))
    opts = {}
    if op in ("eig", "gram", "tall", "ritz", "product"):
        opts["precond"] = slrf.PRECOND_JACOBI            # no hierarchy: these calls do not precondition
    if op == "product" and case["mesh"] == "3d":
        opts["spmm_kernel"] = api.SPMM_NODEBLOCK         # what the solver's own timing picks for elasticity
    if op in ("solve", "filter"):
        opts.update(precision=slrf.PREC_FP64, inner_tol=1e-13)
    s.h = slrf.Handle(_mesh(case["mesh"], case["size"]), slrf.default_opts(**opts))
    s.gamma, s.f = _poles(case["poles"], case["mesh"], case["nev"])
    x = s.x[0]
    if op in ("solve", "filter"):
        s.out = torch.empty_like(x)
        s.theta, s.resid = torch.empty_like(x[0]), torch.empty_like(x[0])
    if op in ("product", "cycle"):
        s.ldp = x.shape[1] // case["poles"]
        s.prec = slrf.PREC_FP64 if x.dtype == torch.complex128 else slrf.PREC_MIXED
        s.out = torch.zeros_like(x)
        s.mu = torch.zeros(case["poles"] * m, dtype=x.dtype, device="cuda")
    return s


def run(s):
    if s.op == "solve":
        theta, X, _, n_conv, _, _ = s.h.subspace_iterate(s.f, s.gamma, s.x[0], theta=s.theta, X=s.out, resid=s.resid)
        return {"theta": theta, "X": X, "n_conv": n_conv}   # (the residuals are at rounding level)
    if s.op == "filter":
        return {"U": s.h.filter_apply(s.f, s.x[0], s.out)[0]}
    if s.op == "product":
        return {"Q": s.h.shifted_spmm(s.f, s.x[0], s.m, s.ldp, prec=s.prec, Q=s.out, mu=s.mu), "mu": s.mu}
    if s.op == "cycle":
        return {"Z": s.h.precond_apply(s.f, s.x[0], s.m, s.ldp, prec=s.prec, Z=s.out, mu=s.mu)[0], "mu": s.mu}
    if s.op == "ritz":
        theta, X, resid = s.h.rayleigh_ritz(s.x[0])
        return {"theta": theta, "X": X, "resid": resid}
    if s.op == "eig":
        lam, Q = s.h.syev(s.x[0])
        return {"lam": lam, "Q": Q}
    if s.op == "gram":
        return {"G": s.h.gram(*s.x)}
    return {"C": s.h.tall_product(*s.x)}


def work(case):
    """Bytes of inputs read once and outputs written once, and the arithmetic of the definition.  A Krylov iteration
    reads and writes its three blocks and the pencil; the iteration counts are those the method needs on these
    meshes (about 25 with multigrid to a tolerance of 1e-13; 6 outer steps)."""
    n, nnz, m, N = float(_rows(case)), float(_nnz(case)), case["cols"], case["poles"]
    op, W = case["op"], case["cols"] * case["poles"]
    double = case.get("double", False)
    z, pencil = (16.0 if double else 8.0), 4.0 * n + nnz * (4 + (16 if double else 8))
    product = dict(bytes=pencil + 2 * z * n * W, flops=8.0 * nnz * W)
    # products A U, B U, B Q, A Q, A X, B X; Grams of U, Q and A; the two tall products
    ritz = dict(bytes=4 * n + 20 * nnz + 16 * n * m, flops=12.0 * nnz * m + 10.0 * n * m * m)
    if op == "product":
        return product
    if op == "cycle":       # two gathered products of the fine level, once over the block and back
        return dict(bytes=product["bytes"], flops=2.5 * product["flops"])
    if op == "ritz":
        return ritz
    if op == "eig":
        return dict(bytes=16.0 * m * m, flops=9.0 * m ** 3)
    if op == "gram":
        return dict(bytes=16 * n * m + 8 * m * m, flops=2 * n * m * m)
    if op == "tall":
        return dict(bytes=16 * n * m + 8 * m * m, flops=2 * n * m * m)
    iters, steps = (25, 6) if op == "solve" else (25, 1)
    one = dict(bytes=iters * (pencil + 6 * z * n * W), flops=iters * 3.5 * product["flops"])
    more = ritz if op == "solve" else dict(bytes=16 * n * m, flops=2 * nnz * m)
    return {k: steps * (one[k] + more[k]) for k in one}


# ---------------------------------------------------------------- the same in plain 64-bit torch
def _csr(p, values):
    return torch.sparse_csr_tensor(torch.from_numpy(p.row_ptr.astype(np.int64)), torch.from_numpy(p.col_idx.astype(np.int64)),
                                   torch.from_numpy(values), size=(p.n, p.n), dtype=torch.float64).cuda()


def _times(M, X):
    """Sparse times dense, real or complex, in column chunks."""
    if X.is_complex():
        return torch.complex(_times(M, X.real.contiguous()), _times(M, X.imag.contiguous()))
    return torch.cat([M @ X[:, c:c + 256].contiguous() for c in range(0, X.shape[1], 256)], dim=1)


def exact(case, seed):
    op, m, N = case["op"], case["cols"], case["poles"]
    if op in ("solve", "cycle") or (op == "filter" and _rows(case) > 8000):
        return None      # iterates of the method, its own hierarchy; a dense solve per pole that takes too long
    x = _inputs(case, seed)
    if op == "eig":
        return {"lam": torch.linalg.eigvalsh(x[0]), "Q": None}
    if op == "gram":
        return {"G": x[0].T @ x[1]}
    if op == "tall":
        return {"C": x[0] @ x[1]}
    p = _mesh(case["mesh"], case["size"])
    _, f = _poles(N, case["mesh"], case["nev"])
    A, B = _csr(p, p.a_val), _csr(p, p.b_val)
    if op == "product":
        ldp = x[0].shape[1] // N
        Q, mu = torch.empty(p.n, N * ldp, dtype=torch.complex128, device="cuda"), []
        for j in range(N):
            P = x[0][:, j * ldp:(j + 1) * ldp].to(torch.complex128)
            Q[:, j * ldp:(j + 1) * ldp] = _times(A, P) - complex(f.sigma[j]) * _times(B, P)
            mu.append((P * Q[:, j * ldp:(j + 1) * ldp]).sum(dim=0)[:m])
        return {"Q": Q, "mu": torch.cat(mu)}
    if op == "filter":
        F, U = _times(B, x[0]), torch.zeros_like(x[0])
        Ad, Bd = A.to_dense(), B.to_dense()
        for sigma, w in zip(f.sigma, f.w):
            Y = torch.linalg.solve(Ad - complex(sigma) * Bd, F.to(torch.complex128))
            U += 2 * (complex(w) * Y).real
        return {"U": U}
    Q = x[0] / x[0].norm(dim=0)
    for _ in range(2):   # Cholesky-QR2 in the B inner product
        R = torch.linalg.cholesky(Q.T @ _times(B, Q), upper=True)
        Q = torch.linalg.solve_triangular(R, Q, upper=True, left=False)
    H = Q.T @ _times(A, Q)
    theta, S = torch.linalg.eigh((H + H.T) / 2)
    X = Q @ S
    AX, BX = _times(A, X), _times(B, X)
    resid = (AX - theta * BX).norm(dim=0) / (theta.abs() * BX.norm(dim=0))
    return {"theta": theta, "X": None, "resid": resid}   # eigenvectors: up to sign
