"""Performance cases of the library: the calls its users make, over the sizes,
storage formats, preconditioners and solvers it is used with.

A case is a plain dict.  ``listed()`` names the standing ones, ``draw(rng)``
gives others of the same families and ranges; ``prepare`` builds the inputs
and the handles a program keeps, ``run`` makes one pass through the public
entry points, ``work`` states what a pass cannot do without and ``exact``
what it should return, computed in FP64 with plain torch.

Families
  apply   y = A x, or y = alpha A x + beta y, with a kept operator
  setup   a new operator: format conversion, preconditioner generation and
          their first use (an implicit time step or a Newton step assembles
          one of these per solve)
  solve   a preconditioned Krylov solve with a kept solver
  batch   thousands of independent small systems in one call
  infer   BF16 inference of the warm-start network
  train   loss and gradients of the warm-start network (FP32)

Solves run to a relative residual of 1e-12, so that the solution is
determined well beyond the rounding of the reductions; GMRES, which would
need thousands of steps on its matrix, runs a fixed number of them.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

import paper_2006_16852_gb300 as gk
from paper_2006_16852_gb300 import learned

DEV = "cuda:0"
TOL = 1e-12
STENCIL5 = ((-1, 0), (0, -1), (0, 0), (0, 1), (1, 0))
STENCIL7 = ((-1, 0, 0), (0, -1, 0), (0, 0, -1), (0, 0, 0), (0, 0, 1), (0, 1, 0), (1, 0, 0))
STENCIL27 = tuple((a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1))


def listed():
    return [
        # The smallest call: one advanced apply of a small ragged operator
        # (a coarse multigrid level, a network Laplacian); launch latency.
        dict(name="apply_ragged_4k", family="apply", matrix="ragged", n=4099, fmt="csr", adv=True),
        # An irregular operator at full size in the default format: the
        # power-law matrix of the benchmark (rows of 1 to 10,000 entries).
        dict(name="apply_powerlaw_1m", family="apply", matrix="powerlaw", n=1_000_000, fmt="csr", adv=False),
        # A newly assembled operator with block Jacobi, at a size that is no
        # multiple of anything: 7-point diffusion on 99 x 101 x 103.
        dict(name="setup_diffusion3d_1m", family="setup", matrix="diffusion3d", nz=99, ny=101, nx=103, fmt="csr", bs=8),
        # The small solve (configuration 0 of the benchmark): Poisson 64^2.
        dict(name="cg_poisson2d_64", family="solve", kind="cg", matrix="poisson2d", ny=64, nx=64, fmt="csr", prec=1),
        # The mid-size solve: variable-coefficient diffusion on 256^2, the
        # grid of the warm-start network's problems.
        dict(name="cg_diffusion2d_256", family="solve", kind="cg", matrix="diffusion2d", ny=256, nx=256, fmt="csr",
             prec=1),
        # The large solve of the benchmark: 27-point stencil on 128^3.
        dict(name="cg_stencil27_128", family="solve", kind="cg", matrix="stencil27", nz=128, ny=128, nx=128, fmt="ell",
             prec=1),
        # A nonsymmetric mid-size solve on a ragged grid (an implicit
        # transport step).
        dict(name="bicgstab_convdiff_201x199", family="solve", kind="bicgstab", matrix="convdiff", ny=201, nx=199,
             fmt="csr", prec=1),
        # Restarted GMRES on a large nonsymmetric system: two cycles of 30.
        dict(name="gmres_convdiff_1024", family="solve", kind="gmres", matrix="convdiff", ny=1024, nx=1024, fmt="ell",
             prec=1, steps=60),
        # The mixed-precision solve: FP64 refinement around FP32 CG with
        # adaptive FP16/FP32 block Jacobi, on the benchmark's log-normal
        # diffusion at half its side.
        dict(name="ir_diffusion3d_128", family="solve", kind="ir_cg", matrix="diffusion3d", nz=128, ny=128, nx=128,
             fmt="ell", prec=8),
        # The batched workload of the benchmark: 10,000 systems of 36 to
        # 1024 rows, per-system refinement.
        dict(name="batch_ir_10000", family="batch", kind="ir_cg", systems=10_000, side_lo=6, side_hi=32),
        # Serving the warm-start network: one full batch of 256^2 problems.
        dict(name="infer_256_b64", family="infer", batch=64),
        # Training it: loss and gradients of one batch of 16.
        dict(name="train_256_b16", family="train", side=256, batch=16, loss="energy"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["apply", "apply", "setup", "solve", "solve", "solve", "solve", "batch", "infer", "train"])
    if family == "apply":
        fmt = rng.choice(["csr", "csr_merge", "ell", "hyb"])
        adv = rng.random() < 0.4
        matrix = rng.choice(["stencil27", "diffusion3d"] if fmt == "ell" else ["ragged", "powerlaw", "stencil27"])
        if matrix in ("ragged", "powerlaw"):
            return dict(family=family, matrix=matrix, n=_log_int(rng, 2_000, 1_000_000), fmt=fmt, adv=adv)
        return dict(family=family, matrix=matrix, nz=_log_int(rng, 12, 110), ny=_log_int(rng, 12, 110),
                    nx=_log_int(rng, 12, 110), fmt=fmt, adv=adv)
    if family == "setup":
        fmt = rng.choice(["csr", "ell", "hyb"])
        return dict(family=family, matrix="diffusion3d", nz=_log_int(rng, 10, 100), ny=_log_int(rng, 10, 100),
                    nx=_log_int(rng, 10, 100), fmt=fmt, bs=rng.choice([1, 4, 8, 16]))
    if family == "solve":
        kind = rng.choice(["cg", "cg", "cg", "fcg", "bicgstab", "gmres", "ir_cg"])
        if kind in ("bicgstab", "gmres"):
            hi = 260 if kind == "bicgstab" else 1000
            c = dict(family=family, kind=kind, matrix="convdiff", ny=_log_int(rng, 40, hi), nx=_log_int(rng, 40, hi),
                     fmt=rng.choice(["csr", "ell"]), prec=1)
            if kind == "gmres":
                c["steps"] = rng.choice([30, 45, 60])
            return c
        if kind == "cg":
            matrix = rng.choice(["poisson2d", "diffusion2d", "diffusion2d", "stencil27", "diffusion3d"])
        else:
            matrix = rng.choice(["stencil27", "diffusion3d"])
        c = dict(family=family, kind=kind, matrix=matrix)
        if matrix in ("poisson2d", "diffusion2d"):
            c.update(ny=_log_int(rng, 20, 400), nx=_log_int(rng, 20, 400))
        else:
            c.update(nz=_log_int(rng, 10, 100), ny=_log_int(rng, 10, 100), nx=_log_int(rng, 10, 100))
        prec = rng.choice([1, 8] if kind == "ir_cg" else [0, 1, 1, 4, 8] if kind == "cg" else [0, 1])
        c.update(fmt=rng.choice(["csr", "ell"]), prec=prec)
        return c
    if family == "batch":
        lo = rng.randint(4, 16)
        return dict(family=family, kind=rng.choice(["ir_cg", "cg"]), systems=_log_int(rng, 100, 10_000), side_lo=lo,
                    side_hi=rng.randint(lo, 32))
    if family == "infer":
        return dict(family=family, batch=_log_int(rng, 1, 64))
    return dict(family=family, side=rng.choice([64, 128, 256]), batch=_log_int(rng, 1, 16),
                loss=rng.choice(["energy", "mse"]))


# ---- inputs ---------------------------------------------------------------------

def _rng(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _uniform(n, g):
    return torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * 2.0 - 1.0


class _Grid:
    """A stencil operator, one (neighbour column, value) pair of vectors per
    stencil offset in increasing column order; value 0 outside the grid."""

    def __init__(self, delta, ok, values):
        self.delta, self.ok, self.values = delta, ok, values
        self.n = ok[0].numel()

    def csr(self):
        rows = torch.arange(self.n, device=DEV, dtype=torch.int32)
        mask = torch.stack(self.ok, 1)
        rowptr = torch.zeros(self.n + 1, device=DEV, dtype=torch.int32)
        rowptr[1:] = mask.sum(1).cumsum(0)
        val = torch.stack(self.values, 1)[mask]
        col = torch.stack([rows + d.to(torch.int32) for d in self.delta], 1)[mask]
        return rowptr, col, val

    def apply(self, x):
        rows = torch.arange(self.n, device=DEV)
        y = torch.zeros_like(x)
        for d, ok, v in zip(self.delta, self.ok, self.values):
            y += torch.where(ok, v * x[(rows + d).clamp_(0, self.n - 1)], 0.0)
        return y

    def diagonal(self):
        return self.values[len(self.values) // 2]


def _shifted(shape, offsets):
    """Column offset and in-grid mask of every stencil offset."""
    n = math.prod(shape)
    strides = [math.prod(shape[d + 1:]) for d in range(len(shape))]
    rows = torch.arange(n, device=DEV)
    axes = [(rows // strides[d]) % shape[d] for d in range(len(shape))]
    delta, oks = [], []
    for off in offsets:
        ok = torch.ones(n, dtype=torch.bool, device=DEV)
        for d, o in enumerate(off):
            if o:
                ok &= (axes[d] + o >= 0) & (axes[d] + o < shape[d])
        delta.append(torch.tensor(sum(o * s for o, s in zip(off, strides)), device=DEV))
        oks.append(ok)
    return delta, oks


def _constant(shape, offsets, weights):
    delta, oks = _shifted(shape, offsets)
    return _Grid(delta, oks, [torch.where(ok, float(w), 0.0).double() for ok, w in zip(oks, weights)])


def _diffusion(coef, delta, oks):
    """Variable-coefficient diffusion: faces the harmonic mean of the two
    cells' coefficients, a face on the boundary the cell's own."""
    rows = torch.arange(coef.numel(), device=DEV)
    diag = torch.zeros_like(coef)
    values = []
    for k, (d, ok) in enumerate(zip(delta, oks)):
        if k == len(delta) // 2:
            values.append(diag)
            continue
        other = coef[(rows + d).clamp_(0, coef.numel() - 1)]
        face = torch.where(ok, 2.0 * coef * other / (coef + other), coef)
        diag += face
        values.append(torch.where(ok, -face, 0.0))
    return _Grid(delta, oks, values)


def _grid(case, g):
    m = case["matrix"]
    shape = tuple(case[a] for a in ("nz", "ny", "nx") if a in case)
    if m == "poisson2d":
        return _constant(shape, STENCIL5, (-1, -1, 4, -1, -1))
    if m == "convdiff":  # first-order upwind, wind 0.5 along +x
        return _constant(shape, STENCIL5, (-1, -1.5, 4.5, -1, -1))
    if m == "stencil27":
        return _constant(shape, STENCIL27, [26 if o == (0, 0, 0) else -1 for o in STENCIL27])
    sigma = 0.5 if m == "diffusion2d" else 1.0
    coef = torch.exp(sigma * torch.randn(math.prod(shape), generator=g, device=DEV, dtype=torch.float64))
    return _diffusion(coef, *_shifted(shape, STENCIL5 if m == "diffusion2d" else STENCIL7))


def _batch_grid(case, g):
    """The block-diagonal matrix of many small 2D diffusion problems, and the
    offsets of their rows: every side equally often, in a random order."""
    at = torch.randperm(case["systems"], generator=g, device=DEV)
    side = case["side_lo"] + at % (case["side_hi"] - case["side_lo"] + 1)
    ptr = torch.zeros(case["systems"] + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = (side * side).cumsum(0)
    n = int(ptr[-1])
    of = torch.repeat_interleave(torch.arange(case["systems"], device=DEV), side * side)
    s, loc = side[of], torch.arange(n, device=DEV) - ptr[of]
    i, j = loc // s, loc % s
    zero = torch.zeros_like(s)
    delta = [-s, zero - 1, zero, zero + 1, s]
    oks = [i > 0, j > 0, s > 0, j < s - 1, i < s - 1]
    coef = torch.exp(0.5 * torch.randn(n, generator=g, device=DEV, dtype=torch.float64))
    return _diffusion(coef, delta, oks), ptr


def _csr_from_entries(n, row, col, val):
    key, at = torch.sort(row * n + col)
    val = val[at]
    first = torch.ones_like(key, dtype=torch.bool)
    first[1:] = key[1:] != key[:-1]
    key, val = key[first], val[first]
    rowptr = torch.zeros(n + 1, device=DEV, dtype=torch.int32)
    rowptr[1:] = torch.bincount(key // n, minlength=n).cumsum(0)
    return rowptr, (key % n).to(torch.int32), val


def _irregular(case, g):
    """ragged: rows of 0 to 40 entries, a tenth of them empty.  powerlaw: row
    lengths of a Zipf(1.8) law capped at 10^4, columns uniform, the pattern
    symmetrised, a dominant diagonal."""
    n = case["n"]
    if case["matrix"] == "ragged":
        lens = torch.randint(0, 41, (n,), generator=g, device=DEV)
        lens[torch.rand(n, generator=g, device=DEV) < 0.1] = 0
    else:
        k = torch.arange(1, min(n, 10_000) + 1, device=DEV, dtype=torch.float64)
        cdf = torch.cumsum(k ** -1.8, 0)
        u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * cdf[-1]
        lens = torch.searchsorted(cdf, u).clamp_(max=k.numel() - 1) + 1
    row = torch.repeat_interleave(torch.arange(n, device=DEV), lens)
    col = torch.randint(0, n, (row.numel(),), generator=g, device=DEV)
    val = torch.randn(row.numel(), generator=g, device=DEV, dtype=torch.float64)
    if case["matrix"] == "powerlaw":
        d = torch.arange(n, device=DEV)
        weight = torch.full((n,), 1000.0, device=DEV, dtype=torch.float64)
        row, col, val = torch.cat([row, col, d]), torch.cat([col, row, d]), torch.cat([val, val, weight])
    return _csr_from_entries(n, row, col, val)


def _fields(count, side, g):
    """Smooth random log-coefficient fields and sources of unit mean square,
    as the network's inputs (count, 2, side, side)."""
    t = (torch.arange(side, device=DEV, dtype=torch.float64) + 1.0) / (side + 1.0)
    out = torch.empty((count, 2, side, side), device=DEV, dtype=torch.float64)
    for ch, (modes, width) in enumerate(((16, 1.6), (8, 3.0))):
        k = torch.randn((count, modes, 2), generator=g, device=DEV, dtype=torch.float64) * (width * 2.0 * math.pi)
        phase = torch.rand((count, modes, 1), generator=g, device=DEV, dtype=torch.float64) * (2.0 * math.pi)
        u = k[:, :, 0:1] * t + phase
        v = k[:, :, 1:2] * t
        f = torch.cos(v).mT @ torch.cos(u) - torch.sin(v).mT @ torch.sin(u)
        out[:, ch] = f * math.sqrt(2.0 / modes)
    out[:, 1] /= out[:, 1].square().mean((1, 2), keepdim=True).sqrt()
    return out


def _weights_file():
    return os.path.join(learned.DATA_DIR, "wsnet_256.npz")


def _network_inputs(case, seed):
    g = _rng(seed)
    side = case.get("side", 256)
    f = _fields(case["batch"], side, g)
    x = f.float().contiguous()
    target = 0.3 * torch.flip(f[:, 1:2], (2,)).float().contiguous()
    return x, target


# ---- the calls --------------------------------------------------------------------

def prepare(case, seed):
    g = _rng(seed)
    family = case["family"]
    if family == "apply":
        csr = _grid(case, g).csr() if case["matrix"] in ("stencil27", "diffusion3d") else _irregular(case, g)
        A = gk.Matrix(*csr, fmt=case["fmt"])
        x, y = _uniform(A.n_cols, g), _uniform(A.n_rows, g)
        return dict(family=family, A=A, x=x, y=y, adv=case["adv"])
    if family == "setup":
        grid = _grid(case, g)
        return dict(family=family, csr=grid.csr(), x=_uniform(grid.n, g), fmt=case["fmt"], bs=case["bs"])
    if family == "solve":
        grid = _grid(case, g)
        b = grid.apply(_uniform(grid.n, g))
        A = gk.Matrix(*grid.csr(), fmt=case["fmt"])
        P = gk.Precond(A, case["prec"]) if case["prec"] else None
        more = dict(max_iters=20_000, reduction_factor=TOL)
        if case["kind"] == "gmres":
            more = dict(max_iters=case["steps"], reduction_factor=1e-300, krylov_dim=30)
        return dict(family=family, solver=gk.Solver(A, P, case["kind"], **more), b=b)
    if family == "batch":
        grid, ptr = _batch_grid(case, g)
        b = grid.apply(_uniform(grid.n, g))
        return dict(family=family, batch=gk.Batch(ptr.cpu().numpy(), *grid.csr()), b=b, kind=case["kind"])
    if family == "infer":
        x, _ = _network_inputs(case, seed)
        net, _, _ = learned.load(_weights_file(), batch_max=case["batch"])
        return dict(family=family, net=net, x=x, y=torch.empty((case["batch"], 1, 256, 256), device=DEV))
    x, target = _network_inputs(case, seed)
    side = case["side"]
    net = gk.WsNet(side, side, case["batch"], learned.dilations_for(side))
    net.set_params(learned.init_params(seed))
    net.set_loss(case["loss"])
    return dict(family=family, net=net, x=x, target=target)


def run(state):
    family = state["family"]
    if family == "apply":
        if state["adv"]:
            return gk.apply_adv(2.0, state["A"], state["x"], 0.5, state["y"])
        return gk.apply(state["A"], state["x"], state["y"])
    if family == "setup":
        A = gk.Matrix(*state["csr"], fmt=state["fmt"])
        P = gk.Precond(A, state["bs"])
        y, z = torch.empty_like(state["x"]), torch.empty_like(state["x"])
        gk.apply(A, state["x"], y)
        gk.precond_apply(P, y, z)
        return y, z
    if family == "solve":
        x = torch.zeros_like(state["b"])
        st = gk.solve(state["solver"], state["b"], x)
        return x, st.stop_reason
    if family == "batch":
        x = torch.zeros_like(state["b"])
        st = state["batch"].solve(state["b"], x, state["kind"], max_iters=4000, reduction_factor=TOL)
        return x, st["stop_reason"]
    if family == "infer":
        return state["net"].infer_bf16(state["x"], state["y"])
    loss, grads = state["net"].gradients(state["x"], state["target"])
    return loss, grads


# ---- what a pass cannot do without ----------------------------------------------------

def _size(case):
    """Rows and stored entries (expected ones where they are random)."""
    m = case.get("matrix")
    if m == "ragged":
        return case["n"], int(case["n"] * 18)
    if m == "powerlaw":
        cap = min(case["n"], 10_000)
        k = np.arange(1, cap + 1, dtype=np.float64)
        return case["n"], int(case["n"] * (2.0 * (k ** -0.8).sum() / (k ** -1.8).sum() + 1.0))
    shape = [case[a] for a in ("nz", "ny", "nx") if a in case]
    n = math.prod(shape)
    if m == "stencil27":
        return n, math.prod(3 * s - 2 for s in shape)
    return n, n + sum(2 * (n - n // s) for s in shape)


def _iterations(case):
    """About how many iterations a solve to 1e-12 takes, from its matrix's
    condition (CG's count grows with the longest side)."""
    long_side = max(case[a] for a in ("nz", "ny", "nx") if a in case)
    per_side = {"poisson2d": 3.6, "diffusion2d": 3.9, "stencil27": 2.4, "diffusion3d": 4.6, "convdiff": 1.4}
    return max(20, int(per_side[case["matrix"]] * long_side))


def work(case):
    family = case["family"]
    if family == "apply":
        n, nnz = _size(case)
        return {"bytes": 12 * nnz + 4 * n + 16 * n + (8 * n if case["adv"] else 0), "flops": 2 * nnz}
    if family == "setup":
        n, nnz = _size(case)
        bs = case["bs"]
        # the caller's arrays once, the stored operator and the inverse
        # blocks written and read once, the three vectors
        return {"bytes": 12 * nnz + 4 * n + 2 * (12 * nnz + 8 * n * bs) + 24 * n,
                "flops": 2 * nnz + 2 * n * bs * bs + 2 * n * bs}
    if family == "solve":
        n, nnz = _size(case)
        if case["kind"] == "gmres":
            its, basis = case["steps"], 15.5
            # per step the operator and, at least once, the basis so far
            return {"bytes": its * (12 * nnz + 16 * n + 8 * n * basis), "flops": its * (2 * nnz + 8 * n * basis)}
        its = _iterations(case)
        two = 2 if case["kind"] == "bicgstab" else 1
        wide = 4 if case["kind"] == "ir_cg" else 8
        if n * 60 < 1.2e8:  # the whole solve fits in L2: the operator, b and x once
            moved = 12 * nnz + 24 * n
        else:
            moved = its * two * ((wide + 4) * nnz + 9 * wide * n)
        return {"bytes": moved, "flops": its * two * (2 * nnz + 12 * n)}
    if family == "batch":
        sides = np.arange(case["side_lo"], case["side_hi"] + 1, dtype=np.float64)
        n, nnz = (sides ** 2).mean() * case["systems"], (5 * sides ** 2 - 4 * sides).mean() * case["systems"]
        its = 3.0 * sides.mean()
        return {"bytes": 12 * nnz + 28 * n, "flops": its * (2 * nnz + 12 * n)}
    pixels = case["batch"] * case.get("side", 256) ** 2
    macs = 9 * (2 * 32 + 4 * 32 * 32 + 32)
    if family == "infer":
        # features in, four BF16 activations out and in, the output
        return {"bytes": pixels * (2 * 4 + 4 * 2 * 64 + 64 + 64 + 4), "flops": 2 * macs * pixels}
    # forward, data gradients and weight gradients; every activation written
    # and read by the next layer and by the backward pass
    return {"bytes": pixels * 4 * (2 + 5 * 32 * 6 + 4), "flops": 6 * macs * pixels}


# ---- what a pass should return ------------------------------------------------------------

def _csr_apply(csr, x):
    rowptr, col, val = csr
    n = rowptr.numel() - 1
    row = torch.repeat_interleave(torch.arange(n, device=DEV), (rowptr[1:] - rowptr[:-1]).long())
    return torch.zeros(n, device=DEV, dtype=torch.float64).index_add_(0, row, val * x[col.long()])


def _block_solve(grid, bs, r):
    """M^{-1} r for the block-diagonal part M of the operator, blocks of bs
    rows (the last one shorter)."""
    n = grid.n
    pad = -n % bs
    dense = torch.zeros(((n + pad) // bs, bs, bs), device=DEV, dtype=torch.float64)
    rows = torch.arange(n, device=DEV)
    for d, ok, v in zip(grid.delta, grid.ok, grid.values):
        col = rows + d
        inside = ok & (torch.div(col, bs, rounding_mode="floor") == rows // bs)
        at = rows[inside]
        dense[at // bs, at % bs, col[inside] % bs] = v[inside]
    for k in range(pad):
        dense[-1, bs - 1 - k, bs - 1 - k] = 1.0
    rhs = torch.cat([r, torch.zeros(pad, device=DEV, dtype=torch.float64)]).view(-1, bs, 1)
    return torch.linalg.solve(dense, rhs).view(-1)[:n]


def _gmres(grid, b, m, steps):
    """Right-preconditioned (Jacobi) restarted GMRES, `steps` steps in all."""
    inv = 1.0 / grid.diagonal()
    x = torch.zeros_like(b)
    while steps > 0:
        k_max = min(m, steps)
        r = b - grid.apply(x)
        beta = r.norm()
        V, H = [r / beta], np.zeros((k_max + 1, k_max))
        for j in range(k_max):
            w = grid.apply(inv * V[j])
            for _ in range(2):
                for i in range(j + 1):
                    h = torch.dot(V[i], w)
                    H[i, j] += float(h)
                    w = w - h * V[i]
            H[j + 1, j] = float(w.norm())
            V.append(w / H[j + 1, j])
        e = np.zeros(k_max + 1)
        e[0] = float(beta)
        y = np.linalg.lstsq(H, e, rcond=None)[0]
        x = x + inv * sum(float(c) * v for c, v in zip(y, V))
        steps -= k_max
    return x


def _layers(vec):
    ch = learned.CHANNELS
    k, out = 0, []
    for ci, co in zip(ch[:-1], ch[1:]):
        w = vec[k:k + co * ci * 9].view(co, ci, 3, 3)
        k += co * ci * 9
        out.append((w, vec[k:k + co]))
        k += co
    return out


def _forward(layers, x, dilations):
    """The dilated 3 x 3 convolutions with zero padding, tap by tap, ReLU
    after every layer but the last."""
    side = x.shape[-1]
    for l, ((w, bias), d) in enumerate(zip(layers, dilations)):
        p = torch.nn.functional.pad(x, (d, d, d, d))
        y = bias.view(1, -1, 1, 1).expand(x.shape[0], -1, side, side)
        for ky in range(3):
            for kx in range(3):
                tap = p[:, :, ky * d:ky * d + side, kx * d:kx * d + side]
                y = y + torch.einsum("oc,bchw->bohw", w[:, :, ky, kx], tap)
        x = torch.relu(y) if l < len(layers) - 1 else y
    return x


def _energy(e, log_coef):
    """Mean of e (A e), A each sample's 5-point diffusion operator: the sum
    over the faces of face * (difference of e across it)^2."""
    c = torch.exp(log_coef)
    total = 0.0
    for ax in (1, 2):
        n = c.shape[ax]
        lo, hi = c.narrow(ax, 0, n - 1), c.narrow(ax, 1, n - 1)
        de = e.narrow(ax, 1, n - 1) - e.narrow(ax, 0, n - 1)
        total = total + (2.0 * lo * hi / (lo + hi) * de * de).sum()
        for end in (0, n - 1):
            total = total + (c.narrow(ax, end, 1) * e.narrow(ax, end, 1) ** 2).sum()
    return total / e.numel()


def exact(case, seed):
    g = _rng(seed)
    family = case["family"]
    if family == "apply":
        csr = _grid(case, g).csr() if case["matrix"] in ("stencil27", "diffusion3d") else _irregular(case, g)
        n = csr[0].numel() - 1
        x, y = _uniform(n, g), _uniform(n, g)
        ax = _csr_apply(csr, x)
        return 2.0 * ax + 0.5 * y if case["adv"] else ax
    if family == "setup":
        grid = _grid(case, g)
        y = grid.apply(_uniform(grid.n, g))
        return y, _block_solve(grid, case["bs"], y)
    if family == "solve":
        grid = _grid(case, g)
        xs = _uniform(grid.n, g)
        if case["kind"] == "gmres":
            return _gmres(grid, grid.apply(xs), 30, case["steps"]), None
        return xs, None
    if family == "batch":
        grid, _ = _batch_grid(case, g)
        return _uniform(grid.n, g), None
    x, target = _network_inputs(case, seed)
    if family == "infer":
        z = np.load(_weights_file())
        layers = _layers(torch.from_numpy(z["params"]).to(DEV).double())
        dil = [int(d) for d in z["dilations"]]
        return torch.cat([_forward(layers, x[k:k + 4].double(), dil) for k in range(0, x.shape[0], 4)])
    vec = torch.from_numpy(learned.init_params(seed)).to(DEV).double().requires_grad_(True)
    total = 0.0
    grads = torch.zeros_like(vec)
    for k in range(0, x.shape[0], 2):  # two samples at a time: the tape of a whole batch is large
        xb, tb = x[k:k + 2].double(), target[k:k + 2].double()
        e = (_forward(_layers(vec), xb, learned.dilations_for(case["side"])) - tb)[:, 0]
        share = e.shape[0] / x.shape[0]
        loss = share * (_energy(e, xb[:, 0]) if case["loss"] == "energy" else e.square().mean())
        grads += torch.autograd.grad(loss, vec)[0]
        total += float(loss.detach())
    return total, grads.cpu().numpy()
