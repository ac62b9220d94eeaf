"""The work that programs have this package do, as cases that can be timed and compared.

A case names a grid problem (the 5- or 7-point matrices of Section 6.1 of arXiv 1505.04340, constant
or finite-volume coefficients), its box partition, the handle's options and one public call:

  apply   z = M^{-1} r, what a caller's own Krylov method or smoother calls once per iteration
  bsolve  t = B^{-1} f, the subdomain solves alone (block Jacobi on the interiors)
  csolve  y = C^{-1} g, the interface solve alone
  stilde  y = S~^{-1} g, the interface preconditioner alone (a caller's own Schur complement method)
  pcg     a whole solve of A x = b to a tolerance, the usual use
  gmres   a whole solve of a shifted, symmetric indefinite problem

``apply`` and ``stilde`` run with caller-given eigenpairs (``set_lowrank``: vectors kept from an
earlier run), so that a result does not depend on how the setup's Lanczos run rounded; ``pcg`` and
``gmres`` use the vectors that the setup finds.  The mixed handle computes in FP32 and widens its
result to FP64; ``run`` returns it in FP32 again, which loses nothing.
"""
from __future__ import annotations

import functools
import math

import torch

from paper_1505_04340_gb300.slr import SLR

_DEV = "cuda"


def _case(name, call, nx, ny, nz, bx, by, bz, k, precision, nrhs=1, tc="off", fv=0.0, cz=1.0, shift=0.0,
          tol=0.0, iters=0):
    """Grid nx x ny x nz (nz = 1: 2-D) in bx x by x bz boxes; rank k; ``tc`` the tensor-core option of the
    band solve and the low-rank products; ``fv`` = f > 0: finite volumes with cell coefficients log-uniform in
    [1/f, f] (another matrix for each seed), else axis coefficients (1, 1, cz) minus shift I; ``iters``: about
    how many iterations a whole solve takes (for ``work``)."""
    c = dict(call=call, nx=nx, ny=ny, nz=nz, bx=bx, by=by, bz=bz, k=k, precision=precision, nrhs=nrhs, tc=tc,
             fv=fv, cz=cz, shift=shift, tol=tol, iters=iters)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest grid of the tests and examples: launches and latency only
        _case("apply-2d-32-fp64", "apply", 32, 32, 1, 2, 2, 1, 8, "fp64"),
        # the ordinary 3-D model problem, one right-hand side, in either precision
        _case("apply-3d-64-fp64", "apply", 64, 64, 64, 4, 4, 4, 32, "fp64"),
        _case("apply-3d-64-mixed", "apply", 64, 64, 64, 4, 4, 4, 32, "mixed"),
        # a large 2-D field with strongly varying coefficients: long narrow band chains
        _case("apply-2d-fv-1024-mixed", "apply", 1024, 1024, 1, 16, 16, 1, 64, "mixed", fv=1e3),
        # the block workload: 32 right-hand sides on the tensor cores, the largest apply
        _case("apply-3d-96-tf32-r32", "apply", 96, 96, 96, 6, 6, 6, 64, "mixed", nrhs=32, tc="tf32", cz=1e-2),
        # the serving pool: ragged grids, a few columns at a time
        _case("apply-3d-fv-47-mixed-r5", "apply", 47, 47, 47, 4, 4, 4, 32, "mixed", nrhs=5, fv=1e2),
        _case("apply-2d-fv-357-mixed-r8", "apply", 357, 357, 1, 12, 12, 1, 16, "mixed", nrhs=8, fv=1e2),
        # FP64 blocks of an odd width: the two solves that everything else is made of
        _case("bsolve-3d-61-fp64-r11", "bsolve", 61, 61, 61, 4, 4, 4, 0, "fp64", nrhs=11),
        _case("csolve-3d-75-mixed-r16", "csolve", 75, 70, 81, 5, 5, 5, 0, "mixed", nrhs=16),
        # whole solves: the smallest, the block workload, a symmetric indefinite one.  On a cube or a square with
        # constant coefficients the eigenvalues are double and the setup's second copies are rounding's own, so
        # these have varying coefficients or unequal sides.
        _case("pcg-2d-fv-32-fp64", "pcg", 32, 32, 1, 2, 2, 1, 8, "fp64", fv=1e2, tol=1e-8, iters=17),
        _case("pcg-3d-fv-96-tf32-r32", "pcg", 96, 96, 96, 6, 6, 6, 64, "mixed", nrhs=32, tc="tf32", fv=10.0, tol=1e-8,
              iters=28),
        _case("gmres-3d-67-mixed", "gmres", 67, 61, 57, 4, 4, 4, 64, "mixed", shift=0.05, tol=1e-9, iters=24),
    ]


def draw(rng):
    """A case of the same ranges: 2-D sides 32..1024 (whole solves 32..256) in boxes of 16..64, 3-D sides 16..72
    in boxes of 8..18, unequal sides, ranks 8..64, 1..32 right-hand sides."""
    call = rng.choice(["apply"] * 6 + ["bsolve", "csolve", "stilde", "pcg"])
    two_d = rng.random() < 0.4
    if two_d:
        side = int(round(32 * 2.0 ** ((3 if call == "pcg" else 5) * rng.random())))
        box = rng.randint(min(16, side // 2), min(64, side // 2))
        nx, ny, nz = side, max(32, int(side * rng.uniform(0.8, 1.0))), 1
        bx, by, bz = max(2, nx // box), max(2, ny // box), 1
    else:
        side = int(round(16 * 4.5 ** rng.random()))
        box = rng.randint(8, min(18, side // 2))
        nx, ny, nz = side, max(16, int(side * rng.uniform(0.8, 1.0))), max(16, int(side * rng.uniform(0.8, 1.1)))
        bx, by, bz = (max(2, v // box) for v in (nx, ny, nz))
    precision = rng.choice(["fp64", "mixed", "mixed"])
    nrhs = rng.choice([1, 1, int(round(2.0 ** (5 * rng.random())))])
    most = 500_000 if call == "pcg" else 4_000_000       # no dearer than the listed whole solve
    nrhs = max(1, min(nrhs, most // (nx * ny * nz)))
    tc = rng.choice(["off", "tf32"]) if precision == "mixed" and nrhs >= 8 else "off"
    fv = rng.choice([0.0, 1e2])
    if call == "pcg":
        fv, precision, tc = 1e2, "fp64", "off"
    return _case("", call, nx, ny, nz, bx, by, bz, 0 if call in ("bsolve", "csolve") else rng.choice([8, 16, 32, 64]),
                 precision, nrhs=nrhs, tc=tc, fv=fv, tol=1e-8 if call == "pcg" else 0.0,
                 iters=30 if call == "pcg" else 0)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _uniform(seed, stream, *shape):
    g = torch.Generator(device=_DEV).manual_seed(1_000_003 * (seed % (1 << 40)) + stream)
    return torch.rand(*shape, generator=g, dtype=torch.float64, device=_DEV)


@functools.lru_cache(maxsize=4)
def _grid(nx, ny, nz, bx, by, bz):
    """The couplings (one way, axis by axis) and the box of every cell; x is the fastest index."""
    idx = torch.arange(nx * ny * nz, device=_DEV).view(nz, ny, nx)
    pairs = [(idx[:, :, :-1], idx[:, :, 1:]), (idx[:, :-1], idx[:, 1:]), (idx[:-1], idx[1:])]
    pairs = [(a.reshape(-1), b.reshape(-1)) for a, b in pairs]
    x, y, z = (torch.arange(m, device=_DEV) * b // m for m, b in ((nx, bx), (ny, by), (nz, bz)))
    part = (z[:, None, None] * by + y[None, :, None]) * bx + x[None, None, :]
    return pairs, part.reshape(-1)


def _matrix(case, seed):
    """A as sorted CSR on the GPU (int64 indices), and the part of every row."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    n = nx * ny * nz
    pairs, part = _grid(nx, ny, nz, case["bx"], case["by"], case["bz"])
    axes = 3 if nz > 1 else 2
    rows, cols, vals = [], [], []
    if case["fv"]:
        a = case["fv"] ** (2.0 * _uniform(seed, 1, n) - 1.0)
        grid = a.view(nz, ny, nx)
        diag = torch.zeros(n, dtype=torch.float64, device=_DEV)
        for ax in range(axes):
            for end in (0, -1):                      # a boundary face of cell i has 2 a_i
                edge = torch.zeros_like(grid)
                edge.select(2 - ax, end).copy_(2.0 * grid.select(2 - ax, end))
                diag += edge.view(-1)
    else:
        coef = (1.0, 1.0, case["cz"])
        diag = torch.full((n,), 2.0 * sum(coef[:axes]) - case["shift"], dtype=torch.float64, device=_DEV)
    for ax in range(axes):
        i, j = pairs[ax]
        if case["fv"]:
            t = 2.0 * a[i] * a[j] / (a[i] + a[j])
            diag[i] += t                             # an axis couples each cell once to either side
            diag[j] += t
        else:
            t = torch.full((i.numel(),), coef[ax], dtype=torch.float64, device=_DEV)
        rows += [i, j]
        cols += [j, i]
        vals += [-t, -t]
    every = torch.arange(n, device=_DEV)
    rows, cols, vals = (torch.cat(v) for v in (rows + [every], cols + [every], vals + [diag]))
    order = torch.argsort(rows * n + cols)
    rows, cols, vals = rows[order], cols[order], vals[order]
    ptr = torch.zeros(n + 1, dtype=torch.int64, device=_DEV)
    ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return ptr, rows, cols, vals, part


def _csr(ptr, cols, vals):
    n = ptr.numel() - 1
    return torch.sparse_csr_tensor(ptr, cols, vals, size=(n, n), check_invariants=False)


class _Split:
    """A in the DD order (Eq. 2.2: interiors part by part, then interfaces part by part)."""

    def __init__(self, ptr, rows, cols, vals, part):
        n = ptr.numel() - 1
        face = torch.zeros(n, dtype=torch.int64, device=_DEV)
        face[rows[part[rows] != part[cols]]] = 1
        self.perm = torch.argsort(face * (int(part.max()) + 1) + part, stable=True)
        self.n, self.s = n, int(face.sum())
        self.ni = n - self.s
        place = torch.empty_like(self.perm)
        place[self.perm] = torch.arange(n, device=_DEV)
        r, c = place[rows], place[cols]
        order = torch.argsort(r * n + c)
        r, c, v = r[order], c[order], vals[order]
        new = torch.zeros(n + 1, dtype=torch.int64, device=_DEV)
        new[1:] = torch.cumsum(torch.bincount(r, minlength=n), 0)
        self.a = _csr(new, c, v)
        self.diag = v[r == c]

    def mul(self, lo, hi, x, to_lo, to_hi):
        """Rows to_lo .. to_hi of A times x in positions lo .. hi."""
        full = torch.zeros(self.n, x.shape[1], dtype=torch.float64, device=_DEV)
        full[lo:hi] = x
        return (self.a @ full)[to_lo:to_hi]

    def c(self, y):
        return self.mul(self.ni, self.n, y, self.ni, self.n)

    def b(self, u):
        return self.mul(0, self.ni, u, 0, self.ni)

    def solve(self, op, diag, f):
        """Conjugate gradients with the diagonal, in 64 bits, to where rounding stops it."""
        d = (1.0 / diag)[:, None]
        x, r = torch.zeros_like(f), f.clone()
        z = d * r
        p, rz = z.clone(), (r * z).sum(0)
        goal = 1e-14 * f.norm(dim=0)
        for it in range(6000):
            q = op(p)
            alpha = rz / (p * q).sum(0).clamp_min(1e-300)
            x += alpha * p
            r -= alpha * q
            z = d * r
            rz, old = (r * z).sum(0), rz
            p = z + (rz / old.clamp_min(1e-300)) * p
            if it % 16 == 15 and bool((r.norm(dim=0) <= goal).all()):
                break
        return x

    def bsolve(self, f):
        return self.solve(self.b, self.diag[: self.ni], f)

    def csolve(self, g):
        return self.solve(self.c, self.diag[self.ni:], g)


def _lowrank(case, seed, split):
    """k C-orthonormal vectors, their eigenvalue estimates (falling towards theta) and theta."""
    k = min(case["k"], split.s)
    z = 2.0 * _uniform(seed, 2, split.s, k) - 1.0
    factor = torch.linalg.cholesky((z.t() @ split.c(z)).cpu())      # k x k, on the host
    z = z @ torch.linalg.inv(factor).t().to(_DEV)
    lam = 0.6 + 0.35 * (1.0 - torch.arange(k, dtype=torch.float64) / k) ** 2
    return z, lam.to(_DEV), 0.6


def _rhs(case, seed, rows):
    """Uniform in [-1, 1), column by column as the library takes a block: rows x nrhs."""
    return (2.0 * _uniform(seed, 3, case["nrhs"], rows) - 1.0).t()


class _State:
    def __init__(self, case, handle, x):
        self.case, self.handle, self.x = case, handle, x


def prepare(case, seed):
    ptr, rows, cols, vals, part = _matrix(case, seed)
    call, r = case["call"], case["nrhs"]
    given = call in ("apply", "stilde")
    # bsolve and csolve use the factors only, so their handle has no vectors
    handle = SLR(ptr.int().cpu().numpy(), cols.int().cpu().numpy(), vals.cpu().numpy(), part.int().cpu().numpy(),
                 case["bx"] * case["by"] * case["bz"], k=0 if given else case["k"], precision=case["precision"],
                 nrhs_max=r, flexible_cg=case["precision"] == "mixed", indefinite=case["shift"] > 0,
                 u_dtype="fp32" if case["tc"] == "off" else case["tc"], band_mma=case["tc"])
    if given:
        z, lam, theta = _lowrank(case, seed, _Split(ptr, rows, cols, vals, part))
        handle.set_lowrank(z.cpu().numpy(), lam.cpu().numpy(), theta)
    if call in ("pcg", "gmres"):
        x = (_csr(ptr, cols, vals) @ _rhs(case, seed, ptr.numel() - 1)).t().contiguous().t()
    else:
        x = _rhs(case, seed, {"apply": handle.n, "bsolve": handle.n_interior}.get(call, handle.s))
    return _State(case, handle, x[:, 0].contiguous() if r == 1 else x)


def run(state):
    case, h = state.case, state.handle
    call = case["call"]
    if call in ("pcg", "gmres"):
        x, iterations, _, _ = (h.pcg if call == "pcg" else h.gmres)(state.x, tol=case["tol"])
        return {"x": x, "iterations": iterations}
    y = {"apply": h.apply, "bsolve": h.bsolve, "csolve": h.csolve, "stilde": h.stilde_solve}[call](state.x)
    return y.float() if case["precision"] == "mixed" else y


# ---------------------------------------------------------------------------
# what the calls cannot do without, and what they return in 64 bits
# ---------------------------------------------------------------------------

def _lengths(n, b):
    """(length, interior length) of the b boxes along an axis of n cells (box of cell i: i b // n)."""
    first = [-(-i * n // b) for i in range(b + 1)]
    return [(first[i + 1] - first[i], first[i + 1] - first[i] - (i > 0) - (i + 1 < b)) for i in range(b)]


def work(case):
    nx, ny, nz, r = case["nx"], case["ny"], case["nz"], case["nrhs"]
    n, two_d = nx * ny * nz, nz == 1
    xs, ys, zs = (_lengths(m, b) for m, b in ((nx, case["bx"]), (ny, case["by"]), (nz, case["bz"])))
    inner = band = 0
    for _, a in xs:
        for _, b in ys:
            for _, c in zs:
                inner += a * b * c
                band += a * b * c * (a if two_d else a * b)     # rows times half-bandwidth
    s = n - inner
    # a nested-dissection factor of C: about 3.5 s^(4/3) entries on the 3-D grids, s log2 s on the 2-D ones
    cfac = s * math.log2(s + 2) if two_d else 3.5 * s ** (4.0 / 3.0)
    cfac = min(cfac, s * (s + 1) / 2.0)
    w = 8 if case["precision"] == "fp64" else 4
    call, k = case["call"], min(case["k"], s)
    # a factor is read once forward and once backward; a vector in and a vector out
    bsolve = (2.0 * band * w, 4.0 * band * r)
    csolve = (2.0 * cfac * w, 4.0 * cfac * r)
    stilde = (csolve[0] + 2.0 * s * k * w, csolve[1] + 4.0 * s * k * r)
    apply = (2 * bsolve[0] + stilde[0] + 12.0 * s * w, 2 * bsolve[1] + stilde[1] + 12.0 * s * r)
    if call in ("pcg", "gmres"):
        # per iteration a product with A and, at the least, x, r and p read and written
        its, nnz = case["iters"], (5.0 if two_d else 7.0) * n
        return {"bytes": its * (apply[0] + 12.0 * nnz + 48.0 * n * r) + 16.0 * n * r,
                "flops": its * (apply[1] + 2.0 * nnz * r + 10.0 * n * r)}
    got, rows = {"apply": (apply, n), "bsolve": (bsolve, inner), "csolve": (csolve, s), "stilde": (stilde, s)}[call]
    return {"bytes": got[0] + rows * r * (8.0 + w), "flops": got[1]}


def exact(case, seed):
    """The same results by conjugate gradients on B and C in 64 bits; for a whole solve the x that b was made of."""
    ptr, rows, cols, vals, part = _matrix(case, seed)
    call = case["call"]
    if call in ("pcg", "gmres"):
        x = _rhs(case, seed, ptr.numel() - 1)
        return {"x": x[:, 0] if case["nrhs"] == 1 else x, "iterations": None}
    m = _Split(ptr, rows, cols, vals, part)
    x = _rhs(case, seed, {"apply": m.n, "bsolve": m.ni}.get(call, m.s))
    if call == "bsolve":
        y = m.bsolve(x)
    elif call == "csolve":
        y = m.csolve(x)
    else:
        z, lam, theta = _lowrank(case, seed, m)
        d = (1.0 / (1.0 - lam) - 1.0 / (1.0 - theta))[:, None]

        def stilde(g):                     # Proposition 4.3: C^{-1} g / (1 - theta) + Z (d o Z^T g)
            return m.csolve(g) / (1.0 - theta) + z @ (d * (z.t() @ g))

        if call == "stilde":
            y = stilde(x)
        else:                              # Eq. 4.1 with the block LU of Eq. 2.4
            t = m.bsolve(x[: m.ni])
            v = stilde(x[m.ni:] - m.mul(0, m.ni, t, m.ni, m.n))
            y = torch.cat([t - m.bsolve(m.mul(m.ni, m.n, v, 0, m.ni)), v])
    return y[:, 0] if case["nrhs"] == 1 else y
