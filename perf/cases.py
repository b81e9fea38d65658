"""Performance cases of the block ILU(0) + FGMRES library.

Each case is one call (or the few calls that belong together) that a flow solver makes through
the package's public functions, on block systems shaped like cell-centred finite-volume Jacobians
of a triangulated quad grid (at most three face neighbours per cell, 4x4 blocks), with the values
and solver settings of the repository's own workloads.  `listed()` holds the fixed cases, `draw()`
gives more of the same kinds with sizes, aspect ratios, CFL numbers, precisions and modes drawn
from the ranges the repository's generators and tests use.

Meshes are fixed per size (a user's mesh does not change between steps); block values and
right-hand sides come from the seed.  `exact()` is the same method in FP64 torch operations.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import abilu_inputs as gen
from paper_1912_00539_gb300 import abilu as ab

DEV = "cuda"


# ------------------------------------------------------------------ the cases
def _solve(name, nx, ny, dtype, mode, build, sweeps, cfl, order="rcm", wall=1.0, restart=30,
           rtol=1e-6, kind="solve"):
    return dict(name=name, kind=kind, nx=nx, ny=ny, dtype=dtype, mode=mode, build=build,
                sweeps=sweeps, cfl=cfl, order=order, wall=wall, restart=restart, rtol=rtol)


def listed():
    return [
        # the smallest workload of the repository: one implicit step on a coarse grid, where
        # launches and latency count
        _solve("solve_64x64_f32_async", 64, 64, "f32", "async", 4, 3, 100.0),
        # the benchmark's own solve: 524,288 cells, A larger than L2
        _solve("solve_512x512_f32_async", 512, 512, "f32", "async", 6, 4, 1000.0),
        # boundary-layer grid: strong wall-normal coupling, more sweeps and more Krylov steps
        _solve("solve_viscous_1024x256_f32_async", 1024, 256, "f32", "async", 8, 6, 1e4, wall=100.0,
               restart=50),
        # the plain FP64 method with synchronous (reproducible) sweeps, an odd-sized grid
        _solve("solve_301x217_f64_sync", 301, 217, "f64", "sync", 4, 3, 100.0),
        # one step of pseudo-time marching: shift the Jacobian's diagonal, then a loose solve with
        # one build sweep (the continuation driver's defaults)
        _solve("pseudotime_256x256_f32_sync", 256, 256, "f32", "sync", 1, 3, 10.0, rtol=0.1,
               kind="pseudotime"),
        # factorising only, factors read back in FP64 (preconditioner reused by the caller's own
        # Krylov solver, or diagnosed)
        dict(name="build_512x512_f32_sync", kind="build", nx=512, ny=512, dtype="f32", build=6,
             cfl=1000.0),
        # preconditioner application from a caller's own Krylov solver, narrow factors, ragged size
        dict(name="apply_331x197_bf16_sync", kind="apply", nx=331, ny=197, dtype="bf16", build=4,
             sweeps=3, cfl=100.0),
        # the FP64 block product by itself (residual evaluations of a flow solver)
        dict(name="spmv_512x512_f64", kind="spmv", nx=512, ny=512, cfl=1000.0),
        # 64 uneven systems (2k-200k cells) set, solved in shared launches and read back
        dict(name="batch_64_f32_async", kind="batch", systems=64, lo=2000, hi=200000, spec=4,
             dtype="f32", mode="async", build=4, sweeps=3),
        # one step of continuous batching: the value updates of four admitted requests
        dict(name="server_step_4_f32_async", kind="server", systems=4, lo=4000, hi=120000, spec=11,
             dtype="f32", mode="async", build=4, sweeps=3),
        # FGMRES with the multigrid V-cycle (block ILU smoothing, set-up inside the solve)
        dict(name="multigrid_512x512_f32_sync", kind="mg", nx=512, ny=512, dtype="f32", build=4,
             sweeps=2, cfl=1000.0),
        # threshold factorisation (two fill-and-drop steps), its pattern and factors
        dict(name="parilut_192x160_f32", kind="parilut", nx=192, ny=160, dtype="f32", fill=1.5,
             iters=2, build=2, cfl=1000.0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _grid(rng, lo, hi):
    """Quads per side: cells log-uniform in [lo, hi], aspect ratio log-uniform in [1/8, 8]."""
    cells, ar = _log(rng, lo, hi), _log(rng, 0.125, 8.0)
    ny = max(2, round(math.sqrt(cells / 2.0 / ar)))
    return max(2, round(cells / 2.0 / ny)), ny


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "pseudotime", "build", "apply", "spmv", "batch",
                       "server", "mg", "parilut"])
    cfl = _log(rng, 10.0, 1e4)
    dtype = rng.choice(["f32", "f32", "bf16", "f64"])
    if kind in ("solve", "pseudotime"):
        nx, ny = _grid(rng, 2000, 520000)
        if kind == "pseudotime":
            c = _solve("", nx, ny, dtype, "sync", 1, 3, cfl, rtol=0.1, kind=kind)
        elif rng.random() < 0.3:
            c = _solve("", nx, ny, "f32", "async", 8, 6, cfl, rng.choice(["rcm", "line"]), 100.0, 50)
        else:
            c = _solve("", nx, ny, dtype, rng.choice(["async", "sync"]), rng.choice([4, 5, 6]),
                       rng.choice([3, 4]), cfl)
        del c["name"]
        return c
    if kind in ("batch", "server"):
        top = 48 if kind == "batch" else 6
        return dict(kind=kind, systems=rng.randint(2, top), lo=2000, hi=120000,
                    spec=rng.randrange(1 << 20), dtype=rng.choice(["f32", "f32", "bf16"]),
                    mode="async", build=4, sweeps=rng.choice([2, 3]))
    hi = {"parilut": 61000, "mg": 520000}.get(kind, 520000)
    nx, ny = _grid(rng, 4000 if kind in ("mg", "parilut") else 2000, hi)
    c = dict(kind=kind, nx=nx, ny=ny, cfl=cfl)
    if kind == "build":
        c.update(dtype=dtype, build=rng.choice([3, 4, 6]))
    elif kind == "apply":
        c.update(dtype=dtype, build=4, sweeps=rng.choice([2, 3, 4, 6]))
    elif kind == "mg":
        c.update(dtype="f32", build=4, sweeps=2)
    elif kind == "parilut":
        c.update(dtype=rng.choice(["f32", "f64"]), fill=rng.choice([1.5, 2.0]), iters=rng.choice([1, 2]),
                 build=2)
    return c


# ------------------------------------------------------------------ meshes and values
@functools.lru_cache(maxsize=160)
def _mesh(nx, ny, order="rcm"):
    """The block pattern of the nx x ny triangulated grid in the given ordering, on the GPU:
    rowptr, colind (int32), the row of every block, each row's diagonal block, a table of each
    row's off-diagonal blocks (padded with nnzb) and which blocks couple wall-normal neighbours."""
    grid = gen.tri_quad_grid(nx, ny, 1000003 * nx + ny)
    n = grid.ncells
    e = torch.from_numpy(grid.edges).to(DEV)
    diag = torch.arange(n, device=DEV)
    i = torch.cat([e[:, 0], e[:, 1], diag])
    j = torch.cat([e[:, 1], e[:, 0], diag])

    def csr(i, j):
        key = torch.sort(i * n + j)[0]
        rows, cols = key // n, key % n
        return rows, cols, torch.cat([key.new_zeros(1), torch.bincount(rows, minlength=n).cumsum(0)])

    if order == "rcm":
        rows, cols, ptr = csr(i, j)
        perm = torch.from_numpy(ab.order(ptr.int().cpu().numpy(), cols.int().cpu().numpy(), "rcm")[0])
    else:   # whole wall-normal columns as lines
        perm = torch.from_numpy(gen.line_order(nx, ny))
    perm = perm.long().to(DEV)
    new = torch.empty_like(perm)
    new[perm] = diag
    rows, cols, ptr = csr(new[i], new[j])
    nnzb = rows.numel()
    off = torch.nonzero(rows != cols).squeeze(1)
    pos = torch.nonzero(rows == cols).squeeze(1)
    slot = torch.arange(nnzb, device=DEV) - ptr[rows]
    table = torch.full((n, int((ptr[1:] - ptr[:-1]).max())), nnzb, device=DEV)
    table[rows[off], slot[off]] = off
    quad = perm // 2
    wall = (quad[rows] - quad[cols]).abs() != 1
    return dict(n=n, nnzb=nnzb, rowptr=ptr.int(), colind=cols.int(), rows=rows, diag=pos, table=table,
                wall=wall & (rows != cols))


def _values(m, cfl, seed, wall=1.0):
    """Block values and right-hand side: off-diagonal blocks 0.5 N(0,1) (times `wall` between
    wall-normal neighbours), diagonal 1/CFL + the absolute sum of the row's off-diagonal entries."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    A = torch.randn((m["nnzb"], 4, 4), dtype=torch.float64, device=DEV, generator=g).mul_(0.5)
    if wall != 1.0:
        A[m["wall"]] *= wall
    s = torch.zeros((m["nnzb"] + 1, 4), dtype=torch.float64, device=DEV)
    s[:-1] = A.abs().sum(2)
    A[m["diag"]] = torch.diag_embed(1.0 / cfl + s[m["table"]].sum(1))
    b = torch.randn((m["n"], 4), dtype=torch.float64, device=DEV, generator=g)
    return A, b


def _members(case):
    """(nx, ny, cfl) of the systems of a batch or a server step."""
    return [(s["nx"], s["ny"], s["cfl"]) for s in gen.batch_specs(case["systems"], case["spec"], case["lo"], case["hi"])]


def _pseudo_shift(m, A, cfl):
    """Pseudo-time shift per unknown: the mean diagonal entry of the cell's block over CFL."""
    d = A[m["diag"]].diagonal(dim1=1, dim2=2).mean(1, keepdim=True) / cfl
    return d.expand(-1, 4).contiguous()


# ------------------------------------------------------------------ what is measured
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("batch", "server"):
        mem = [(_mesh(nx, ny), cfl) for nx, ny, cfl in _members(case)]
        vals = [_values(m, cfl, seed + 7919 * k) for k, (m, cfl) in enumerate(mem)]
        off = np.cumsum([0] + [m["n"] for m, _ in mem])
        x = torch.zeros((int(off[-1]), 4), dtype=torch.float64, device=DEV)
        st = dict(case=case, vals=vals, x=x, xs=[x[off[k]:off[k + 1]] for k in range(len(mem))],
                  opts=dict(build_sweeps=case["build"], apply_sweeps_lower=case["sweeps"],
                            apply_sweeps_upper=case["sweeps"], mode=case["mode"]))
        if kind == "batch":
            st["batch"] = ab.Batch([(m["rowptr"], m["colind"]) for m, _ in mem], dtype=case["dtype"])
        else:
            rows = sum(-(-m["n"] // 64) * 64 for m, _ in mem)
            blocks = sum(m["nnzb"] + 64 for m, _ in mem)
            st["server"] = ab.NativeServer(rows, blocks, len(mem), case["dtype"])
            st["ids"] = [st["server"].add(m["rowptr"], m["colind"]) for m, _ in mem]
        return st
    m = _mesh(case["nx"], case["ny"], case.get("order", "rcm"))
    A, b = _values(m, case["cfl"], seed, case.get("wall", 1.0))
    st = dict(case=case, A=A, b=b, x=torch.zeros_like(b), pat=ab.Pattern(m["rowptr"], m["colind"]))
    if kind in ("solve", "pseudotime", "build", "apply"):
        st["fac"] = ab.Factors(st["pat"], case["dtype"])
    if kind == "pseudotime":
        st["shift"], st["A_tau"] = _pseudo_shift(m, A, case["cfl"]), torch.empty_like(A)
    if kind == "apply":
        st["fac"].build(A, case["build"], mode="sync")
    if kind == "mg":
        st["mg"] = ab.Multigrid(st["pat"], A, factor_dtype=case["dtype"], build_sweeps=case["build"],
                                apply_sweeps_lower=case["sweeps"], apply_sweeps_upper=case["sweeps"])
    return st


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind in ("solve", "pseudotime"):
        A = state["A"]
        if kind == "pseudotime":
            A = state["A_tau"]
            ab.add_block_diagonal(state["pat"], state["A"], A, state["shift"])
        ab.fgmres_solve(state["pat"], A, state["fac"], state["b"], state["x"], restart=c["restart"],
                        rtol=c["rtol"], build_sweeps=c["build"], apply_sweeps_lower=c["sweeps"],
                        apply_sweeps_upper=c["sweeps"], mode=c["mode"], zero_guess=True)
        return state["x"]
    if kind == "build":
        state["fac"].build(state["A"], c["build"], mode="sync")
        return state["fac"].export()
    if kind == "apply":
        state["fac"].apply(state["b"], state["x"], c["sweeps"], c["sweeps"], mode="sync")
        return state["x"]
    if kind == "spmv":
        ab.bsr_spmv(state["pat"], state["A"], state["b"], state["x"])
        return state["x"]
    if kind == "batch":
        for k, (A, b) in enumerate(state["vals"]):
            state["batch"].set_system(k, A, b)
        state["batch"].solve(**state["opts"])
        for k, x in enumerate(state["xs"]):
            state["batch"].solution(k, x)
        return state["x"]
    if kind == "server":
        state["server"].step(state["ids"], [A for A, _ in state["vals"]], [b for _, b in state["vals"]],
                             state["xs"], **state["opts"])
        return state["x"]
    if kind == "mg":
        ab.fgmres_solve_mg(state["mg"], state["A"], state["b"], state["x"], zero_guess=True)
        return state["x"]
    pat, fac = ab.parilut(state["pat"], state["A"], fill=c["fill"], iters=c["iters"], sweeps=c["build"],
                          dtype=c["dtype"])
    return [*pat.arrays(), *fac.export()]


def work(case):
    """Matrix (FP64 blocks, column indices, row pointers) and input vectors read once, results
    written once; two flops per entry of one product with A."""
    kind = case["kind"]
    sizes = _members(case) if kind in ("batch", "server") else [(case["nx"], case["ny"], 0)]
    n = sum(2 * nx * ny for nx, ny, _ in sizes)
    nnzb = sum(2 * nx * ny + 2 * (3 * nx * ny - nx - ny) for nx, ny, _ in sizes)
    size = {"f64": 8, "f32": 4, "bf16": 2}[case.get("dtype", "f64")]
    matrix, vec = 132 * nnzb + 4 * (n + 1), 32 * n
    if kind == "build":
        return dict(bytes=matrix + 128 * (nnzb + n), flops=32 * nnzb)
    if kind == "apply":
        return dict(bytes=(16 * size + 4) * nnzb + 4 * (n + 1) + 2 * vec, flops=32 * nnzb)
    if kind == "parilut":
        kept = n + int(case["fill"] * (nnzb - n))
        return dict(bytes=matrix + 132 * kept + 128 * n, flops=32 * kept)
    return dict(bytes=matrix + 2 * vec + (vec if kind == "pseudotime" else 0), flops=32 * nnzb)


def tolerance(case):
    """About four times the error against `exact` that was measured (spmv 1.5e-16; FP32 factors
    4e-8, BF16 ones 1.8e-3; solutions at a relative residual of 1e-6: up to 8e-7)."""
    kind, dtype = case["kind"], case.get("dtype", "f64")
    if kind == "spmv":
        return {"rel": 1e-15}
    if kind in ("build", "apply", "parilut"):
        return {"rel": {"f64": 1e-14, "f32": 5e-7, "bf16": 8e-3}[dtype]}
    if kind == "pseudotime":
        return {"rel": {"f64": 1e-13, "f32": 1e-6, "bf16": 8e-3}[dtype]}
    return {"rel": 4e-6}


# ------------------------------------------------------------------ FP64 statement of the method
def _inv(D):
    return torch.linalg.inv(D)


class _Ref:
    """Block ILU(0) sweeps, triangular sweeps and FGMRES of one system in FP64 torch."""

    def __init__(self, rows, cols, n, A):
        self.rows, self.cols, self.n, self.A = rows, cols, n, A
        self.key = rows * n + cols
        self.ptr = torch.cat([rows.new_zeros(1), torch.bincount(rows, minlength=n).cumsum(0)])
        self.d = torch.nonzero(rows == cols).squeeze(1)
        self.l = torch.nonzero(rows > cols).squeeze(1)
        self.u = torch.nonzero(rows < cols).squeeze(1)
        self.X, self.D = A.clone(), _inv(A[self.d])

    def fill_pairs(self, start):
        """For every L block (i,k), the blocks of row k from its diagonal + start on."""
        k = self.cols[self.l]
        first = self.d[k] + start
        cnt = self.ptr[k + 1] - first
        lp = torch.repeat_interleave(self.l, cnt)
        up = torch.arange(lp.numel(), device=lp.device) - torch.repeat_interleave(cnt.cumsum(0) - cnt, cnt)
        return lp, up + torch.repeat_interleave(first, cnt)

    def pairs(self):
        lp, up = self.fill_pairs(1)
        want = self.rows[lp] * self.n + self.cols[up]
        p = torch.searchsorted(self.key, want).clamp_(max=self.key.numel() - 1)
        hit = self.key[p] == want
        return p[hit], lp[hit], up[hit]

    def sweeps(self, count):
        p, lp, up = self.pairs()
        const = torch.ones_like(self.rows, dtype=torch.bool)
        const[p] = False
        const &= self.rows < self.cols
        self.X[const] = self.A[const]
        for _ in range(count):
            S = self.A.clone().index_add_(0, p, self.X[lp] @ self.X[up], alpha=-1.0)
            D = _inv(S[self.d])
            S[self.l] = S[self.l] @ self.D[self.cols[self.l]]
            self.X, self.D = S, D
        return self

    def part(self, which, v):
        w = (self.X[which] @ v[self.cols[which]].unsqueeze(2)).squeeze(2)
        return torch.zeros_like(v).index_add_(0, self.rows[which], w)

    def apply(self, r, nl, nu):
        y = r
        for _ in range(nl - 1):
            y = r - self.part(self.l, y)
        x = (self.D @ y.unsqueeze(2)).squeeze(2)
        for _ in range(nu - 1):
            x = (self.D @ (y - self.part(self.u, x)).unsqueeze(2)).squeeze(2)
        return x

    def product(self, v):
        w = (self.A @ v[self.cols].unsqueeze(2)).squeeze(2)
        return torch.zeros_like(v).index_add_(0, self.rows, w)

    def fgmres(self, b, nl, nu, rtol, restart, most=600):
        x, bn, its = torch.zeros_like(b), float(b.norm()), 0
        while its < most:
            r = b - self.product(x) if its else b
            beta = float(r.norm())
            if beta <= rtol * bn:
                return x
            V, Z, H = [r / beta], [], np.zeros((restart + 1, restart))
            for j in range(restart):
                Z.append(self.apply(V[j], nl, nu))
                w = self.product(Z[j])
                for _ in range(2):
                    for k in range(j + 1):
                        h = float((V[k] * w).sum())
                        H[k, j] += h
                        w = w - h * V[k]
                H[j + 1, j] = float(w.norm())
                e1 = np.zeros(j + 2)
                e1[0] = beta
                y = np.linalg.lstsq(H[:j + 2, :j + 1], e1, rcond=None)[0]
                its += 1
                if np.linalg.norm(e1 - H[:j + 2, :j + 1] @ y) <= rtol * bn or H[j + 1, j] == 0.0:
                    break
                V.append(w / H[j + 1, j])
            for k in range(len(y)):
                x = x + y[k] * Z[k]
        return None

    def solution(self, b):
        """A^-1 b to about FP64 accuracy (None if it does not converge)."""
        return self.sweeps(6).fgmres(b, 4, 4, 2e-14, 40)


def _ref(m, A):
    return _Ref(m["rows"], m["colind"].long(), m["n"], A)


def _parilut(R, fill, iters, sweeps):
    bl, bu = int(fill * R.l.numel()), int(fill * R.u.numel())
    A0, key0 = R.A, R.key
    R.sweeps(sweeps)

    def moved(key, old_key, old):
        out = torch.zeros((key.numel(), 4, 4), dtype=torch.float64, device=key.device)
        p = torch.searchsorted(key, old_key).clamp_(max=key.numel() - 1)
        hit = key[p] == old_key
        out[p[hit]] = old[hit]
        return out

    def on(key):
        new = _Ref(key // R.n, key % R.n, R.n, moved(key, key0, A0))
        new.X, new.D = moved(key, R.key, R.X), R.D
        return new.sweeps(sweeps)

    for _ in range(iters):
        lp, up = R.fill_pairs(0)
        R = on(torch.unique(torch.cat([R.key, R.rows[lp] * R.n + R.cols[up]])))
        norm = (R.X * R.X).sum((1, 2))
        keep = torch.zeros_like(R.rows, dtype=torch.bool)
        keep[R.d] = True
        for which, budget in ((R.l, bl), (R.u, bu)):
            w = norm[which]
            cut = torch.sort(w, descending=True)[0][budget] if w.numel() > budget else -1.0
            keep[which] = w > cut
        R = on(R.key[keep])
    return R


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "server"):
        xs = []
        for k, (nx, ny, cfl) in enumerate(_members(case)):
            m = _mesh(nx, ny)
            A, b = _values(m, cfl, seed + 7919 * k)
            x = _ref(m, A).solution(b)
            if x is None:
                return None
            xs.append(x)
        return torch.cat(xs)
    m = _mesh(case["nx"], case["ny"], case.get("order", "rcm"))
    A, b = _values(m, case["cfl"], seed, case.get("wall", 1.0))
    if kind == "pseudotime":
        A_tau = A.clone()
        A_tau[m["diag"]] += torch.diag_embed(_pseudo_shift(m, A, case["cfl"]))
        return _ref(m, A_tau).sweeps(case["build"]).fgmres(b, case["sweeps"], case["sweeps"],
                                                           case["rtol"], case["restart"])
    R = _ref(m, A)
    if kind in ("solve", "mg"):
        return R.solution(b)
    if kind == "spmv":
        return R.product(b)
    if kind == "build":
        R.sweeps(case["build"])
        return [R.X, R.D]
    if kind == "apply":
        return R.sweeps(case["build"]).apply(b, case["sweeps"], case["sweeps"])
    P = _parilut(R, case["fill"], case["iters"], case["build"])
    return [P.ptr.int(), P.cols.int(), P.X, P.D]
