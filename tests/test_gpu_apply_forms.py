"""Forms of the preconditioner application chosen by the pattern's size and rows."""
import numpy as np
import pytest

import abilu_inputs as gen


def _check(rowptr, colind, vals, dtype, counts, modes=("sync",)):
    """Applications on the exported factors against the oracle's FP64 sweeps
    with them (a few dozen FP32 roundings of diagonally dominant sums), and
    the right-hand side rounded as torch rounds it."""
    import torch
    import oracle
    import paper_1912_00539_gb300.abilu as ab
    n = len(rowptr) - 1
    pat = ab.Pattern(torch.from_numpy(rowptr).cuda(), torch.from_numpy(colind).cuda())
    fac = ab.Factors(pat, dtype)
    fac.build(torch.from_numpy(vals).cuda(), 3, mode="sync")
    X, D = (t.cpu().numpy() for t in fac.export())
    r = np.random.default_rng(n).standard_normal((n, 4))
    rt = torch.from_numpy(r).cuda()
    z, z32 = torch.empty_like(rt), torch.empty_like(rt)
    for nl, nu in counts:
        fac.apply(rt, z, nl, nu, mode="sync")
        fac.apply(rt.float().double(), z32, nl, nu, mode="sync")
        assert torch.equal(z, z32)
        zo = oracle.apply(rowptr, colind, X, D, r, nl, nu)
        assert np.abs(z.cpu().numpy() - zo).max() < 1e-5 * np.abs(zo).max()
    if "async" in modes:   # both reach the triangular solves
        fac.apply(rt, z, 80, 80, mode="async")
        ys = oracle.lower_solve(rowptr, colind, X, r)
        zo = oracle.upper_solve(rowptr, colind, X, D, ys)
        assert np.abs(z.cpu().numpy() - zo).max() < 1e-5 * np.abs(zo).max()


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("nx,ny", [(223, 224), (223, 225)])
def test_rounding_in_the_first_sweep_and_in_a_pass(nx, ny, dtype):
    """Both sides of 150,000 L blocks, where the right-hand side of a synchronous
    application is rounded by a pass of its own; one lower update, which needs
    none."""
    s = gen.small_system(nx, ny, seed=2)
    _check(s.rowptr, s.colind, s.vals, dtype, ((2, 1), (3, 3), (1, 2)))


def _band(n, lower, upper, seed):
    """Row i: up to `lower` blocks left of the diagonal, `upper` right of it, at
    distances 1, 3, 6, 10, ..., diagonally dominant."""
    rng = np.random.default_rng(seed)
    rowptr, colind = [0], []
    dist = np.cumsum(np.arange(1, max(lower, upper) + 1))
    for i in range(n):
        js = [i - d for d in dist[:lower][::-1] if i >= d] + [i] + [i + d for d in dist[:upper] if i + d < n]
        colind += js
        rowptr.append(len(colind))
    rowptr, colind = np.array(rowptr, np.int32), np.array(colind, np.int32)
    A = 0.5 * rng.standard_normal((len(colind), 4, 4))
    rows = np.repeat(np.arange(n), np.diff(rowptr))
    s = np.zeros((n, 4))
    np.add.at(s, rows, np.abs(A).sum(axis=2))
    d = np.flatnonzero(colind == rows)
    A[d] += np.einsum("nq,qk->nqk", s + 0.5, np.eye(4))
    return rowptr, colind, A


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n,lower,upper", [(2, 1, 1), (700, 2, 2), (700, 3, 3), (1000, 9, 9), (1000, 9, 1), (1000, 1, 9),
                                           (20000, 4, 3)])
def test_long_rows(n, lower, upper, dtype):
    """Chunks of 64 rows with more factor blocks than a stage holds, on both sides,
    one or none (the sweeps without stages), synchronous and in place."""
    _check(*_band(n, lower, upper, n + lower), dtype, ((2, 2), (1, 3), (4, 1), (4, 4)), modes=("sync", "async"))


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_long_rows_in_fgmres(dtype):
    """FGMRES hands over the FP32 right-hand side and the start of the sweeps; at
    most two steps more than the FP64 oracle with synchronous sweeps, and a true
    residual within the tolerance."""
    import torch
    import oracle
    import paper_1912_00539_gb300.abilu as ab
    rowptr, colind, A = _band(3000, 9, 9, 4)
    b = np.random.default_rng(5).standard_normal((3000, 4))
    Xo, Do, _ = oracle.bilu_sync(rowptr, colind, A, 3)
    xo, ro = oracle.fgmres(rowptr, colind, A, Xo, Do, b, 3, 3, restart=30, rtol=1e-6)
    pat = ab.Pattern(torch.from_numpy(rowptr).cuda(), torch.from_numpy(colind).cuda())
    At, bt = torch.from_numpy(A).cuda(), torch.from_numpy(b).cuda()
    for mode in ("sync", "async"):
        x = torch.zeros_like(bt)
        res = ab.fgmres_solve(pat, At, ab.Factors(pat, dtype), bt, x, rtol=1e-6, build_sweeps=3, mode=mode)
        assert res.converged and res.iters <= ro.iters + 2
        r = b - np.array([sum(A[p] @ x.cpu().numpy()[colind[p]] for p in range(rowptr[i], rowptr[i + 1]))
                          for i in range(3000)])
        assert np.linalg.norm(r) <= 1.01e-6 * np.linalg.norm(b)
