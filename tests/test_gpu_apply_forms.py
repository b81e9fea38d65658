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
