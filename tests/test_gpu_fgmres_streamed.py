"""FGMRES on systems large enough for the streamed row products."""
import numpy as np
import pytest

import abilu_inputs as gen


@pytest.mark.gpu
@pytest.mark.parametrize("form", ["single", "classical", "cgs2"])
@pytest.mark.parametrize("nx,ny", [(300, 201), (260, 251)])
def test_streamed_solution_equals_oracle(nx, ny, form):
    """120,600 and 130,520 rows (ragged last passes) in every Gram-Schmidt form,
    more steps than one pass takes dots of (6), so every width of the fused
    kernel runs; the bound is that of the same comparison on smaller systems."""
    import torch
    import oracle
    import paper_1912_00539_gb300.abilu as ab
    s = gen.small_system(nx, ny, seed=3, cfl=1e4)
    rtol = 1e-6 if form == "single" else 1e-8
    Xo, Do, _ = oracle.bilu_sync(s.rowptr, s.colind, s.vals, 2)
    xo, ro = oracle.fgmres(s.rowptr, s.colind, s.vals, Xo, Do, s.b, 1, 1, restart=30, rtol=rtol)
    assert ro.iters > 7
    pat = ab.Pattern(torch.from_numpy(s.rowptr).cuda(), torch.from_numpy(s.colind).cuda())
    A, b = torch.from_numpy(s.vals).cuda(), torch.from_numpy(s.b).cuda()
    fac = ab.Factors(pat, "f64")
    x = torch.empty_like(b)
    res = ab.fgmres_solve(pat, A, fac, b, x, restart=30, rtol=rtol, build_sweeps=2,
                          apply_sweeps_lower=1, apply_sweeps_upper=1, mode="sync",
                          reorth=form == "cgs2", zero_guess=True)
    assert res.converged and res.iters == ro.iters, (res.iters, ro.iters)
    xn = x.cpu().numpy()
    assert np.linalg.norm(xn - xo) / np.linalg.norm(xo) < 1e-11
