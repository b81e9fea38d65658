"""Tickets of the asynchronous block build chosen by the size of the work list."""
import numpy as np
import pytest

import abilu_inputs as gen


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 3), (107, 108), (109, 108), (304, 306), (306, 307)])
def test_default_tickets_reach_the_sequential_factors(nx, ny):
    """One block, a ragged last ticket, both sides of one step per warp (8
    blocks on each of 7,296 resident warps) and of the line to 128-block
    tickets (64 blocks per warp): the in-place build reaches sequential block
    ILU(0).  The bound is the FP32 one of the other ticket sizes."""
    import torch
    import oracle
    import paper_1912_00539_gb300.abilu as ab
    s = gen.small_system(nx, ny, seed=5)
    pat = ab.Pattern(torch.from_numpy(s.rowptr).cuda(), torch.from_numpy(s.colind).cuda())
    A = torch.from_numpy(s.vals).cuda()
    Xs, Ds, _ = oracle.bilu0_seq(s.rowptr, s.colind, s.vals)
    fac = ab.Factors(pat, "f32")
    fac.build(A, 40, mode="async")
    X, D = fac.export()
    assert np.abs(X.cpu().numpy() - Xs).max() / np.abs(Xs).max() < 1e-4
    assert np.abs(D.cpu().numpy() - Ds).max() / np.abs(Ds).max() < 1e-4
