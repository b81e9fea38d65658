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


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny", [(32, 16), (90, 90), (150, 150), (230, 230)])
def test_default_tickets_keep_the_iterations_along_lines(nx, ny):
    """Cells in wall-normal lines, coupled 100 times as strongly along them: FGMRES on
    the default tickets' factors takes the iterations of 128-block tickets, one
    more at most (tickets of 8 to 40 blocks took up to three times as many), over
    repeats, as the in-place build is not deterministic."""
    import torch
    import paper_1912_00539_gb300.abilu as ab
    g = gen.tri_quad_grid(nx, ny, 5)
    n, perm = g.ncells, gen.line_order(nx, ny)
    new = np.empty(n, np.int64)
    new[perm] = np.arange(n)
    i, j = new[np.concatenate([g.edges[:, 0], g.edges[:, 1]])], new[np.concatenate([g.edges[:, 1], g.edges[:, 0]])]
    key = np.sort(np.concatenate([i * n + j, np.arange(n) * (n + 1)]))
    rows, cols = key // n, key % n
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=n))]).astype(np.int32)
    rng = np.random.default_rng(3)
    A = 0.5 * rng.standard_normal((len(rows), 4, 4))
    quad = perm // 2
    A[(np.abs(quad[rows] - quad[cols]) != 1) & (rows != cols)] *= 100.0
    s = np.zeros((n, 4))
    off = rows != cols
    np.add.at(s, rows[off], np.abs(A[off]).sum(axis=2))
    A[~off] = np.einsum("nq,qk->nqk", 1e-3 + s, np.eye(4))
    pat = ab.Pattern(torch.from_numpy(rowptr).cuda(), torch.from_numpy(cols.astype(np.int32)).cuda())
    At, b = torch.from_numpy(A).cuda(), torch.from_numpy(rng.standard_normal((n, 4))).cuda()
    its = []
    for chunk in (128, 0):
        fac = ab.Factors(pat, "f32")
        fac.set_build_chunk(chunk)
        its.append([ab.fgmres_solve(pat, At, fac, b, torch.zeros_like(b), rtol=1e-6, build_sweeps=6,
                                    apply_sweeps_lower=4, apply_sweeps_upper=4, mode="async").iters
                    for _ in range(5)])
    assert max(its[1]) <= max(its[0]) + 1, its
