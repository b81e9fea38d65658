"""FP64 factor kernels that share a CTA's rows out by their block counts."""
import numpy as np
import pytest


def _system(n, longest, seed):
    """n rows of 1 .. `longest` blocks each (structurally unsymmetric, the
    count varying from row to row), diagonally dominant."""
    rng = np.random.default_rng(seed)
    rowptr, colind = [0], []
    for i in range(n):
        k = min(n - 1, int(rng.integers(0, longest)))
        js = set(int(j) for j in rng.choice(n, size=k, replace=False)) | {i}
        colind += sorted(js)
        rowptr.append(len(colind))
    rowptr, colind = np.array(rowptr, np.int32), np.array(colind, np.int32)
    A = 0.5 * rng.standard_normal((len(colind), 4, 4))
    for i in range(n):
        s = np.abs(A[rowptr[i]:rowptr[i + 1]]).sum(axis=(0, 2))
        d = rowptr[i] + int(np.searchsorted(colind[rowptr[i]:rowptr[i + 1]], i))
        A[d] += np.diag(s + 0.5)
    return rowptr, colind, A, rng.standard_normal((n, 4))


@pytest.mark.gpu
@pytest.mark.parametrize("n,longest", [(1, 1), (7, 3), (32, 5), (33, 2), (64, 9), (65, 4), (200, 1),
                                       (333, 14), (130, 3), (96, 40)])
def test_f64_build_and_sweeps_match_the_oracle(n, longest):
    """Ragged groups of 32 and 64 rows, rows of one block, rows with more blocks
    than the counts that are told apart (4), L and U blocks with and without
    product pairs: in no row, few rows and most rows of a CTA.  The oracle runs the same sweeps in FP64 in another order
    of operations: a few hundred roundings of diagonally dominant blocks."""
    import torch
    import oracle
    import paper_1912_00539_gb300.abilu as ab
    rowptr, colind, A, r = _system(n, longest, 10 * n + longest)
    Xo, Do, _ = oracle.bilu_sync(rowptr, colind, A, 3)
    pat = ab.Pattern(torch.from_numpy(rowptr).cuda(), torch.from_numpy(colind).cuda())
    At, rt = torch.from_numpy(A).cuda(), torch.from_numpy(r).cuda()
    fac = ab.Factors(pat, "f64")
    fac.build(At, 3, mode="sync")
    X, D = fac.export()
    assert np.abs(X.cpu().numpy() - Xo).max() / np.abs(Xo).max() < 1e-13
    assert np.abs(D.cpu().numpy() - Do).max() / np.abs(Do).max() < 1e-13
    z = torch.empty_like(rt)
    for nl, nu in ((1, 1), (2, 3), (4, 2)):
        zo = oracle.apply(rowptr, colind, Xo, Do, r, nl, nu)
        fac.apply(rt, z, nl, nu, mode="sync")
        assert np.abs(z.cpu().numpy() - zo).max() / np.abs(zo).max() < 1e-13
    # in place: both reach the sequential factors and the exact triangular solves
    Xs, Ds, _ = oracle.bilu0_seq(rowptr, colind, A)
    fac.build(At, 60, mode="async")
    X, D = fac.export()
    assert np.abs(X.cpu().numpy() - Xs).max() / np.abs(Xs).max() < 1e-12
    fac.apply(rt, z, 80, 80, mode="async")
    ys = oracle.lower_solve(rowptr, colind, Xs, r)
    zs = oracle.upper_solve(rowptr, colind, Xs, Ds, ys)
    assert np.abs(z.cpu().numpy() - zs).max() / np.abs(zs).max() < 1e-12


@pytest.mark.gpu
@pytest.mark.parametrize("n,longest", [(2, 3), (20, 9), (33, 14), (64, 7), (64, 65)])
def test_f64_in_place_keeps_the_order_of_a_row(n, longest):
    """One in-place sweep over at most 64 rows, which one CTA does: U and Dinv are
    still A's when the L blocks are formed, so L_ij = (A_ij - sum_{k<j} L_ik A_kj)
    A_jj^-1 with the L_ik of the same sweep, whatever the timing (up to a full
    lower triangle, 63 blocks in a row, 62 product pairs).  The bound is that of
    the comparison with the oracle above."""
    import torch
    import paper_1912_00539_gb300.abilu as ab
    rowptr, colind, A, _ = _system(n, longest, 7 * n + longest)
    pos = {(i, int(colind[p])): p for i in range(n) for p in range(rowptr[i], rowptr[i + 1])}
    want, pairs = A.copy(), 0
    for (i, j), p in sorted(pos.items()):
        if j >= i:
            continue
        s = A[p].copy()
        for k in range(j):
            if (i, k) in pos and (k, j) in pos:
                s -= want[pos[i, k]] @ A[pos[k, j]]
                pairs += 1
        want[p] = s @ np.linalg.inv(A[pos[j, j]])
    assert pairs > 0 or longest < 9
    pat = ab.Pattern(torch.from_numpy(rowptr).cuda(), torch.from_numpy(colind).cuda())
    fac = ab.Factors(pat, "f64")
    fac.build(torch.from_numpy(A).cuda(), 1, mode="async")
    X = fac.export()[0].cpu().numpy()
    low = np.array([p for (i, j), p in pos.items() if j < i], np.int64)
    assert np.abs(X[low] - want[low]).max(initial=0.0) < 1e-13 * np.abs(want).max()
