"""add_block_diagonal: A_out = A_in + diag(d_i) on the diagonal blocks."""
import numpy as np
import pytest


@pytest.mark.gpu
@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("n,longest", [(1, 1), (63, 4), (64, 5), (65, 9), (200, 13)])
def test_equal_to_numpy(n, longest, in_place):
    """Ragged 64-row CTAs, rows of 1 .. `longest` blocks (four in flight at a time),
    the diagonal block at every place of its row, input and output apart or
    the same array; the copies and the one addition round as numpy's."""
    import torch
    import paper_1912_00539_gb300.abilu as ab
    rng = np.random.default_rng(n)
    rowptr, colind = [0], []
    for i in range(n):
        js = set(int(j) for j in rng.choice(n, size=min(n - 1, int(rng.integers(0, longest))), replace=False)) | {i}
        colind += sorted(js)
        rowptr.append(len(colind))
    rowptr, colind = np.array(rowptr, np.int32), np.array(colind, np.int32)
    A = rng.standard_normal((len(colind), 4, 4))
    A[rng.random(A.shape) < 0.1] = -0.0
    A[0, 0, 0] = np.inf
    d = rng.standard_normal((n, 4))
    want = A.copy()
    diag = np.flatnonzero(np.repeat(np.arange(n), np.diff(rowptr)) == colind)
    for q in range(4):
        want[diag, q, q] += d[:, q]
    pat = ab.Pattern(torch.from_numpy(rowptr).cuda(), torch.from_numpy(colind).cuda())
    Ain = torch.from_numpy(A).cuda()
    out = Ain if in_place else torch.full_like(Ain, np.nan)
    ab.add_block_diagonal(pat, Ain, out, torch.from_numpy(d).cuda())
    assert np.array_equal(out.cpu().numpy().view(np.int64), want.view(np.int64))
    if not in_place:
        assert np.array_equal(Ain.cpu().numpy().view(np.int64), A.view(np.int64))
