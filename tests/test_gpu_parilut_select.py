"""Selection of the kept blocks of the threshold factorisation."""
import numpy as np
import pytest

import abilu_inputs as gen


def _compare(s, vals, fill):
    """One fill-and-drop step without sweeps: the factors stay A's own blocks on
    the kept pattern, so the pattern depends on the selection alone."""
    import torch
    import oracle
    import paper_1912_00539_gb300.abilu as ab
    pat = ab.Pattern(torch.from_numpy(s.rowptr).cuda(), torch.from_numpy(s.colind).cuda())
    got, _ = ab.parilut(pat, torch.from_numpy(vals).cuda(), fill=fill, iters=1, sweeps=0)
    rp, ci = (t.cpu().numpy() for t in got.arrays())
    rpo, cio, _, _ = oracle.parilut(s.rowptr, s.colind, vals, fill=fill, iters=1, sweeps=0)
    assert np.array_equal(rp, rpo) and np.array_equal(ci, cio)


@pytest.mark.gpu
@pytest.mark.parametrize("fill", [0.0, 0.01, 0.3, 0.75, 1.0, 1.2])
@pytest.mark.parametrize("nx,ny", [(2, 2), (11, 12), (16, 8), (37, 11)])
def test_kept_blocks(nx, ny, fill):
    """No block of a side kept, few, most, all; rows below, at and above a CTA's
    256."""
    s = gen.small_system(nx, ny, seed=4)
    _compare(s, s.vals, fill)


@pytest.mark.gpu
@pytest.mark.parametrize("fill", [0.0, 0.3, 0.75])
@pytest.mark.parametrize("scale", [1.0, 1e-160, 1e-170])
def test_ties(fill, scale):
    """Off-diagonal blocks of three distinct norms, so the wanted rank falls among
    equal keys (squared norms): normal; subnormal and still distinct (4, 16 and 36
    times 1e-320); all zero (1e-340)."""
    s = gen.small_system(13, 9, seed=6)
    vals = s.vals.copy()
    rows = np.repeat(np.arange(s.n), np.diff(s.rowptr))
    off = rows != s.colind
    vals[off] = np.eye(4) * scale * (1.0 + (s.colind[off] % 3))[:, None, None]
    keys = np.unique((vals[off] * vals[off]).sum(axis=(1, 2)))
    assert len(keys) == (1 if scale == 1e-170 else 3)
    _compare(s, vals, fill)
