"""Row conversions between FP64 and the factors' FP32 and BF16."""
import numpy as np
import pytest

import abilu_inputs as gen


def _special(rng, n):
    """Normal values, ties and their neighbours on the 29 dropped bits, FP32's
    smallest and largest, subnormals, overflow, zeros, infinities, NaN."""
    v = rng.standard_normal(n)
    bits = v.view(np.uint64)
    k = rng.integers(0, 8, n)
    bits[k == 0] = (bits[k == 0] & ~np.uint64(0x1FFFFFFF)) | np.uint64(0x10000000)
    bits[k == 1] = (bits[k == 1] & ~np.uint64(0x1FFFFFFF)) | np.uint64(0x10000001)
    bits[k == 2] = bits[k == 2] | np.uint64(0xFFFFFFFFF)
    edge = np.array([0.0, -0.0, 2.0**-126, 2.0**-127, 2.0**-149, 2.0**-150, 2.0**-151, 1e-310,
                     2.0**-126 * (1 - 2.0**-25), 3.4028234663852886e38, 3.4028235677973366e38, 1e39, -1e300,
                     np.inf, -np.inf, np.nan])
    pick = rng.random(n) < 0.2
    v[pick] = rng.choice(edge, pick.sum())
    return v


def _bf16(f):
    """FP32 -> BF16 -> FP32, nearest even."""
    u = f.view(np.uint32).astype(np.uint64)
    r = ((u + np.uint64(0x7FFF) + ((u >> np.uint64(16)) & np.uint64(1))) >> np.uint64(16)) << np.uint64(16)
    out = r.astype(np.uint32).view(np.float32).copy()
    out[np.isnan(f)] = np.nan
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("seed", range(4))
def test_initial_factors_are_the_rounded_blocks(dtype, seed):
    """With no sweep the off-diagonal factors are A's blocks in the storage type,
    so a build and an export pass every value through both conversions."""
    import torch
    import paper_1912_00539_gb300.abilu as ab
    s = gen.small_system(23, 17, seed=seed)
    rng = np.random.default_rng(seed)
    A = s.vals.copy()
    rows = np.repeat(np.arange(s.n), np.diff(s.rowptr))
    off = rows != s.colind
    A[off] = _special(rng, off.sum() * 16).reshape(-1, 4, 4)
    pat = ab.Pattern(torch.from_numpy(s.rowptr).cuda(), torch.from_numpy(s.colind).cuda())
    fac = ab.Factors(pat, dtype)
    fac.build(torch.from_numpy(A).cuda(), 0, mode="sync")
    X = fac.export()[0].cpu().numpy()[off]
    with np.errstate(over="ignore"):
        want = A[off].astype(np.float32)
    if dtype == "bf16":
        want = _bf16(want.ravel()).reshape(want.shape)
    want = want.astype(np.float64)
    assert np.array_equal(np.isnan(X), np.isnan(want))
    ok = ~np.isnan(want)
    assert np.array_equal(X[ok].view(np.uint64), want[ok].view(np.uint64))


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_zero_guess_ignores_x(dtype):
    """x is written, not read, by a solve from a zero guess: with NaN in it, for a
    solve of several cycles, one that may take no step, and b = 0."""
    import torch
    import paper_1912_00539_gb300.abilu as ab
    s = gen.small_system(37, 11, seed=2)
    pat = ab.Pattern(torch.from_numpy(s.rowptr).cuda(), torch.from_numpy(s.colind).cuda())
    A, b = torch.from_numpy(s.vals).cuda(), torch.from_numpy(s.b).cuda()
    fac = ab.Factors(pat, dtype)
    kw = dict(rtol=1e-6, build_sweeps=4, apply_sweeps_lower=3, apply_sweeps_upper=3, mode="sync")
    x0 = torch.zeros_like(b)
    r0 = ab.fgmres_solve(pat, A, fac, b, x0, restart=2, zero_guess=False, **kw)
    x = torch.full_like(b, float("nan"))
    r = ab.fgmres_solve(pat, A, fac, b, x, restart=2, zero_guess=True, **kw)
    assert r.converged and r.restarts > 1 and r.iters == r0.iters
    assert float((x - x0).norm() / x0.norm()) < 1e-6
    x.fill_(float("nan"))
    ab.fgmres_solve(pat, A, fac, b, x, restart=2, zero_guess=True, max_iters=0, **kw)
    assert torch.equal(x, torch.zeros_like(x))
    x.fill_(float("nan"))
    r = ab.fgmres_solve(pat, A, fac, torch.zeros_like(b), x, restart=2, zero_guess=True, **kw)
    assert r.converged and torch.equal(x, torch.zeros_like(x))
