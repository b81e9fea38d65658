"""The FP64 block product's integer sums (third and fourth block of a row)."""
from fractions import Fraction

import numpy as np
import pytest


def _system(blocks, seed, fill):
    """Rows of 1 .. `blocks` blocks; `fill(rng, n)` draws n values."""
    rng = np.random.default_rng(seed)
    n = 40
    rows = []
    for i in range(n):
        others = [j for j in range(n) if j != i]
        rng.shuffle(others)
        rows.append(sorted([i] + others[:i % blocks]))
    rowptr = np.cumsum([0] + [len(r) for r in rows]).astype(np.int32)
    colind = np.concatenate(rows).astype(np.int32)
    A = fill(rng, rowptr[-1] * 16).reshape(-1, 4, 4)
    return rowptr, colind, A, fill(rng, n * 4).reshape(n, 4)


def _run(rowptr, colind, A, x):
    import torch
    import paper_1912_00539_gb300.abilu as ab
    pat = ab.Pattern(torch.from_numpy(rowptr).cuda(), torch.from_numpy(colind).cuda())
    y = torch.empty(x.shape, dtype=torch.float64, device="cuda")
    ab.bsr_spmv(pat, torch.from_numpy(A).cuda(), torch.from_numpy(x).cuda(), y)
    return y.cpu().numpy()


def _normal(rng, n):
    return rng.standard_normal(n)


def _wide(rng, n):
    return np.ldexp(rng.standard_normal(n), rng.integers(-300, 300, n))


def _tiny(rng, n):   # every product below the integer range, many subnormal
    return np.ldexp(rng.standard_normal(n), rng.integers(-560, -480, n))


def _huge(rng, n):   # operands above the integer range
    return np.ldexp(rng.standard_normal(n), rng.integers(478, 505, n))


def _zeros(rng, n):
    v = rng.standard_normal(n) * (rng.random(n) < 0.4)
    v[rng.random(n) < 0.1] = -0.0
    v[rng.random(n) < 0.1] = 5e-324
    return v


@pytest.mark.gpu
@pytest.mark.parametrize("fill", [_normal, _wide, _tiny, _huge, _zeros])
@pytest.mark.parametrize("blocks", [1, 2, 3, 4, 7])
def test_product_against_exact_sums(blocks, fill):
    """Each entry within k u (sum |a x|) of the exact sum, k the number of
    products (u = 2^-53): the bound of a sum of FMAs, which the integer part
    (3 x 8 units of 2^-58 of the largest product, one rounding) keeps; products
    below the normal range add half a subnormal unit each."""
    rowptr, colind, A, x = _system(blocks, 3 * blocks, fill)
    y = _run(rowptr, colind, A, x)
    for i in range(x.shape[0]):
        for q in range(4):
            s, m, k = Fraction(0), Fraction(0), 0
            for p in range(rowptr[i], rowptr[i + 1]):
                for c in range(4):
                    t = Fraction(float(A[p, q, c])) * Fraction(float(x[colind[p], c]))
                    s, m, k = s + t, m + abs(t), k + 1
            err = abs(Fraction(float(y[i, q])) - s)
            assert err <= k * m / 2**53 + k * Fraction(5e-324), (i, q)


@pytest.mark.gpu
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_infinities_and_nans_pass_through(bad):
    rowptr, colind, A, x = _system(4, 1, _normal)
    x[7, 2] = bad
    x[9, 1] = 0.0
    p = rowptr[11] + 3
    A[p, 1, 1] = bad
    y = _run(rowptr, colind, A, x)
    want = np.zeros_like(y)
    with np.errstate(invalid="ignore"):
        for i in range(x.shape[0]):
            for q in range(rowptr[i], rowptr[i + 1]):
                want[i] += A[q] @ x[colind[q]]
    assert np.array_equal(np.isfinite(y), np.isfinite(want))
    assert np.array_equal(np.isnan(y), np.isnan(want))
    inf = np.isinf(want)
    assert np.array_equal(y[inf], want[inf])


@pytest.mark.gpu
def test_integers_are_exact():
    rowptr, colind, A, x = _system(5, 2, lambda r, n: r.integers(-2**20, 2**20, n).astype(np.float64))
    y = _run(rowptr, colind, A, x)
    for i in range(x.shape[0]):
        for q in range(4):
            s = sum(int(A[p, q, c]) * int(x[colind[p], c]) for p in range(rowptr[i], rowptr[i + 1]) for c in range(4))
            assert y[i, q] == float(s)


def _only_integer_part(n, seed):
    """Rows 4 .. n-1 of blocks in columns 0, 1, 2 and the diagonal, x zero in columns
    0 and 1: the sum is that of the third and fourth block alone."""
    rng = np.random.default_rng(seed)
    cols = [sorted({i}) if i < 4 else [0, 1, 2, i] for i in range(n)]
    rowptr = np.cumsum([0] + [len(c) for c in cols]).astype(np.int32)
    return rng, rowptr, np.concatenate(cols).astype(np.int32)


def _exact_rows(rowptr, A, x, colind, rows):
    for i in rows:
        for q in range(4):
            t = [Fraction(float(A[p, q, c])) * Fraction(float(x[colind[p], c]))
                 for p in range(rowptr[i], rowptr[i + 1]) for c in range(4)]
            yield i, q, sum(t), max(abs(v) for v in t)


@pytest.mark.gpu
@pytest.mark.parametrize("gap", [0, 20, 45, 70])
def test_cancelling_products_keep_the_bound_of_the_largest(gap):
    """Two products of 2^gap and its negative ahead of six of about 1: each product is
    kept to 3 units of 2^-58 of the largest, and one rounding follows.  (FMAs in this
    order would keep the small ones whatever the gap.)"""
    n = 40
    rng, rowptr, colind = _only_integer_part(n, gap)
    A = rng.standard_normal((rowptr[-1], 4, 4))
    x = rng.standard_normal((n, 4))
    x[:2] = 0.0
    x[2, 0] = x[2, 1] = 1.75 * 2.0**(gap // 2)
    third = rowptr[4:-1] + 2
    A[third, :, 0] *= 2.0**(gap - gap // 2)
    A[third, :, 1] = -A[third, :, 0]
    y = _run(rowptr, colind, A, x)
    for i, q, s, m in _exact_rows(rowptr, A, x, colind, range(4, n)):
        got = Fraction(float(y[i, q]))
        assert abs(got - s) <= 24 * m / 2**58 + abs(got) / 2**53, (i, q)


@pytest.mark.gpu
def test_integers_up_to_2_25_are_exact():
    n = 60
    rng, rowptr, colind = _only_integer_part(n, 1)
    A = rng.integers(-2**25, 2**25 + 1, (rowptr[-1], 4, 4)).astype(np.float64)
    x = rng.integers(-2**25, 2**25 + 1, (n, 4)).astype(np.float64)
    x[:2] = 0.0
    x[2], x[7] = 2.0**25, 2.0**25
    A[rowptr[7] + 2:rowptr[7] + 4] = 2.0**25   # eight products of 2^50
    y = _run(rowptr, colind, A, x)
    for i, q, s, _ in _exact_rows(rowptr, A, x, colind, range(4, n)):
        assert y[i, q] == float(s) and Fraction(float(y[i, q])) == s, (i, q)


@pytest.mark.gpu
@pytest.mark.parametrize("n,blocks", [(119999, 4), (120000, 4), (120001, 7), (121599, 3), (121601, 5),
                                      (120001, 9), (250000, 9)])
def test_streamed_rows_match_the_direct_form(n, blocks):
    """Both sides of the size where the rows go through shared memory, row counts
    that leave the last 160-row pass of some CTAs ragged, rows of 1 .. `blocks`
    blocks (none to five beyond the staged four; five a row and more on average:
    direct below 250,000 rows).  Both forms run the same
    operations in the same order, so a system's rows give the same bits alone
    (direct) and as the tail of a larger one (streamed)."""
    import torch
    import paper_1912_00539_gb300.abilu as ab
    rng = np.random.default_rng(n + blocks)
    cnt = 1 + np.arange(n) % blocks
    rowptr = np.concatenate([[0], np.cumsum(cnt)]).astype(np.int32)
    row = np.repeat(np.arange(n), cnt)
    k = np.arange(len(row)) - rowptr[row]
    # columns within the last or the first 60,000 rows of each half, sorted and
    # distinct: row - a few .. row, kept inside the row's half
    half = np.where(row >= n - 60000, n - 60000, 0)
    colind = np.where(row - cnt[row] + 1 >= half, row - (cnt[row] - 1 - k), np.maximum(half, row) + k)
    colind = np.minimum(colind, n - 1).astype(np.int32)
    A = torch.from_numpy(rng.standard_normal((len(row), 4, 4))).cuda()
    x = torch.from_numpy(rng.standard_normal((n, 4))).cuda()
    y0 = torch.from_numpy(rng.standard_normal((n, 4))).cuda()
    pat = ab.Pattern(torch.from_numpy(rowptr).cuda(), torch.from_numpy(colind).cuda())
    y, y2 = torch.empty_like(x), y0.clone()
    ab.bsr_spmv(pat, A, x, y)
    ab.bsr_spmv(pat, A, x, y2, alpha=-0.5, beta=2.0)
    # the last 60,000 rows as a system of their own
    o, p = n - 60000, int(rowptr[n - 60000])
    sub = ab.Pattern(torch.from_numpy(rowptr[o:] - p).cuda(), torch.from_numpy(colind[p:] - o).cuda())
    z, z2 = torch.empty_like(x[o:]), y0[o:].clone()
    ab.bsr_spmv(sub, A[p:], x[o:], z)
    ab.bsr_spmv(sub, A[p:], x[o:], z2, alpha=-0.5, beta=2.0)
    assert torch.equal(y[o:], z) and torch.equal(y2[o:], z2)
    want = np.zeros((n, 4))
    np.add.at(want, row, np.einsum("prc,pc->pr", A.cpu().numpy(), x.cpu().numpy()[colind]))
    assert np.abs(y.cpu().numpy() - want).max() < 1e-13 * np.abs(want).max()
