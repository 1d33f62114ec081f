"""The digit split of the tcgen05 Gram and update, to its last bit.

An FP64 operand x with exponent bound E (|x| < 2^E, shared by a row or column)
is cut into S digits whose sum is F = round(|x| 2^(8S-1-E)), half up in
magnitude.  Sixteen equal entries against sixteen factors 0.5 (one digit of 64,
one MMA of K = 16) give 16 * 64 F in units that the FP32 accumulators and the
2^-30 rounding of the int64 sums hold exactly, so the product must equal
8 F 2^(E-8S+1): one digit fewer, a second rounding or another rounding of a tie
shows.  For S = 6 the accumulator that digits 3, 4 and 5 share aligns every
product to the largest term with about 24 bits, and the last digit's products
end at 2^-34, so there |d_3| <= 8: 16 * 64 d_3 2^-24 then stays below 2^-10.
With seven slices the sums keep 2^-30 (update) or 2^-34 (Gram) of a product of
leading digits; the bounds there are those roundings.
"""
import numpy as np
import pytest

import paper_1704_07458_gb300 as gb
from gpu_util import torch_cuda, dev, host

pytestmark = pytest.mark.gpu

TC = gb.LOBPCG_GEMM_OZAKI_TC


def _cut(x, E, slices):
    """F of each x (Python integers: exact)."""
    out = []
    for v, e in zip(x, E):
        m, be = np.frexp(abs(v))
        mant, sh = int(np.ldexp(m, 53)), 53 - (8 * slices - 1) + (int(e) - int(be))
        f = mant << -sh if sh <= 0 else (mant + (1 << (sh - 1))) >> sh
        out.append(-f if v < 0 else f)
    return out


def _values(count, slices, seed):
    """Mantissas in [0.5, 1) of every kind a rounding can get wrong: random, on
    the last digit's grid, on its ties and beside them, ends of the binade;
    both signs; and how far below the bound each shall lie."""
    rng = np.random.default_rng(seed)
    m = (1 << 52) + rng.integers(0, 1 << 52, count)
    drop = np.where(np.arange(count) % 2 == 0, 0, rng.integers(0, 50, count))
    for i in range(count):
        low = min(52, 53 - (8 * slices - 1) + int(drop[i]))  # bits below the last digit
        if slices == 6 and low + 19 < 52:  # a small fourth digit
            top = min(52, low + 24)
            m[i] = int(m[i]) & ~((1 << top) - (1 << (low + 19))) | (1 << 52)
        kind = i % 8
        if kind >= 4 and low >= 1:
            m[i] = (int(m[i]) >> low << low) + (0 if kind == 4 else (1 << (low - 1)))
            if kind >= 6:
                m[i] += 1 if kind == 6 else -1
    # ends of the binade, and of the low 29 bits that a float's mantissa leaves
    m[:4] = [1 << 52, (1 << 53) - 1, (1 << 53) - (1 << 29), (1 << 53) - (1 << 29) + 1]
    drop[:4] = 0
    x = np.ldexp(m.astype(np.float64), -53) * np.where(rng.random(count) < 0.5, -1.0, 1.0)
    return x, drop


def _check(got, x, E, slices, terms, frac):
    """got: sums of `terms` products of x with 0.5."""
    F, fewer = _cut(x, E, slices), _cut(x, E, slices - 1)
    assert any(f != g << 8 for f, g in zip(F, fewer))
    if slices <= 6:
        want = np.array([np.ldexp(float(terms * f), int(e) - 8 * slices) for f, e in zip(F, E)])
        np.testing.assert_array_equal(got, want)
        return
    # half a unit of the last digit, the int64 sums' rounding and 16 FP32 sums
    # below 2^-11, in units of the leading digits' product (2^-14 of the bounds)
    err = terms * 64 * 0.5 * 2.0 ** -48 + 0.5 * 2.0 ** -frac + 16 * 2.0 ** -35
    lost = terms * 64 * 0.5 * 2.0 ** -40  # largest error of one digit fewer
    assert err < lost / 4
    scaled = np.abs(np.ldexp(got, -E.astype(int)) - 0.5 * terms * np.ldexp(x, -E.astype(int)))
    assert np.all(scaled <= err * 2.0 ** -14)


def _operand(slices, count, seed):
    """x with exponent bounds E = 0, and whether an entry must set the bound.
    With seven slices every x lies right below it."""
    x, drop = _values(count, slices, seed)
    if slices == 7:
        drop[:] = 0
    if slices == 6:  # what is left with a large fourth digit (it leads, or a carry)
        F = _cut(np.ldexp(x, -drop), np.zeros(count), slices)
        fourth = np.array([((((f + 0x8080) >> 16) + 128) % 256) - 128 for f in F])
        x[np.abs(fourth) > 8] = 0.5
        drop[np.abs(fourth) > 8] = 0
    return np.ldexp(x, -drop), drop > 0


# groups of 32 columns or rows share the decision for the fast split: 2^-950 puts
# a group beyond its exponents
@pytest.mark.parametrize("slices", [3, 4, 5, 6, 7])
@pytest.mark.parametrize("side", ["U", "V"])
@pytest.mark.parametrize("scale", [0, -950, 300])
def test_gram_digits_are_one_rounding(slices, side, scale):
    torch = torch_cuda()
    terms, cols = (16, 96) if slices <= 6 else (256, 80)
    x, below = _operand(slices, cols, 100 + 11 * slices)
    E = np.full(cols, scale)
    x = np.ldexp(x, E)
    A = np.zeros((terms + 16, cols) if slices <= 6 else (terms, cols))
    A[:terms] = x
    if slices <= 6:
        A[terms] = np.ldexp(0.75, E) * below  # sets the bound; multiplied by zero
    B = np.zeros((len(A), 16))
    B[:terms] = 0.5
    U, V = (A, B) if side == "U" else (B, A)
    p, q = U.shape[1], V.shape[1]
    G = dev(np.full(p * q, np.nan))
    rc = gb.lobpcg_gram(len(A), dev(U, p), p, p, dev(V, q), q, q, G, p, TC, slices)
    torch.cuda.synchronize()
    assert rc == 0
    got = host(G).reshape(q, p)
    for r in got if side == "U" else got.T:
        _check(r, x, E, slices, terms, 34)


@pytest.mark.parametrize("slices", [3, 4, 5, 6, 7])
@pytest.mark.parametrize("scale", [0, -950, 300])
def test_update_digits_are_one_rounding(slices, scale):
    torch = torch_cuda()
    terms, n = 16 if slices <= 6 else 256, 160
    x, below = _operand(slices, n, 200 + 7 * slices)
    E = np.zeros(n, dtype=int)
    E[64:96] = scale  # one group of rows
    x = np.ldexp(x, E)
    top = int(np.frexp(x)[1].max())  # a column's exponent, by which it is balanced
    S = np.zeros((n, terms + 16) if slices <= 6 else (n, terms))
    S[:, :terms] = x[:, None]
    if slices <= 6:  # column `terms` (its factors are zero) sets the rows' bounds
        S[:, terms] = np.where(below, np.ldexp(0.75, E - top), 0.0)
        S[0, terms] = np.ldexp(0.75, int(E[0]) - top)
        S[64, terms] = np.ldexp(0.75, int(E[64]) - top)
        assert np.frexp(S[:, terms])[1].max() == 0
    s = S.shape[1]
    C = np.zeros((s, 16))
    C[:terms] = 0.5
    Y = dev(np.full((n, 16), np.nan), 16)
    rc = gb.lobpcg_update(n, dev(S, s), s, s, dev(C.T.copy().reshape(-1)), s, 16, 1.0, 0.0, None,
                          0, Y, 16, TC, slices)
    torch.cuda.synchronize()
    assert rc == 0
    got = host(Y, 16)
    for j in (0, 7, 15):
        _check(got[:, j], x, E, slices, terms, 30)


def test_update_adds_y0_before_it_rounds():
    """Over several blocks of 256 columns a sum may need more than the 53 bits
    of a double; Y0 joins it before the one rounding.  2,049 products of 64 x 64
    digits (2^53 + 2^42 in units of 2^-30) and one unit: less the first, the unit
    is left, exactly."""
    torch = torch_cuda()
    n, m, s = 130, 16, 2050
    S = np.full((n, s), 0.5)
    C = np.full((s, m), 0.5)
    C[-1] = 2.0 ** -43
    big, unit = 2049 * 0.25, 2.0 ** -44
    Y0 = np.tile([-big, big, 1.0, 0.0], (n, m // 4))
    Y = dev(np.full((n, m), np.nan), m)
    rc = gb.lobpcg_update(n, dev(S, s), s, s, dev(C.T.copy().reshape(-1)), s, m, 1.0, 1.0,
                          dev(Y0, m), m, Y, m, TC, 6)
    torch.cuda.synchronize()
    assert rc == 0
    got = host(Y, m)
    np.testing.assert_array_equal(got[:, ::4], unit)
    for c in (1, 2, 3):  # big + unit, one part in 2^53, is lost in a double
        np.testing.assert_array_equal(got[:, c::4], big + Y0[0, c])
