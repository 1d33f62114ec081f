"""lobpcg_chebyshev_apply on cases whose result is known to the last bit."""
import numpy as np
import pytest

import paper_1704_07458_gb300 as gb
from gpu_util import torch_cuda, dev, dev_i32, host

pytestmark = pytest.mark.gpu

N = 70


def _apply(rows, R, m, ldr, degree, in_place=False):
    """rows: per row a list of (column, value)."""
    torch = torch_cuda()
    rp = dev_i32(np.cumsum([0] + [len(r) for r in rows]))
    ci = dev_i32(np.array([c for r in rows for c, _ in r]))
    va = dev(np.array([v for r in rows for _, v in r]))
    Rd, W = dev(R, ldr), dev(np.full((len(rows), m), np.nan), ldr)
    W = Rd if in_place else W
    c = gb.lobpcg_chebyshev_create(len(rows), rp, ci, va, None, degree, 0.05, 2.0, m)
    rc = gb.lobpcg_chebyshev_apply(c, len(rows), m, Rd, ldr, W, ldr, None)
    torch.cuda.synchronize()
    gb.lobpcg_chebyshev_destroy(c)
    assert rc == 0
    return host(W, m)


@pytest.mark.parametrize("m,ldr", [(1, 1), (4, 4), (5, 5), (5, 8), (71, 72)])
@pytest.mark.parametrize("degree", [2, 5])
def test_terms_that_cancel_in_a_w_cost_r_no_bits(m, ldr, degree):
    """Rows 0 and 1 hold the same values, so +-2^40 times them adds an exact zero
    to A w: the result is that of the diagonal matrix, bit for bit."""
    rng = np.random.default_rng(m + degree)
    d = 1.0 + rng.random(N)
    d[1] = d[0]
    R = rng.standard_normal((N, m))
    R[1] = R[0]
    big = 2.0 ** 40
    plain = [[(i, d[i])] for i in range(N)]
    coupled = plain[:2] + [[(0, big), (1, -big), (i, d[i])] for i in range(2, N)]
    np.testing.assert_array_equal(_apply(coupled, R, m, ldr, degree),
                                  _apply(plain, R, m, ldr, degree))


@pytest.mark.parametrize("m,ldr", [(1, 1), (4, 4), (5, 5), (5, 8), (71, 72)])
@pytest.mark.parametrize("degree", [1, 2, 5])
def test_result_may_replace_r(m, ldr, degree):
    """Every element of R is read before W's takes its place."""
    R = np.random.default_rng(m).standard_normal((N, m))
    rows = [[(j, 4.0 if i == j else -1.0) for j in (i - 7, i - 1, i, i + 1, i + 7) if 0 <= j < N]
            for i in range(N)]
    np.testing.assert_array_equal(_apply(rows, R, m, ldr, degree, in_place=True),
                                  _apply(rows, R, m, ldr, degree))


@pytest.mark.parametrize("m", [1, 5, 31, 71])
def test_blocks_may_end_at_their_last_column(m):
    """Nothing past the m columns of a row belongs to the call: R and X end with
    the last row's m-th value, and the padding of the other rows is NaN."""
    torch = torch_cuda()
    n, ld = N, m + 1
    rng = np.random.default_rng(m)
    X, b = rng.standard_normal((n, m)), 1.0 + rng.random(n)
    rows = [[(j, 4.0 if i == j else -1.0) for j in (i - 7, i - 1, i, i + 1, i + 7) if 0 <= j < N]
            for i in range(N)]
    rp = dev_i32(np.cumsum([0] + [len(r) for r in rows]))
    ci = dev_i32(np.array([c for r in rows for c, _ in r]))
    va = dev(np.array([v for r in rows for _, v in r]))
    flat = np.full((n, ld), np.nan)
    flat[:, :m] = X
    tight, full = dev(flat.reshape(-1)[:(n - 1) * ld + m]), dev(X, ld)
    out = []
    for x in (tight, full):
        Y, BY = (dev(np.full((n, ld), np.nan)) for _ in range(2))
        assert gb.lobpcg_spmm(n, rp, ci, va, x, ld, m, Y, ld, dev(b), BY, ld, None) == 0
        W = dev(np.full((n, ld), np.nan))
        c = gb.lobpcg_chebyshev_create(n, rp, ci, va, None, 4, 0.05, 2.0, m)
        assert gb.lobpcg_chebyshev_apply(c, n, m, x, ld, W, ld, None) == 0
        torch.cuda.synchronize()
        gb.lobpcg_chebyshev_destroy(c)
        out.append([host(t) for t in (Y, BY, W)])
    for got, want in zip(*out):
        np.testing.assert_array_equal(got, want)
        assert np.all(np.isnan(got[:, m:])) and not np.any(np.isnan(got[:, :m]))
