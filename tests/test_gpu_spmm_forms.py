"""The three forms of the sparse product (column pairs, one and two single
columns a thread) on integers, where every order of summation is exact: all
remainders of a row's length, empty rows beside long ones, ragged widths, and
sizes on both sides of the rules that choose the form."""
import numpy as np
import pytest
import scipy.sparse as sp

import paper_1704_07458_gb300 as gb
from gpu_util import torch_cuda, dev, dev_i32, host

pytestmark = pytest.mark.gpu


def _matrix(n, seed):
    rng = np.random.default_rng(seed)
    length = np.where(np.arange(n) % 50 < 40, rng.integers(0, 9, n), np.arange(n) % 9)
    rowptr = np.concatenate([[0], np.cumsum(length)])
    col = rng.integers(0, n, rowptr[-1])
    col[rng.random(len(col)) < 0.1] = n - 1
    return rowptr, col, rng.integers(-9, 10, rowptr[-1]).astype(np.float64)


@pytest.mark.parametrize("n", [97, 140001])
@pytest.mark.parametrize("m,ld", [(1, 1), (2, 2), (3, 3), (3, 4), (4, 4), (5, 7), (5, 61), (6, 9),
                                  (8, 9), (9, 10), (13, 13), (13, 14), (14, 17), (33, 33), (66, 67),
                                  (81, 82)])
def test_spmm_forms_on_integers(n, m, ld):
    torch = torch_cuda()
    rowptr, col, val = _matrix(n, m)
    rng = np.random.default_rng(n + m)
    X, b = (rng.integers(-9, 10, s).astype(np.float64) for s in ((n, m), n))
    Y, BY = (dev(np.full((n, ld + 1), np.nan)) for _ in range(2))
    rc = gb.lobpcg_spmm(n, dev_i32(rowptr), dev_i32(col), dev(val), dev(X, ld), ld, m, Y, ld + 1,
                        dev(b), BY, ld + 1, None)
    torch.cuda.synchronize()
    assert rc == 0
    A = sp.csr_matrix((val, col, rowptr), shape=(n, n))
    np.testing.assert_array_equal(host(Y, m), A @ X)
    np.testing.assert_array_equal(host(BY, m), b[:, None] * X)
    assert np.all(np.isnan(host(Y)[:, m:])) and np.all(np.isnan(host(BY)[:, m:]))
