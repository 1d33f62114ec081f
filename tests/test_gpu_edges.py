"""Edges of the kernels' tilings and of their dispatch, through the C ABI.

Tolerances are those of the kernel parity tests: the classical bound
gamma_n |x|^T |y| for FP64 sums, plus the digit bound of the emulated products.
"""
import numpy as np
import pytest

import synth
from oracle import kernels as ok
import paper_1704_07458_gb300 as gb
from gpu_util import torch_cuda, dev, host, dev_i32, gamma

pytestmark = pytest.mark.gpu

TC = gb.LOBPCG_GEMM_OZAKI_TC


def _unit(slices):
    return 4 * (4 + 4 * slices) * 2.0 ** (-8 * slices)


# more than one column tile (40 items: pairs with an even ld, single columns else),
# tiles of unequal use, and a last pair with one column
@pytest.mark.parametrize("m,ld", [(41, 41), (80, 80), (81, 82), (97, 100), (161, 163), (282, 288)])
def test_spmm_column_tiles(m, ld):
    torch = torch_cuda()
    A = synth.diffusion_3d_lognormal(9, 1.0, 4)
    X = synth.normal_block(2, 1, A.n, m)
    b = synth.uniform_block(2, 2, A.n, 1.0, 2.0)
    Y, BY = dev(np.zeros((A.n, m)), ld), dev(np.zeros((A.n, m)), ld)
    rc = gb.lobpcg_spmm(A.n, dev_i32(A.rowptr), dev_i32(A.col), dev(A.val), dev(X, ld), ld, m, Y,
                        ld, dev(b), BY, ld)
    torch.cuda.synchronize()
    assert rc == 0
    ref = ok.spmm(A.rowptr, A.col, A.val, X)
    absref = ok.spmm(A.rowptr, A.col, np.abs(A.val), np.abs(X))
    assert np.all(np.abs(host(Y, m) - ref) <= 2 * gamma(8) * absref + 1e-300)
    np.testing.assert_array_equal(host(BY, m), b[:, None] * X)
    assert np.all(host(Y)[:, m:] == 0) and np.all(host(BY)[:, m:] == 0)


@pytest.mark.parametrize("degree", [1, 2, 3, 6])
@pytest.mark.parametrize("m,ldr,ldw", [(1, 1, 1), (6, 6, 7), (83, 84, 83), (96, 97, 96)])
def test_chebyshev_apply_steps(degree, m, ldr, ldw):
    """Saad's Algorithm 12.1 on the host; each step is a 7-term product and
    three operations per element with factors below 4, so the difference stays
    below degree * 16 * 4 units of the largest intermediate."""
    torch = torch_cuda()
    A = synth.diffusion_3d_lognormal(7, 0.5, 3)
    lo, hi = 0.05, 2.0
    rows = np.repeat(np.arange(A.n), np.diff(A.rowptr))
    diag = np.zeros(A.n)
    diag[rows[rows == A.col]] = A.val[rows == A.col]
    R = synth.normal_block(3, 1, A.n, m)
    rp, ci, va = dev_i32(A.rowptr), dev_i32(A.col), dev(A.val)
    c = gb.lobpcg_chebyshev_create(A.n, rp, ci, va, None, degree, lo, hi, m)
    W = dev(np.zeros((A.n, m)), ldw)
    rc = gb.lobpcg_chebyshev_apply(c, A.n, m, dev(R, ldr), ldr, W, ldw)
    torch.cuda.synchronize()
    gb.lobpcg_chebyshev_destroy(c)
    assert rc == 0
    theta, delta = 0.5 * (hi + lo), 0.5 * (hi - lo)
    sigma = theta / delta
    rho = 1.0 / sigma
    d = R / diag[:, None] / theta
    w = d.copy()
    top = np.abs(w).max()
    for _ in range(1, degree):
        z = (R - ok.spmm(A.rowptr, A.col, A.val, w)) / diag[:, None]
        new = 1.0 / (2.0 * sigma - rho)
        d = new * rho * d + (2.0 * new / delta) * z
        w, rho = w + d, new
        top = max(top, np.abs(w).max())
    assert np.abs(host(W, m) - w).max() <= degree * 64 * 2.0 ** -53 * top
    assert np.all(host(W)[:, m:] == 0)


# row remainders of the 16-row chunks, the 64- and 256-row exponent blocks, and
# the tile widths in U (128) and V (96, 80 with seven slices); scale: exponents
# beyond those that the float split takes
@pytest.mark.parametrize("n", [15, 16, 17, 63, 65, 255, 257, 1025])
@pytest.mark.parametrize("p,q", [(1, 1), (33, 16), (128, 80), (129, 97)])
@pytest.mark.parametrize("slices", [3, 5, 6, 7])
@pytest.mark.parametrize("scale", [0, 960])
def test_gram_tc_edges(n, p, q, slices, scale):
    torch = torch_cuda()
    U, V = synth.normal_block(3, 1, n, p), synth.normal_block(4, 1, n, q)
    U[:, 0] = 0.0
    G = dev(np.full(p * q, np.nan))
    rc = gb.lobpcg_gram(n, dev(np.ldexp(U, -scale), p), p, p, dev(np.ldexp(V, scale), q), q, q, G,
                        p, TC, slices)
    torch.cuda.synchronize()
    assert rc == 0
    got = host(G).reshape(q, p).T
    absg, tops = np.abs(U).T @ np.abs(V), np.outer(np.abs(U).max(0), np.abs(V).max(0))
    blocks = (n + 63) // 64
    bound = (2 * gamma(n) + 2.0 ** -44) * absg + (
        _unit(slices) * 4 * 256 * ((n + 255) // 256) + blocks * 2.0 ** -42) * tops
    assert np.all(np.abs(got - U.T @ V) <= bound)
    assert np.all(got[0] == 0.0)


# remainders of the 16-column chunks and 256-column blocks, of the 128-row and
# 96- / 80-column tiles; one chunk in all; more tiles than CTAs
@pytest.mark.parametrize("n,s,m", [(1, 1, 1), (127, 15, 96), (129, 16, 97), (300, 17, 81),
                                   (300, 256, 16), (300, 257, 17), (20000, 31, 10)])
@pytest.mark.parametrize("slices", [3, 6, 7])
@pytest.mark.parametrize("scale", [0, 960])
@pytest.mark.parametrize("beta", [0.0, 1.0])
def test_update_tc_edges(n, s, m, slices, scale, beta):
    torch = torch_cuda()
    S, C = synth.normal_block(5, 1, n, s), synth.normal_block(6, 1, s, m)
    Y0 = synth.normal_block(7, 1, n, m)
    S[0] = 0.0
    Y = dev(np.full((n, m), np.nan), m + 1)
    rc = gb.lobpcg_update(n, dev(np.ldexp(S, -scale), s + 1), s + 1, s,
                          dev(np.ldexp(C, scale).T.copy().reshape(-1)), s, m, 1.0, beta,
                          dev(Y0, m), m, Y, m + 1, TC, slices)
    torch.cuda.synchronize()
    assert rc == 0
    ref = beta * Y0 + S @ C
    Ct = np.abs(C) * (2 * np.abs(S).max(0))[:, None]
    bound = (2 * gamma(s + 1) * (np.abs(S) @ np.abs(C) + beta * np.abs(Y0)) +
             _unit(slices) * 4 * s * Ct.max(0)[None, :] + 2.0 ** -52 * np.abs(ref))
    assert np.all(np.abs(host(Y, m) - ref) <= bound + 1e-300)
    np.testing.assert_array_equal(host(Y, m)[0], beta * Y0[0])


# the FP64 forms: unequal tiles of 16-wide units, one unit, 16-row slabs and
# stages with a remainder; the update's 64-row (many rows) and 16-row tiles
@pytest.mark.parametrize("n,s,m", [(1, 1, 1), (17, 15, 16), (1024, 30, 10), (1000, 81, 65),
                                   (609, 213, 142), (20001, 33, 130), (39000, 17, 16)])
def test_fp64_contraction_tiles(n, s, m):
    torch = torch_cuda()
    S, C = synth.normal_block(5, 1, n, s), synth.normal_block(6, 1, s, m)
    V = synth.normal_block(7, 1, n, m)
    Sd, Vd = dev(S, s + 1), dev(V, m + 3)
    Y, G = dev(np.full((n, m), np.nan), m + 1), dev(np.full(s * m, np.nan))
    assert gb.lobpcg_update(n, Sd, s + 1, s, dev(C.T.copy().reshape(-1)), s, m, -1.5, 0.5, Vd,
                            m + 3, Y, m + 1, gb.LOBPCG_GEMM_F64, 0) == 0
    assert gb.lobpcg_gram(n, Sd, s + 1, s, Vd, m + 3, m, G, s, gb.LOBPCG_GEMM_F64, 0) == 0
    torch.cuda.synchronize()
    bound = 2 * gamma(s + 2) * (1.5 * np.abs(S) @ np.abs(C) + 0.5 * np.abs(V))
    assert np.all(np.abs(host(Y, m) - (0.5 * V - 1.5 * (S @ C))) <= bound)
    got = host(G).reshape(m, s).T
    assert np.all(np.abs(got - S.T @ V) <= 2 * gamma(n) * (np.abs(S).T @ np.abs(V)))


# fewer rows than a CTA's row lanes, one column, several column tiles (128)
@pytest.mark.parametrize("n,m,c0", [(2, 128, 0), (7, 129, 0), (700, 282, 25), (700, 1, 0),
                                    (4097, 257, 256)])
@pytest.mark.parametrize("kdiag", [False, True])
def test_residual_column_tiles(n, m, c0, kdiag):
    torch = torch_cuda()
    X, AX, BX = (synth.normal_block(i, 1, n, m) for i in (8, 9, 10))
    th = np.linspace(-1, 3, m)
    kd = synth.uniform_block(9, 2, n, 2.0, 6.0)
    w = m - c0
    W, be = dev(np.full((n, w), np.nan), w + 1), dev(np.zeros(w))
    rc = gb.lobpcg_residual(n, dev(X, m), dev(AX, m), dev(BX, m), m, m, c0, dev(th),
                            dev(kd) if kdiag else None, W, w + 1, 7.5, 1.25, be)
    torch.cuda.synchronize()
    assert rc == 0
    R = ok.residual(AX, BX, th)[:, c0:]
    scale = (np.abs(AX) + np.abs(BX * th[None, :]))[:, c0:]
    div = kd[:, None] if kdiag else 1.0
    assert np.all(np.abs(host(W, w) - R / div) <= 4 * 2.0 ** -53 * scale / div)
    ref = np.linalg.norm(R, axis=0) / ((7.5 + np.abs(th[c0:]) * 1.25) *
                                       np.linalg.norm(X[:, c0:], axis=0))
    np.testing.assert_allclose(host(be), ref, rtol=1e-13)


# every register tile count of the tridiagonalisation, its largest order and
# the shared-memory form above it
@pytest.mark.parametrize("n", [1, 2, 3, 31, 32, 33, 64, 65, 96, 97, 128, 129, 160, 161, 192, 193,
                               223, 224, 225, 256])
def test_syev_orders(n):
    torch = torch_cuda()
    A = synth.normal_block(11, 1, n, n)
    A = 0.5 * (A + A.T)
    At = dev(A.T.copy().reshape(-1))
    w = dev(np.zeros(n))
    assert gb.lobpcg_syev(n, At, n, w, 2) == 0
    torch.cuda.synchronize()
    wl = np.linalg.eigvalsh(A)
    w, Z, norm = host(w), host(At).reshape(n, n).T, np.abs(wl).max()
    tol = 1e-13 * max(1, n / 50)
    assert np.abs(w - wl).max() <= tol * norm
    assert np.abs(Z.T @ Z - np.eye(n)).max() <= tol
    assert np.abs(A @ Z - Z * w).max() <= tol * norm


def test_entry_points_under_capture():
    """Scratch of a captured call belongs to the graph: a replay gives the bits
    of the direct call."""
    torch = torch_cuda()
    n, m = 3000, 24
    X, AX = dev(synth.normal_block(8, 1, n, m)), dev(synth.normal_block(9, 1, n, m))
    th, kd = dev(np.linspace(1, 2, m)), dev(np.full(n, 3.0))
    C = dev(synth.normal_block(6, 1, m, m).reshape(-1))
    out = [torch.zeros((n, m), dtype=torch.float64, device="cuda") for _ in range(2)]
    small = [torch.zeros(m * m, dtype=torch.float64, device="cuda"),
             torch.zeros(m, dtype=torch.float64, device="cuda")]

    def call(stream):
        return [gb.lobpcg_residual(n, X, AX, None, m, m, 0, th, kd, out[0], m, 2.0, 1.0, small[1],
                                   stream),
                gb.lobpcg_gram(n, X, m, m, AX, m, m, small[0], m, TC, 6, None, 0, stream),
                gb.lobpcg_update(n, X, m, m, C, m, m, 1.0, 0.0, None, 0, out[1], m, TC, 6, stream)]

    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    assert call(st.cuda_stream) == [0, 0, 0]
    torch.cuda.synchronize()
    want = [t.clone() for t in out + small]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        rcs = call(st.cuda_stream)
    assert rcs == [0, 0, 0]
    for t in out + small:
        t.zero_()
    g.replay()
    torch.cuda.synchronize()
    for a, b in zip(out + small, want):
        assert torch.equal(a, b)
