"""Performance cases of the library: the work a user of the LOBPCG solver has
it do, through the public entry points of paper_1704_07458_gb300.

The kinds follow the solver's own steps and its callers:

  solve      lobpcg_solve through Solver: the lowest pairs of a particle in a
             trap (distinct eigenvalues, so that vectors can be compared) from
             a random block to backward error 1e-11
  gram       lobpcg_gram: S^T [A W, B W], the projected pencil's blocks
  update     lobpcg_update: [X, P] = S [C_x, C_p]
  spmm       lobpcg_spmm: A W, with the diagonal-B product where there is a B
  residual   lobpcg_residual: residual, preconditioned block, backward errors
  syev       lobpcg_syev: the projected eigenproblem
  chebyshev  lobpcg_chebyshev_apply: the polynomial preconditioner
  adjoint    lobpcg_eig_adjoint through Solver: gradients of the eigenpairs

Sizes are those of the test, bench and full-size configurations (32^2 grid
k = 8; 64^3 pencil k = 64; 128^3 diffusion k = 256; 512^2 k = 32), with the
block width n_x = k + max(ceil(k / 10), 2) and S = [X, P, W] of 3 n_x columns.
"""
import math

import numpy as np
import torch

import paper_1704_07458_gb300 as gb

F64 = torch.float64
MODES = {"f64": gb.LOBPCG_GEMM_F64, "ozaki": gb.LOBPCG_GEMM_OZAKI,
         "ozaki_tc": gb.LOBPCG_GEMM_OZAKI_TC}
CHEB_INTERVAL = (0.05, 2.0)  # spectrum of D^-1 A of a Dirichlet Laplacian lies in (0, 2)


def listed():
    return [
        # the smallest whole call: 32 x 32 grid, 8 pairs, the default FP64 form;
        # every kernel is small, so launches, host waits and the dense layer count
        dict(name="solve_32x32_k8", kind="solve", nx=32, ny=32, nz=1, op="trap", b="identity",
             k=8, mode="f64"),
        # a generalised 3D pencil (diagonal B) in the tcgen05 form, start to end
        dict(name="solve_48x40x36_k24", kind="solve", nx=48, ny=40, nz=36, op="trap", b="diag",
             k=24, mode="ozaki_tc"),
        # Grams of the smallest and of the benchmark's iteration: p = 3 n_x, q = 2 n_x
        dict(name="gram_1024_30x20", kind="gram", n=1024, p=30, q=20, pad=0, mode="ozaki_tc",
             slices=6),
        dict(name="gram_262144_213x142", kind="gram", n=262144, p=213, q=142, pad=1,
             mode="ozaki_tc", slices=6),
        # basis updates of the benchmark's and of the 128^3, k = 256 iteration
        dict(name="update_262144_213x142", kind="update", n=262144, s=213, m=142, pad=1,
             mode="ozaki_tc", slices=6, y0=False),
        dict(name="update_2097152_846x564", kind="update", n=2097152, s=846, m=564, pad=1,
             mode="ozaki_tc", slices=6, y0=False),
        # A W and B W of the benchmark's iteration; A W of the 128^3 diffusion operator
        dict(name="spmm_64x64x64_m71", kind="spmm", nx=64, ny=64, nz=64, op="laplace", b="diag",
             m=71, pad=1),
        dict(name="spmm_128x128x128_m282", kind="spmm", nx=128, ny=128, nz=128, op="diffusion",
             b="identity", m=282, pad=1),
        # residual step of the benchmark's iteration
        dict(name="residual_262144_m71", kind="residual", n=262144, m=71, c0=0, pad=1, b=True,
             kdiag=True),
        # projected eigenproblem of the benchmark's iteration (n_s = 3 n_x)
        dict(name="syev_213", kind="syev", n=213),
        # preconditioner of degree 8 on the benchmark's block
        dict(name="chebyshev_64x64x64_m71", kind="chebyshev", nx=64, ny=64, nz=64, op="laplace",
             m=71, degree=8),
        # backward pass: 32 pairs of a 512^2 grid, a capped complement solve
        dict(name="adjoint_512x512_k32", kind="adjoint", nx=512, ny=512, k=32, mode="ozaki_tc",
             cg=40),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid3(rng, lo, hi):
    """A 3D grid with between lo and hi points, edges within a factor of two."""
    e = _log(rng, lo, hi) ** (1.0 / 3.0)
    d = [max(4, int(round(e * 2.0 ** rng.uniform(-0.4, 0.4)))) for _ in range(3)]
    while d[0] * d[1] * d[2] > hi:
        d[d.index(max(d))] -= 1
    return d


def draw(rng):
    kind = rng.choice(["solve", "gram", "gram", "update", "update", "spmm", "spmm", "residual",
                       "syev", "syev", "chebyshev", "adjoint"])
    if kind == "solve":
        two = rng.random() < 0.6
        return dict(kind=kind, nx=rng.randint(32, 48), ny=rng.randint(26, 40),
                    nz=1 if two else rng.randint(24, 36), op="trap",
                    b=rng.choice(["identity", "diag"]), k=rng.randint(4, 12 if two else 24),
                    mode=rng.choice(["f64", "ozaki_tc"]) if two else "ozaki_tc")
    if kind in ("gram", "update"):
        n = _log(rng, 1024, 1 << 20)
        w = _log(rng, 10, 282 if n <= 1 << 19 else 120)  # n_x
        mode = "f64" if n * w * w <= 1 << 28 and rng.random() < 0.3 else "ozaki_tc"
        slices = rng.choice([6, 6, 7])
        if kind == "gram":
            return dict(kind=kind, n=n, p=rng.choice([w, 2 * w, 3 * w]), q=rng.choice([w, 2 * w]),
                        pad=rng.choice([0, 1, 5]), mode=mode, slices=slices)
        return dict(kind=kind, n=n, s=rng.choice([w, 2 * w, 3 * w]), m=rng.choice([w, 2 * w]),
                    pad=rng.choice([0, 1, 5]), mode=mode, slices=slices, y0=rng.random() < 0.25)
    if kind in ("spmm", "chebyshev"):
        cheb = kind == "chebyshev"
        if rng.random() < 0.3:
            g = [rng.randint(24, 512), rng.randint(24, 512), 1]
        else:
            g = _grid3(rng, 16384, 262144 if cheb else 2097152)
        m = _log(rng, 4, 96 if cheb else 288)
        c = dict(kind=kind, nx=g[0], ny=g[1], nz=g[2],
                 op=rng.choice(["laplace", "diffusion", "potential"]), m=m)
        if cheb:
            c["op"] = "laplace"
            c["degree"] = rng.randint(2, 12)
        else:
            c["b"] = rng.choice(["identity", "diag"])
            c["pad"] = rng.choice([0, 1, 5])
        return c
    if kind == "residual":
        m = _log(rng, 8, 282)
        return dict(kind=kind, n=_log(rng, 1024, 1 << 20), m=m, c0=rng.choice([0, 0, m // 5]),
                    pad=rng.choice([0, 1, 5]), b=rng.random() < 0.5, kdiag=rng.random() < 0.8)
    if kind == "syev":
        return dict(kind=kind, n=rng.randint(24, 256))
    return dict(kind=kind, nx=rng.randint(96, 512), ny=rng.randint(96, 512), k=rng.randint(4, 40),
                mode=rng.choice(["f64", "ozaki_tc", "ozaki_tc"]), cg=rng.randint(16, 40))


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _ld(width, pad):
    """Leading dimension of a block: pad 1 is the solver's own (a multiple of
    8 doubles), 0 none, other values that many columns more."""
    return -(-width // 8) * 8 if pad == 1 else width + pad


def _block(g, n, width, pad, scale=1.0):
    """Normal n x width block inside n x ld storage (zero padding)."""
    ld = _ld(width, pad)
    full = torch.randn((n, ld), generator=g, dtype=F64, device="cuda")
    full.mul_(scale)
    if ld > width:
        full[:, width:] = 0.0
    return full, ld


def _basis(g, n, width, pad):
    """A block like S = [X, P, W]: columns of norm about 1, the last third (W,
    preconditioned residuals) of norms spread over six decades."""
    full, ld = _block(g, n, width, pad, 1.0 / math.sqrt(n))
    w = width // 3
    if w:
        full[:, width - w:width] *= 10.0 ** (
            -6.0 * torch.rand(w, generator=g, dtype=F64, device="cuda"))
    return full, ld


def _stencil(case, g):
    """CSR of a 5- or 7-point operator on an nx x ny x nz grid, x fastest:
    laplace (constant), potential (Laplacian + diag U[0, 10]), trap (Laplacian
    + an anisotropic harmonic well, off centre, capped at 10), diffusion
    (log-normal face coefficients, Dirichlet walls)."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    n = nx * ny * nz
    idx = torch.arange(n, device="cuda")
    pos = (idx % nx, (idx // nx) % ny, idx // (nx * ny))
    dims = [(nx, 1), (ny, nx), (nz, nx * ny)][:2 if nz == 1 else 3]
    diag = torch.zeros(n, dtype=F64, device="cuda")
    lower, upper = [], []
    for axis, (size, step) in enumerate(dims):
        if case["op"] == "diffusion":
            hi = torch.exp(torch.randn(n, generator=g, dtype=F64, device="cuda"))
            first = torch.exp(torch.randn(n, generator=g, dtype=F64, device="cuda"))
            lo = torch.where(pos[axis] > 0, torch.roll(hi, step), first)
        else:
            hi = lo = torch.ones(n, dtype=F64, device="cuda")
        diag += hi + lo
        lower.append((idx - step, pos[axis] > 0, -lo))
        upper.append((idx + step, pos[axis] < size - 1, -hi))
    if case["op"] == "potential":
        diag += 10.0 * torch.rand(n, generator=g, dtype=F64, device="cuda")
    if case["op"] == "trap":
        u = torch.rand(6, generator=g, dtype=F64, device="cuda").tolist()
        well = torch.zeros_like(diag)
        for axis, (size, _) in enumerate(dims):
            freq = (1.0, 1.27, 1.61)[axis] * (0.97 + 0.06 * u[axis]) * 3.6 / max(nx, ny, nz)
            well += (freq * (pos[axis] - 0.5 * (size - 1) - (u[3 + axis] - 0.5))) ** 2
        diag += well.clamp(max=10.0)
    parts = lower[::-1] + [(idx, torch.ones(n, dtype=torch.bool, device="cuda"), diag)] + upper
    col = torch.stack([p[0] for p in parts], 1)
    keep = torch.stack([p[1] for p in parts], 1)
    val = torch.stack([p[2] for p in parts], 1)
    rowptr = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    rowptr[1:] = torch.cumsum(keep.sum(1), 0).to(torch.int32)
    return n, rowptr, col[keep].to(torch.int32).contiguous(), val[keep].contiguous(), diag


def _bdiag(g, n):
    return 1.0 + torch.rand(n, generator=g, dtype=F64, device="cuda")


def _nx(k):
    return k + max(-(-k // 10), 2)


def _projected(case, seed):
    """A symmetric matrix with the spectrum of a projected pencil: a dense
    lower third and a wide rest, gaps bounded below."""
    g = _gen(seed)
    n = case["n"]
    u = torch.rand(n, generator=g, dtype=F64, device="cuda")
    t = (torch.arange(n, dtype=F64, device="cuda") + 0.8 * u) / n
    w = 12.0 * t * (0.1 + 0.9 * t)
    q, _ = torch.linalg.qr(torch.randn((n, n), generator=g, dtype=F64, device="cuda"))
    h = (q * w) @ q.T
    return 0.5 * (h + h.T)


def _fix_signs(v):
    """Rows of v (eigenvectors) with their largest entry positive, the rule
    that lobpcg_solve applies to its vectors."""
    big = v.gather(1, v.abs().argmax(1, keepdim=True))
    return v * torch.sign(big)


def _grid_modes(case, seed):
    """The k lowest eigenpairs of a_x Tx + a_y Ty on an nx x ny grid in closed
    form, and the two coefficients."""
    g = _gen(seed)
    nx, ny, k = case["nx"], case["ny"], case["k"]
    ax, ay = (0.6 + 0.8 * torch.rand(2, generator=g, dtype=F64, device="cuda")).tolist()
    kx, ky = np.arange(1, nx + 1), np.arange(1, ny + 1)
    lx = ax * 4.0 * np.sin(np.pi * kx / (2 * (nx + 1))) ** 2
    ly = ay * 4.0 * np.sin(np.pi * ky / (2 * (ny + 1))) ** 2
    tot = (lx[None, :] + ly[:, None]).ravel()
    order = np.argsort(tot, kind="stable")[:k]
    vx = torch.from_numpy(np.sqrt(2.0 / (nx + 1)) * np.sin(
        np.pi * np.outer(kx, order % nx + 1) / (nx + 1))).cuda()
    vy = torch.from_numpy(np.sqrt(2.0 / (ny + 1)) * np.sin(
        np.pi * np.outer(ky, order // nx + 1) / (ny + 1))).cuda()
    x = (vy[:, None, :] * vx[None, :, :]).reshape(nx * ny, k).contiguous()
    return g, ax, ay, torch.from_numpy(tot[order]).cuda(), x


def _grid_csr(nx, ny, ax, ay):
    n, rowptr, col, val, _ = _stencil(dict(nx=nx, ny=ny, nz=1, op="laplace"), None)
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), rowptr[1:] - rowptr[:-1])
    off = (col.long() - rows).abs()
    one = torch.ones((), dtype=F64, device="cuda")
    return n, rowptr, col, torch.where(off == 0, 2.0 * (ax + ay) * one,
                                       torch.where(off == 1, -ax * one, -ay * one)).contiguous()


def prepare(case, seed):
    s = dict(case)
    kind = case["kind"]
    if kind == "adjoint":
        g, ax, ay, lam, x = _grid_modes(case, seed)
        nx, ny, k = case["nx"], case["ny"], case["k"]
        n, rowptr, col, val = _grid_csr(nx, ny, ax, ay)
        s["solver"] = gb.Solver(gemm_mode=case["mode"])
        s["solver"].set_operator(rowptr, col, val)
        s["csr"], s["lam"], s["X"] = (rowptr, col, val), lam, x
        s["glam"] = torch.randn(k, generator=g, dtype=F64, device="cuda")
        s["G"] = torch.randn((n, k), generator=g, dtype=F64, device="cuda")
        return s
    if kind == "syev":
        s["A"] = _projected(case, seed)
        s["V"] = torch.empty_like(s["A"])
        s["w"] = torch.empty(case["n"], dtype=F64, device="cuda")
        return s
    g = _gen(seed)
    if kind == "solve":
        n, rowptr, col, val, _ = _stencil(case, g)
        b = _bdiag(g, n) if case["b"] == "diag" else None
        s["X0"] = torch.randn((n, _nx(case["k"])), generator=g, dtype=F64, device="cuda")
        s["solver"] = gb.Solver(gemm_mode=case["mode"])
        s["solver"].set_operator(rowptr, col, val, b_diag=b)
        s["csr"], s["n"], s["b"] = (rowptr, col, val), n, b
    elif kind == "gram":
        n, p, q = case["n"], case["p"], case["q"]
        s["U"], s["ldu"] = _basis(g, n, p, case["pad"])
        s["V"], s["ldv"] = _basis(g, n, q, case["pad"])
        s["G"] = torch.empty((q, p), dtype=F64, device="cuda")
        s["mode"] = MODES[case["mode"]]
        size = gb.lobpcg_gram_workspace(n, p, q, s["mode"], case["slices"])
        s["work"] = torch.empty(max(size, 16), dtype=torch.uint8, device="cuda")
    elif kind == "update":
        n, w, m = case["n"], case["s"], case["m"]
        s["S"], s["lds"] = _basis(g, n, w, case["pad"])
        s["C"] = torch.randn((m, w), generator=g, dtype=F64, device="cuda") / math.sqrt(w)
        s["Y0"], s["ldy"] = (_block(g, n, m, case["pad"], 1.0 / math.sqrt(n)) if case["y0"]
                             else (None, _ld(m, case["pad"])))
        s["Y"] = torch.zeros((n, s["ldy"]), dtype=F64, device="cuda")
        s["mode"] = MODES[case["mode"]]
    elif kind == "spmm":
        n, rowptr, col, val, _ = _stencil(case, g)
        s["csr"], s["n"] = (rowptr, col, val), n
        s["b"] = _bdiag(g, n) if case["b"] == "diag" else None
        s["X"], s["ld"] = _block(g, n, case["m"], case["pad"], 1.0 / math.sqrt(n))
        s["Y"] = torch.zeros_like(s["X"])
        s["BY"] = torch.zeros_like(s["X"]) if s["b"] is not None else None
    elif kind == "residual":
        n, m = case["n"], case["m"]
        s["X"], s["ld"] = _block(g, n, m, case["pad"], 1.0 / math.sqrt(n))
        s["theta"] = 0.5 + torch.rand(m, generator=g, dtype=F64, device="cuda")
        s["BX"] = s["X"] * _bdiag(g, n)[:, None] if case["b"] else None
        bx = s["BX"] if case["b"] else s["X"]
        s["AX"] = bx.clone()  # A X = B X Theta + residuals of norm about 1e-3
        s["AX"][:, :m] *= s["theta"]
        s["AX"][:, :m] += (1e-3 / math.sqrt(n)) * torch.randn((n, m), generator=g, dtype=F64,
                                                              device="cuda")
        s["kdiag"] = (6.0 * _bdiag(g, n)) if case["kdiag"] else None
        wide = m - case["c0"]
        s["ldw"] = _ld(wide, case["pad"])
        s["W"] = torch.zeros((n, s["ldw"]), dtype=F64, device="cuda")
        s["be"] = torch.empty(wide, dtype=F64, device="cuda")
    elif kind == "chebyshev":
        n, rowptr, col, val, diag = _stencil(case, g)
        s["n"], s["csr"] = n, (rowptr, col, val, diag)
        s["cheb"] = Chebyshev(n, rowptr, col, val, diag, case["degree"], case["m"])
        s["R"], s["ld"] = _block(g, n, case["m"], 1, 1.0 / math.sqrt(n))
        s["W"] = torch.zeros_like(s["R"])
    return s


class Chebyshev:
    """Owns a lobpcg_chebyshev object."""

    def __init__(self, n, rowptr, col, val, diag, degree, cols):
        self.h = gb.lobpcg_chebyshev_create(n, rowptr, col, val, diag, degree, *CHEB_INTERVAL,
                                            cols)

    def __del__(self):
        gb.lobpcg_chebyshev_destroy(self.h)


# -------------------------------------------------------------------- passes

def _ok(rc):
    if rc != gb.LOBPCG_OK:
        raise RuntimeError(f"status {rc}")


def run(s):
    kind = s["kind"]
    if kind == "solve":
        lam, x, _, _, _ = s["solver"].solve(s["k"], tol=1e-11, X0=s["X0"], device=True)
        return {"lam": lam, "X": x}
    if kind == "gram":
        _ok(gb.lobpcg_gram(s["n"], s["U"], s["ldu"], s["p"], s["V"], s["ldv"], s["q"], s["G"],
                           s["p"], s["mode"], s["slices"], s["work"], s["work"].numel()))
        return {"G": s["G"]}
    if kind == "update":
        y0 = s["Y0"]
        _ok(gb.lobpcg_update(s["n"], s["S"], s["lds"], s["s"], s["C"], s["s"], s["m"], 1.0,
                             0.0 if y0 is None else 1.0, y0, s["ldy"], s["Y"], s["ldy"], s["mode"],
                             s["slices"]))
        return {"Y": s["Y"]}
    if kind == "spmm":
        rowptr, col, val = s["csr"]
        _ok(gb.lobpcg_spmm(s["n"], rowptr, col, val, s["X"], s["ld"], s["m"], s["Y"], s["ld"],
                           s["b"], s["BY"], s["ld"] if s["b"] is not None else 0))
        return {"Y": s["Y"], "BY": s["BY"]}
    if kind == "residual":
        _ok(gb.lobpcg_residual(s["n"], s["X"], s["AX"], s["BX"], s["ld"], s["m"], s["c0"],
                               s["theta"], s["kdiag"], s["W"], s["ldw"], 12.0, 2.0, s["be"]))
        return {"W": s["W"], "be": s["be"]}
    if kind == "syev":
        s["V"].copy_(s["A"])
        _ok(gb.lobpcg_syev(s["n"], s["V"], s["n"], s["w"], 2))
        return {"w": s["w"], "V": _fix_signs(s["V"])}
    if kind == "chebyshev":
        _ok(gb.lobpcg_chebyshev_apply(s["cheb"].h, s["n"], s["m"], s["R"], s["ld"], s["W"],
                                      s["ld"]))
        return {"W": s["W"]}
    ga, _, _, _ = s["solver"].adjoint(s["k"], s["lam"], s["X"], s["glam"], s["G"],
                                      cg_maxit=s["cg"])
    return {"gA": ga}


# ----------------------------------------------------------------- the work

def _depth(case):
    return case.get("nz", 1)


def _nnz(case):
    nx, ny, nz = case["nx"], case["ny"], _depth(case)
    n = nx * ny * nz
    return n, n + 2 * (3 * n - ny * nz - nx * nz - nx * ny) if nz > 1 else \
        n + 2 * (2 * n - ny - nx)


def work(case):
    kind = case["kind"]
    if kind == "gram":
        n, p, q = case["n"], case["p"], case["q"]
        return {"bytes": 8 * (n * (p + q) + p * q), "flops": 2 * n * p * q}
    if kind == "update":
        n, w, m = case["n"], case["s"], case["m"]
        return {"bytes": 8 * (n * (w + m * (2 if case["y0"] else 1)) + w * m),
                "flops": 2 * n * w * m}
    if kind == "spmm":
        n, nnz = _nnz(case)
        m, b = case["m"], case["b"] == "diag"
        return {"bytes": 12 * nnz + 4 * (n + 1) + 16 * n * m + (8 * n * (m + 1) if b else 0),
                "flops": 2 * nnz * m + (n * m if b else 0)}
    if kind == "residual":
        n, mm = case["n"], case["m"] - case["c0"]
        return {"bytes": 8 * n * (mm * (4 if case["b"] else 3) + (1 if case["kdiag"] else 0)),
                "flops": 7 * n * mm}
    if kind == "syev":
        n = case["n"]
        return {"bytes": 16 * n * n, "flops": 9 * n ** 3}
    if kind == "chebyshev":
        n, nnz = _nnz(case)
        m, d = case["m"], case["degree"]
        return {"bytes": 12 * nnz + 4 * (n + 1) + 16 * n * m + 8 * n,
                "flops": (d - 1) * (2 * nnz + 6 * n) * m}
    n, nnz = _nnz(case)
    k = case["k"]
    if kind == "adjoint":
        # per CG step: one product, one projection (Gram and update), ten
        # passes over n x k blocks that a step's dot products separate
        return {"bytes": case["cg"] * (12 * nnz + 80 * n * k) + 8 * nnz + 16 * n * k,
                "flops": case["cg"] * (2 * nnz * k + 4 * n * k * k + 14 * n * k) + 4 * nnz * k}
    # solve: per iteration (about 75 in 2D, 140 in 3D) one product, the Gram of
    # the new columns, the update of [X, P] and [A X, A P], the residual
    w, it = _nx(k), 75 if _depth(case) == 1 else 140
    return {"bytes": it * (12 * nnz + 8 * n * w * (2 + 5 + 10 + 4)) + 16 * n * w,
            "flops": it * (2 * nnz * w + 2 * n * 3 * w * 2 * w * 3 + 9 * (3 * w) ** 3)}


# ------------------------------------------------- the same in 64 bits, plain

def _csr_mm(csr, x, n):
    a = torch.sparse_csr_tensor(csr[0].long(), csr[1].long(), csr[2], size=(n, n))
    return a @ x


def _padded(y, width):
    """y inside rows of ld columns, zero in the padding."""
    full = torch.zeros((y.shape[0], width), dtype=F64, device="cuda")
    full[:, :y.shape[1]] = y
    return full


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve" and _nnz(case)[0] > 4096:
        return None  # a dense eigensolver takes too long
    s = prepare(case, seed)
    if kind == "solve":
        n, k = s["n"], case["k"]
        d = torch.ones(n, dtype=F64, device="cuda") if s["b"] is None else s["b"] ** -0.5
        a = torch.sparse_csr_tensor(*(t.long() for t in s["csr"][:2]), s["csr"][2],
                                    size=(n, n)).to_dense()
        w, v = torch.linalg.eigh(d[:, None] * a * d)
        x = _fix_signs((d[:, None] * v[:, :k]).T.contiguous())
        return {"lam": w[:k].clone(), "X": x.T.contiguous()}
    if kind == "gram":
        return {"G": s["V"][:, :case["q"]].T @ s["U"][:, :case["p"]]}
    if kind == "update":
        y = s["S"][:, :case["s"]] @ s["C"].T
        if s["Y0"] is not None:
            y += s["Y0"][:, :case["m"]]
        return {"Y": _padded(y, s["ldy"])}
    if kind == "spmm":
        x = s["X"][:, :case["m"]].contiguous()
        by = None if s["b"] is None else _padded(s["b"][:, None] * x, s["ld"])
        return {"Y": _padded(_csr_mm(s["csr"], x, s["n"]), s["ld"]), "BY": by}
    if kind == "residual":
        c0, m = case["c0"], case["m"]
        x, ax, th = s["X"][:, c0:m], s["AX"][:, c0:m], s["theta"][c0:]
        r = ax - (s["BX"][:, c0:m] if case["b"] else x) * th
        be = r.norm(dim=0) / ((12.0 + 2.0 * th.abs()) * x.norm(dim=0))
        w = r if s["kdiag"] is None else r / s["kdiag"][:, None]
        return {"W": _padded(w, s["ldw"]), "be": be}
    if kind == "syev":
        w, v = torch.linalg.eigh(s["A"])
        return {"w": w, "V": _fix_signs(v.T.contiguous())}
    if kind == "chebyshev":
        # Saad, Iterative Methods for Sparse Linear Systems, Algorithm 12.1
        n, m = s["n"], case["m"]
        csr, dinv = s["csr"], 1.0 / s["csr"][3][:, None]
        lo, hi = CHEB_INTERVAL
        theta, delta = 0.5 * (hi + lo), 0.5 * (hi - lo)
        sigma = theta / delta
        rho = 1.0 / sigma
        r = s["R"][:, :m]
        d = r * dinv / theta
        w = d.clone()
        for _ in range(1, case["degree"]):
            z = (r - _csr_mm(csr, w, n)) * dinv
            new = 1.0 / (2.0 * sigma - rho)
            d = new * rho * d + (2.0 * new / delta) * z
            w, rho = w + d, new
        return {"W": _padded(w, s["ld"])}
    return _exact_adjoint(case, s)


def _exact_adjoint(case, s):
    """First-order perturbation theory with `cg` steps of the projected,
    Jacobi-preconditioned conjugate gradient for the complement."""
    lam, x, g, n, k = s["lam"], s["X"], s["G"], s["X"].shape[0], case["k"]
    rowptr, col, val = s["csr"]
    dinv = 1.0 / val.max()  # the constant diagonal
    m = x.T @ g
    gap = lam[None, :] - lam[:, None]
    cin = torch.where(gap != 0, m / torch.where(gap != 0, gap, torch.ones_like(gap)),
                      torch.zeros_like(gap))
    r = g - x @ m
    u = torch.zeros_like(g)
    z = r * dinv
    z -= x @ (x.T @ z)
    p, rz = z.clone(), (r * z).sum(0)
    for _ in range(case["cg"]):
        q = _csr_mm((rowptr, col, val), p, n) - p * lam
        a = rz / (p * q).sum(0)
        u += a * p
        r = r - a * q
        z = r * dinv
        z -= x @ (x.T @ z)
        new = (r * z).sum(0)
        p = z + (new / rz) * p
        rz = new
    w = x @ cin - u
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), (rowptr[1:] - rowptr[:-1]))
    c = col.long()
    out = torch.empty(len(c), dtype=F64, device="cuda")
    for a in range(0, len(c), 1 << 18):
        i, j = rows[a:a + (1 << 18)], c[a:a + (1 << 18)]
        out[a:a + (1 << 18)] = (x[i] * x[j] * s["glam"] + 0.5 * (w[i] * x[j] + x[i] * w[j])).sum(1)
    return {"gA": out}
