"""Performance cases of the columnwise setup, the preconditioner apply, the
solvers and the W-pattern generators, through the package's public calls.

Operators are the repository's synthetic ones (upwind convection-diffusion on
N^2, complex shifted Helmholtz on N^2, lognormal diffusion-convection on N^3,
the random power-law matrix), assembled here on the GPU from a seed: the seed
draws the velocities, the wavenumber, the coefficient field or the values, so
another seed is another problem of the same structure.

  setup      factor(A, PW, ...), then (apply = True) the first y = W V^-1 x on
             the new factors, which also lays them out for the solves
  apply      y = W V^-1 x on factors that were applied before (one call of a
             Krylov iteration)
  gmres      restarted GMRES(50) with the preconditioner, from A, W, V to x
  sparsified the W pattern by sparsified powers with dropping by count
  propose    the learned W pattern: features, scores, selection
  train      one training step of the proposal network (gradient and Adam)

exact() restates each in plain torch and FP64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1208_3573_gb300 import diaf, learned

DEV = "cuda"
BLOCK = 64  # rows per diagonal block of a block-diagonal V


def listed():
    return [
        # the smallest setup: 1,024 columns, host latency and launches (the 32^2 configuration)
        dict(name="setup_convdiff32", kind="setup", op="convdiff", size=32, wpower=1, alg="S", prec="mixed32", apply=True),
        # the headline configuration: W on pattern(A^2), setup and the first apply
        dict(name="setup_convdiff256", kind="setup", op="convdiff", size=256, wpower=2, alg="S", prec="mixed32",
             apply=True),
        # the other algorithm (unit v_j) at an odd grid size
        dict(name="setup_convdiff181_q", kind="setup", op="convdiff", size=181, wpower=2, alg="Q", prec="mixed32",
             apply=True),
        # factor()'s default precision, plain FP64
        dict(name="setup_convdiff129_fp64", kind="setup", op="convdiff", size=129, wpower=2, alg="S", prec="fp64",
             apply=True),
        # complex values, 262,144 columns of 9 entries (the Helmholtz configuration)
        dict(name="setup_helmholtz512", kind="setup", op="helmholtz", size=512, wpower=1, alg="S", prec="mixed32",
             apply=True),
        # 262,144 columns of 25 entries with the block-diagonal V that converges on this operator
        # (8 entries per column in blocks of 64 rows)
        dict(name="setup_lognormal64", kind="setup", op="lognormal", size=64, wpower=2, alg="S", prec="mixed32",
             apply=True),
        # uneven tiles, up to 60 columns and several hundred rows (the power-law configuration; setup only, its V can
        # be singular)
        dict(name="setup_powerlaw200k", kind="setup", op="powerlaw", size=200_000, wpower=1, alg="S", prec="mixed32",
             apply=False),
        # one preconditioner application inside a solve: 512 levels of a triangular V
        dict(name="apply_convdiff256", kind="apply", op="convdiff", size=256, wpower=2),
        # a whole complex solve, the Helmholtz configuration's solver
        dict(name="gmres_helmholtz150", kind="gmres", op="helmholtz", size=150, wpower=1),
        # the fixed rule for the W pattern at 12 entries per column
        dict(name="sparsified_lognormal64", kind="sparsified", op="lognormal", size=64, keep=12),
        # the learned rule on one operator of the size it is trained on
        dict(name="propose_lognormal40", kind="propose", op="lognormal", size=40, keep=12),
        # one step of its training loop at the default batch: the shortest call
        dict(name="train_8192", kind="train", rows=8192),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["setup", "setup", "setup", "setup", "setup", "apply", "gmres", "sparsified", "propose", "train"])
    if kind == "setup":
        op = rng.choice(["convdiff", "convdiff", "convdiff", "helmholtz", "lognormal", "powerlaw"])
        if op == "convdiff":
            prec = rng.choice(["mixed32", "mixed32", "fp64"])
            return dict(kind=kind, op=op, size=_log_int(rng, 32, 256 if prec == "mixed32" else 129),
                        wpower=rng.choice([1, 2, 2]), alg=rng.choice(["S", "Q"]), prec=prec, apply=True)
        if op == "helmholtz":
            return dict(kind=kind, op=op, size=_log_int(rng, 40, 511), wpower=1, alg="S", prec="mixed32", apply=True)
        if op == "lognormal":
            return dict(kind=kind, op=op, size=_log_int(rng, 16, 63), wpower=2, alg="S", prec="mixed32", apply=True)
        return dict(kind=kind, op=op, size=_log_int(rng, 6_000, 199_999), wpower=1, alg="S", prec="mixed32",
                    apply=False)
    if kind == "apply":
        return dict(kind=kind, op="convdiff", size=_log_int(rng, 32, 255), wpower=rng.choice([1, 2]))
    if kind == "gmres":
        return dict(kind=kind, op="helmholtz", size=_log_int(rng, 40, 149), wpower=1)
    if kind == "sparsified":
        return dict(kind=kind, op="lognormal", size=_log_int(rng, 16, 63), keep=rng.choice([8, 12, 16]))
    if kind == "propose":
        return dict(kind=kind, op="lognormal", size=_log_int(rng, 16, 63), keep=rng.choice([8, 12, 16]))
    return dict(kind=kind, rows=_log_int(rng, 1_000, 65_536))


# ---------------------------------------------------------------- operators
def _gen(seed, device=DEV):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed) & 0x7FFFFFFFFFFF)
    return g


def _grid(N, dim):
    p = torch.arange(N**dim, device=DEV, dtype=torch.int64)
    return p, [p % N, (p // N) % N, p // (N * N)][:dim]


def _offsets(dim, reach, box):
    """Grid offsets of a stencil in ascending index order: |d|_1 <= reach, or max |d| <= reach for a box."""
    r = range(-reach, reach + 1)
    o = [(dx, dy, dz) for dz in (r if dim == 3 else (0,)) for dy in r for dx in r]
    return [d[:dim] for d in o if (max(map(abs, d)) if box else sum(map(abs, d))) <= reach]


def _stencil_pattern(N, dim, offs):
    """Column pointers, row indices and the [n, offsets] mask of a stencil pattern (row = column + offset)."""
    p, xyz = _grid(N, dim)
    rows, mask = [], []
    for d in offs:
        ok = torch.ones_like(p, dtype=torch.bool)
        r = p.clone()
        for a, (x, s) in enumerate(zip(xyz, d)):
            ok &= (x + s >= 0) & (x + s < N)
            r += s * N**a
        rows.append(r)
        mask.append(ok)
    mask = torch.stack(mask, 1)
    rowidx = torch.stack(rows, 1)[mask].to(torch.int32)
    colptr = torch.zeros(p.numel() + 1, dtype=torch.int32, device=DEV)
    colptr[1:] = torch.cumsum(mask.sum(1), 0).to(torch.int32)
    return colptr, rowidx, mask


def _stencil_matrix(N, dim, offs, coeff, dtype):
    """CSC of a stencil operator; coeff(d, columns, inside) are the entries A(p + d, p)."""
    colptr, rowidx, mask = _stencil_pattern(N, dim, offs)
    p = torch.arange(N**dim, device=DEV)
    vals = torch.stack([coeff(d, p, mask[:, i]).to(dtype) for i, d in enumerate(offs)], 1)[mask]
    return diaf.DeviceCSC(N**dim, colptr, rowidx, vals)


def _convdiff(N, g):
    h = 1.0 / (N + 1)
    u = torch.rand(2, generator=g, device=DEV, dtype=torch.float64)
    b1, b2 = (10.0 * 2.0 ** (u[0] - 0.5)).item(), (5.0 * 2.0 ** (u[1] - 0.5)).item()
    # entry of row p + d for column p: the coupling of that row to its neighbour at -d
    c = {(0, 0): 4 / h**2 + b1 / h + b2 / h, (1, 0): -1 / h**2 - b1 / h, (0, 1): -1 / h**2 - b2 / h,
         (-1, 0): -1 / h**2, (0, -1): -1 / h**2}
    return _stencil_matrix(N, 2, _offsets(2, 1, False),
                           lambda d, p, ok: torch.full_like(p, c[d], dtype=torch.float64), torch.float64)


def _helmholtz(N, g):
    h = 1.0 / (N + 1)
    u = torch.rand(1, generator=g, device=DEV, dtype=torch.float64).item()
    k = 2.0 * math.pi / ((9.5 + u) * h)  # about ten points per wavelength
    s = 1.0 / (6.0 * h * h)
    c = {0: 20.0 * s - (k * k + 0.5j * k * k), 1: -4.0 * s, 2: -1.0 * s}
    return _stencil_matrix(N, 2, _offsets(2, 1, True),
                           lambda d, p, ok: torch.full_like(p, c[abs(d[0]) + abs(d[1])], dtype=torch.complex128),
                           torch.complex128)


def _lognormal(N, g):
    h, conv = 1.0 / (N + 1), (20.0, 0.0, 0.0)
    z = torch.randn((N, N, N), generator=g, device=DEV, dtype=torch.float64)
    f = torch.fft.fftfreq(N, device=DEV, dtype=torch.float64)
    gauss = torch.exp(-2.0 * (math.pi * f * 8.0) ** 2)  # a Gaussian of 8 cells, periodic
    z = torch.fft.ifftn(torch.fft.fftn(z) * gauss[:, None, None] * gauss[None, :, None] * gauss[None, None, :]).real
    kap = torch.exp(1.5 * (z - z.mean()) / z.std()).reshape(-1)
    p, xyz = _grid(N, 3)
    diag = torch.zeros(N**3, dtype=torch.float64, device=DEV)
    for a in range(3):
        for s in (-1, 1):
            ok = (xyz[a] + s >= 0) & (xyz[a] + s < N)
            kq = kap[torch.where(ok, p + s * N**a, p)]
            diag += 2.0 * kap * kq / (kap + kq) / h**2
            if s == -1:
                diag += conv[a] / h

    def coeff(d, q, ok):
        if d == (0, 0, 0):
            return diag
        a = next(i for i in range(3) if d[i])
        r = torch.where(ok, q + d[a] * N**a, q)
        v = -2.0 * kap[r] * kap[q] / (kap[r] + kap[q]) / h**2
        return v - conv[a] / h if d[a] == 1 else v  # row upwind of its column

    return _stencil_matrix(N, 3, _offsets(3, 1, False), coeff, torch.float64)


def _powerlaw(n, g):
    """The structure goes with n (so do nnz(W) and nnz(V)); the seed draws the values."""
    values, g = g, _gen(n)
    d = torch.arange(3, 61, device=DEV)
    p = d.double() ** -2.2
    off = d[torch.multinomial(p / p.sum(), n, replacement=True, generator=g)] - 1
    col = torch.repeat_interleave(torch.arange(n, device=DEV), off)
    row = torch.randint(0, n - 1, col.shape, generator=g, device=DEV)
    key = torch.unique(col * n + row + (row >= col))
    while key.numel() < col.numel():  # duplicates within a column: drawn again
        short = off - torch.bincount(key // n, minlength=n)
        c = torch.repeat_interleave(torch.arange(n, device=DEV), short)
        r = torch.randint(0, n - 1, c.shape, generator=g, device=DEV)
        key = torch.unique(torch.cat([key, c * n + r + (r >= c)]))
    v = torch.randn(key.numel(), generator=values, device=DEV, dtype=torch.float64)
    diag = 1.2 * torch.segment_reduce(v.abs(), "sum", lengths=off)
    j = torch.arange(n, device=DEV)
    key, order = torch.sort(torch.cat([key, j * n + j]))
    vals = torch.cat([v, diag])[order]
    colptr = torch.zeros(n + 1, dtype=torch.int32, device=DEV)
    colptr[1:] = torch.cumsum(off + 1, 0).to(torch.int32)
    return diaf.DeviceCSC(n, colptr, (key % n).to(torch.int32), vals)


def _operator(case, g):
    return {"convdiff": _convdiff, "helmholtz": _helmholtz, "lognormal": _lognormal,
            "powerlaw": _powerlaw}[case["op"]](case["size"], g)


def _power_pattern(case, A, power):
    """pattern(A^power), with arrays of its own."""
    if power == 1:
        return diaf.DeviceCSC(A.n, A.colptr.clone(), A.rowidx.clone())
    dim = 3 if case["op"] == "lognormal" else 2
    cp, ri, _ = _stencil_pattern(case["size"], dim, _offsets(dim, power, False))
    return diaf.DeviceCSC(A.n, cp, ri)


def _upper_budget(A):
    """Entries of the upper triangle of pattern(A) per column, the diagonal counted."""
    col = torch.repeat_interleave(torch.arange(A.n, device=DEV), A.colptr.diff().long())
    return (torch.bincount(col[A.rowidx < col], minlength=A.n) + 1).to(torch.int32)


def _vspec(case, A):
    if case["op"] == "lognormal":
        return dict(vrule=diaf.RULE_BLOCK, budget=torch.full((A.n,), 8, dtype=torch.int32, device=DEV),
                    blocks=diaf.contiguous_blocks(A.n, BLOCK))
    return dict(vrule=diaf.RULE_UPPER, budget=_upper_budget(A),
                tie_tol=1e-3 if case["op"] == "helmholtz" else 1e-9)


def _spmv(A, x):
    """A x, summed in a fixed order."""
    col = torch.repeat_interleave(torch.arange(A.n, device=DEV), A.colptr.diff().long())
    row, order = torch.sort(A.rowidx.long(), stable=True)
    p = (A.vals * x[col])[order]
    parts = torch.view_as_real(p) if p.is_complex() else p[:, None]
    y = torch.segment_reduce(parts.contiguous(), "sum", lengths=torch.bincount(row, minlength=A.n), axis=0)
    return torch.view_as_complex(y) if p.is_complex() else y[:, 0]


# ---------------------------------------------------------------- the user's side
def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "train":
        feat = torch.randn((case["rows"], diaf.PROP_NFEAT), generator=g, device=DEV)
        feat[:, 0] = (feat[:, 0] > 1.5).float()  # the indicator and ratio features keep their ranges
        feat[:, 1] = (feat[:, 1] > 0.5).float()
        feat[:, 2:4] = feat[:, 2:4].abs().clamp(max=3.0) / 3.0
        feat[:, 7] = torch.sign(feat[:, 7])
        target = torch.randn(case["rows"], generator=g, device=DEV)
        params = torch.from_numpy(learned.init_params(int(seed) & 0x7FFFFFFF)).to(DEV)
        return dict(case=case, feat=feat, target=target, params=params, m=torch.zeros_like(params),
                    v=torch.zeros_like(params), grad=torch.empty_like(params), loss=torch.empty(1, device=DEV), step=0)
    A = _operator(case, g)
    st = dict(case=case, A=A)
    if kind == "sparsified":
        return st
    if kind == "propose":
        st.update(CAND=_power_pattern(case, A, 2),
                  net=learned.Proposer(learned.init_params(int(seed) & 0x7FFFFFFF)))
        return st
    st.update(PW=_power_pattern(case, A, case["wpower"]), spec=_vspec(case, A))
    st["x"] = torch.randn(A.n, generator=g, device=DEV, dtype=A.vals.dtype)
    if kind in ("apply", "gmres"):
        st["F"] = diaf.factor(A, st["PW"], alg="S", **st["spec"])
        st["F"].apply(st["x"])
    if kind == "gmres":
        st["b"] = _spmv(A, torch.ones_like(st["x"]) + 0.1 * st["x"])
        st["solver"] = diaf.Solver(A)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "setup":
        F = diaf.factor(st["A"], st["PW"], alg=case["alg"], prec=case["prec"], **st["spec"])
        out = dict(W=F.W.vals, V_colptr=F.V.colptr, V_rowidx=F.V.rowidx, V=F.V.vals, res=F.res, flags=F.flags)
        if case["apply"]:
            out["y"] = F.apply(st["x"])
        return out
    if kind == "apply":
        return dict(y=st["F"].apply(st["x"]))
    if kind == "gmres":
        x, info = st["solver"].gmres(st["b"], st["F"], tol=1e-6, restart=50)
        return dict(x=x, iterations=int(info.iterations), relres=float(info.relres))
    if kind == "sparsified":
        P = diaf.sparsified_powers(st["A"], 2, 0, case["keep"])
        return dict(colptr=P.colptr, rowidx=P.rowidx)
    if kind == "propose":
        scores = st["net"].scores(st["A"], st["CAND"])
        P = diaf.propose_select(st["CAND"], scores, case["keep"])
        return dict(scores=scores, colptr=P.colptr, rowidx=P.rowidx)
    diaf.mlp_grad(st["params"], st["feat"], st["target"], st["grad"], st["loss"])
    st["step"] += 1
    diaf.mlp_adam(st["params"], st["grad"], st["m"], st["v"], st["step"], 3e-3)
    return dict(grad=st["grad"], loss=st["loss"], params=st["params"], m=st["m"], v=st["v"])


# ---------------------------------------------------------------- what a pass cannot do without
def _tile_sizes(case):
    """(share of the columns, nnz(A(:,j)), k, m, l, real flops per multiply-add pair / 2) of typical columns."""
    if case["op"] == "powerlaw":
        d = np.arange(3, 61)
        p = d**-2.2 / (d**-2.2).sum()
        mean = float((p * d).sum())
        return [(float(q), float(e), float(e), e * mean - (e - 1), (e - 1) / 2 + 1, 1) for q, e in zip(p, d)]
    if case["op"] == "helmholtz":
        return [(1.0, 9, 9, 25, 5, 4)]
    if case["op"] == "convdiff":
        return [(1.0, 5, 13, 25, 3, 1)] if case["wpower"] == 2 else [(1.0, 5, 5, 13, 3, 1)]
    return [(1.0, 7, 25, 63, 8, 1)]


def work(case):
    kind = case["kind"]
    if kind == "train":
        r, p = case["rows"], diaf.PROP_NPARAM
        return dict(bytes=4 * r * 9 + 4 * p * (4 + 4), flops=6.0 * p * r)
    n = case["size"] ** {"convdiff": 2, "helmholtz": 2, "lognormal": 3, "powerlaw": 1}[case["op"]]
    sizes = _tile_sizes(dict(case, wpower=case.get("wpower", 2)))
    mean = lambda f: float(sum(s[0] * f(*s[1:]) for s in sizes))  # noqa: E731
    nnza = n * mean(lambda e, k, m, l, c: e)
    nnzw = n * mean(lambda e, k, m, l, c: k)
    nnzv = n * mean(lambda e, k, m, l, c: l)
    cplx = sizes[0][5]
    vb = 16 if cplx == 4 else 8
    csc = lambda nnz, b: nnz * (4 + b) + 4 * n  # noqa: E731
    if kind == "sparsified":
        return dict(bytes=csc(nnza, vb) + 4 * n * (case["keep"] + 1), flops=2 * nnza * 7)
    if kind == "propose":
        return dict(bytes=csc(nnza, vb) + csc(nnzw, 0) + 4 * nnzw + 4 * n * (case["keep"] + 1),
                    flops=2 * nnza * 7 + 2.0 * diaf.PROP_NPARAM * nnzw)
    apply = dict(bytes=csc(nnzw, vb) + csc(nnzv, vb) + 2 * vb * n, flops=2 * cplx * (nnzw + nnzv))
    if kind == "apply":
        return apply
    if kind == "gmres":  # about one iteration per grid line; the basis is read twice on average
        its = 0.6 * case["size"]
        return dict(bytes=its * (apply["bytes"] + csc(nnza, vb) + 2 * 25 * vb * n),
                    flops=its * (apply["flops"] + 2 * cplx * nnza + 4 * 25 * 2 * cplx * n))
    # QR of the tile, its row norms, QR of the rows outside I_j, the smallest (largest) singular pair, v, w, residual
    col = lambda e, k, m, l, c: c * (2 * k * k * (m - k / 3) + m * k * k + 2 * k * k * (max(m - l, k) - k / 3)  # noqa: E731
                                     + 8 * k * k + 6 * m * k)
    w = dict(bytes=csc(nnza, vb) + csc(nnzw, 0) + nnzw * vb + csc(nnzv, vb) + 12 * n, flops=n * mean(col))
    if case["apply"]:
        w = dict(bytes=w["bytes"] + 2 * vb * n, flops=w["flops"] + apply["flops"])
    return w


# ---------------------------------------------------------------- the same in plain torch, 64 bits
def _csc_parts(A):
    return A.n, A.colptr.long(), A.rowidx.long(), A.vals


def _tiles(cols, n, Acp, Ari, Av, Pcp, Pri):
    """The tiles A(R_j, J_j) of some columns, padded to [B, M, K], with R_j (-1 beyond m_j) and k_j."""
    k = Pcp[cols + 1] - Pcp[cols]
    K = int(k.max())
    b = torch.repeat_interleave(torch.arange(cols.numel(), device=DEV), k)
    q = torch.arange(b.numel(), device=DEV) - torch.repeat_interleave(torch.cumsum(k, 0) - k, k)
    c = Pri[Pcp[cols][b] + q]
    e = Acp[c + 1] - Acp[c]
    eb, eq = torch.repeat_interleave(b, e), torch.repeat_interleave(q, e)
    at = torch.repeat_interleave(Acp[c], e) + torch.arange(eb.numel(), device=DEV) \
        - torch.repeat_interleave(torch.cumsum(e, 0) - e, e)
    key, inv = torch.unique(eb * n + Ari[at], return_inverse=True)
    ub = key // n
    m = torch.bincount(ub, minlength=cols.numel())
    r = torch.arange(key.numel(), device=DEV) - (torch.cumsum(m, 0) - m)[ub]
    M = int(m.max())
    T = torch.zeros((cols.numel(), M, K), dtype=Av.dtype, device=DEV)
    T[eb, r[inv], eq] = Av[at]
    R = torch.full((cols.numel(), M), -1, dtype=torch.int64, device=DEV)
    R[ub, r] = key % n
    return T, R, k


def _orth(T, pad):
    """Q and R^-1 of T = Q R by two Cholesky factorisations of the scaled Gram matrix (padding columns stay zero)."""
    d = T.abs().square().sum(1).sqrt()
    d = torch.where(d > 0, 1.0 / d, torch.ones_like(d))
    Ri = torch.diag_embed(d).to(T.dtype)
    Q = T * d[:, None, :].to(T.dtype)
    eye = torch.eye(T.shape[2], dtype=T.dtype, device=DEV).expand(T.shape[0], -1, -1)
    for _ in range(2):
        G = Q.mH @ Q + torch.diag_embed(pad.to(T.dtype))
        X = torch.linalg.solve_triangular(torch.linalg.cholesky_ex(G)[0].mH, eye, upper=True)
        Q, Ri = Q @ X, Ri @ X
    return Q, Ri


def _eigh(H):
    """Eigenvectors of a batch of Hermitian matrices, in ascending order of the eigenvalues."""
    size = 16384 if H.shape[1] <= 32 else 1024
    return torch.cat([torch.linalg.eigh(h)[1] for h in H.split(size)])


def _exact_columns(cols, parts, P, spec, alg):
    """Padded per-column results: w [B, K], V's rows and values [B, M] under a mask, the residual."""
    n, Acp, Ari, Av = parts
    T, R, k = _tiles(cols, n, Acp, Ari, Av, *P)
    B, M, K = T.shape
    pad = torch.arange(K, device=DEV)[None, :] >= k[:, None]
    Q, Ri = _orth(T, pad)
    h = Q.abs().square().sum(2)
    j = cols[:, None]
    if spec["vrule"] == diaf.RULE_BLOCK:
        adm = (R >= 0) & (R // BLOCK == j // BLOCK) & (R != j)
    else:
        adm = (R >= 0) & (R < j)
    l = torch.minimum(spec["budget"].long()[cols], 1 + adm.sum(1))
    tau = spec.get("tie_tol", 1e-9)
    I = R == j
    for t in range(int(l.max()) - 1):
        hm = torch.where(adm, h, -torch.inf)
        best = (adm & (hm >= hm.max(1, keepdim=True)[0] - tau)).to(torch.int8).argmax(1)  # the lowest tied row
        on = (t < l - 1) & adm.any(1)
        at = torch.nonzero(on)[:, 0]
        I[at, best[at]] = True
        adm[at, best[at]] = False
    zero = torch.zeros((), dtype=T.dtype, device=DEV)
    if alg == "S":
        H = torch.where(I[:, :, None], zero, T)
        H = H.mH @ H
        big = 4 * torch.diagonal(H, dim1=1, dim2=2).real.sum(1, keepdim=True) + 1.0
        H = H + torch.diag_embed(torch.where(pad, big, torch.zeros_like(big)).to(T.dtype))
        w = _eigh(H)[:, :, 0]
        Tw = (T @ w[:, :, None])[:, :, 0]
        v = torch.where(I, Tw, zero)
    else:
        QI = torch.where(I[:, :, None], Q, zero)
        u = _eigh(QI.mH @ QI)[:, :, -1]
        v = (QI @ u[:, :, None])[:, :, 0]
        v = v / torch.linalg.vector_norm(v, dim=1, keepdim=True)
        w = (Ri @ (Q.mH @ v[:, :, None]))[:, :, 0]
        Tw = (T @ w[:, :, None])[:, :, 0]
    res = torch.linalg.vector_norm(Tw - v, dim=1)
    vjj = torch.where(R == j, v, zero).sum(1)
    big = torch.gather(w, 1, w.abs().argmax(1, keepdim=True))[:, 0]
    s = torch.where(vjj.abs() > 64 * 2.0**-52 * torch.linalg.vector_norm(v, dim=1), vjj, big)
    s = torch.where(s.abs() > 0, s.conj() / s.abs().clamp(min=1e-300), torch.ones_like(s))[:, None]
    return w * s, ~pad, R, v * s, I, res


def _exact_factor(A, PW, spec, alg):
    parts = _csc_parts(A)
    n, Acp, Ari, Av = parts
    P = (PW.colptr.long(), PW.rowidx.long())
    k = P[0].diff()
    W = torch.zeros(PW.nnz, dtype=Av.dtype, device=DEV)
    res = torch.zeros(n, dtype=torch.float64, device=DEV)
    cols_v, rows_v, vals_v = [], [], []
    e = torch.zeros(PW.nnz + 1, dtype=torch.int64, device=DEV)
    e[1:] = torch.cumsum(Acp.diff()[P[1]], 0)
    m = e[P[0][1:]] - e[P[0][:-1]]  # at most so many rows
    order = torch.argsort(k * (1 << 32) + m)
    at = 0
    while at < n:
        biggest = int(k[order[at]]) * int(m[order[at]])
        take = order[at:at + max(64, 24_000_000 // max(1, biggest))]
        while take.numel() > 64 and int(k[take[-1]]) * int(m[take[-1]]) > 2 * biggest + 64:
            take = take[:take.numel() // 2]
        at += take.numel()
        cols = torch.sort(take)[0]
        w, wm, R, v, I, r = _exact_columns(cols, parts, P, spec, alg)
        b, q = torch.nonzero(wm, as_tuple=True)
        W[P[0][cols][b] + q] = w[b, q]
        res[cols] = r
        b, i = torch.nonzero(I, as_tuple=True)
        cols_v.append(cols[b])
        rows_v.append(R[b, i])
        vals_v.append(v[b, i])
    cv, rv, vv = torch.cat(cols_v), torch.cat(rows_v), torch.cat(vals_v)
    order = torch.argsort(cv * n + rv)
    return W, cv[order], rv[order], vv[order], res


def _levels(n, col, row):
    """Depth of every row of an upper triangular matrix in its solve."""
    c, r = col.cpu().numpy(), row.cpu().numpy()
    start = np.searchsorted(c, np.arange(n + 1))
    lev = [0] * n
    r = r.tolist()
    start = start.tolist()
    for j in range(n - 1, -1, -1):
        d = lev[j] + 1
        for p in range(start[j], start[j + 1]):
            i = r[p]
            if i < j and lev[i] < d:
                lev[i] = d
    return torch.tensor(lev, device=DEV)


def _inverse_v(case, n, col, row, val):
    """x -> V^-1 x in plain torch: by levels for a triangular V, by dense blocks for a block-diagonal one."""
    if case["op"] == "lognormal":
        nb = -(-n // BLOCK)
        D = torch.eye(BLOCK, dtype=val.dtype, device=DEV).repeat(nb, 1, 1)
        inside = torch.arange(nb * BLOCK, device=DEV).reshape(nb, BLOCK) < n
        D = torch.where(inside[:, :, None], torch.zeros_like(D), D)
        D[col // BLOCK, row % BLOCK, col % BLOCK] = val

        def solve(x):
            xp = torch.zeros(nb * BLOCK, dtype=x.dtype, device=DEV)
            xp[:n] = x
            return torch.linalg.solve(D, xp.reshape(nb, BLOCK, 1)).reshape(-1)[:n]

        return solve
    lev = _levels(n, col, row)
    diag = torch.zeros(n, dtype=val.dtype, device=DEV)
    diag[row[row == col]] = val[row == col]
    off = row != col
    col, row, val = col[off], row[off], val[off]
    order = torch.argsort(lev[row], stable=True)
    col, row, val = col[order], row[order], val[order]
    nlev = int(lev.max()) + 1
    ends = torch.cumsum(torch.bincount(lev[row], minlength=nlev), 0).tolist()
    rl = torch.argsort(lev, stable=True)
    rends = torch.cumsum(torch.bincount(lev, minlength=nlev), 0).tolist()
    cuts = [(slice(ends[i - 1] if i else 0, ends[i]), rl[rends[i - 1] if i else 0:rends[i]]) for i in range(nlev)]

    def solve(x):
        t = x.clone()
        for s, rows in cuts:
            t.index_add_(0, row[s], -val[s] * t[col[s]])
            t[rows] /= diag[rows]
        return t

    return solve


def _exact_apply(PW, W, vinv):
    pcol = torch.repeat_interleave(torch.arange(PW.n, device=DEV), PW.colptr.diff().long())
    prow = PW.rowidx.long()
    return lambda x: torch.zeros_like(x).index_add_(0, prow, W * vinv(x)[pcol])


def _exact_gmres(mv, prec, b, tol, restart, maxit):
    n, x = b.numel(), torch.zeros_like(b)
    bnorm = torch.linalg.vector_norm(b).item()
    its, rel = 0, 1.0
    while its < maxit and rel > tol:
        r = b - mv(x)
        beta = torch.linalg.vector_norm(r)
        Q = torch.zeros((n, restart + 1), dtype=b.dtype, device=DEV)
        Q[:, 0] = r / beta
        H = torch.zeros((restart + 1, restart), dtype=b.dtype)
        s = 0
        while s < restart and its < maxit and rel > tol:
            w = mv(prec(Q[:, s]))
            h = torch.zeros(s + 1, dtype=b.dtype, device=DEV)
            for _ in range(2):
                c = Q[:, :s + 1].mH @ w
                w = w - Q[:, :s + 1] @ c
                h += c
            nw = torch.linalg.vector_norm(w)
            H[:s + 1, s] = h.cpu()
            H[s + 1, s] = nw.item()
            Q[:, s + 1] = w / nw
            s, its = s + 1, its + 1
            e = torch.zeros(s + 1, dtype=b.dtype)
            e[0] = beta.item()
            y = torch.linalg.lstsq(H[:s + 1, :s], e[:, None], driver="gelsd").solution
            rel = torch.linalg.vector_norm(e - (H[:s + 1, :s] @ y)[:, 0]).item() / bnorm
        x = x + prec((Q[:, :s] @ y.to(DEV))[:, 0])
    return x, torch.linalg.vector_norm(b - mv(x)).item() / bnorm


def _exact_features(A, C):
    n, Acp, Ari, Av = _csc_parts(A)
    acol = torch.repeat_interleave(torch.arange(n, device=DEV), Acp.diff())
    keys, av = acol * n + Ari, Av.abs()
    col = torch.repeat_interleave(torch.arange(n, device=DEV), C.colptr.diff().long())
    row = C.rowidx.long()

    def entry(r, c):
        i = torch.searchsorted(keys, c * n + r).clamp(max=keys.numel() - 1)
        return torch.where(keys[i] == c * n + r, av[i], torch.zeros_like(av[i])), keys[i] == c * n + r

    def column_max(v, c):
        return torch.zeros(n, dtype=torch.float64, device=DEV).scatter_reduce_(0, c, v, "amax")

    diag, _ = entry(torch.arange(n, device=DEV), torch.arange(n, device=DEV))
    a, in_a = entry(row, col)
    e = Acp.diff()[Ari]  # (A^2)(:, j) from the products A(:, q) A(q, j)
    src = torch.repeat_interleave(torch.arange(Ari.numel(), device=DEV), e)
    at = torch.repeat_interleave(Acp[Ari], e) + torch.arange(src.numel(), device=DEV) \
        - torch.repeat_interleave(torch.cumsum(e, 0) - e, e)
    ckeys = col * n + row
    k2 = acol[src] * n + Ari[at]
    i = torch.searchsorted(ckeys, k2).clamp(max=ckeys.numel() - 1)
    hit = ckeys[i] == k2
    sq = torch.zeros(ckeys.numel(), dtype=torch.float64, device=DEV).index_add_(0, i[hit], (Av[at] * Av[src])[hit]).abs()
    div = lambda x, y: torch.where(y > 0, x / y, torch.zeros_like(x))  # noqa: E731
    deg = Acp.diff().double()
    return torch.stack([
        (row == col).double(), in_a.double(), div(a, column_max(av, acol)[col]), div(sq, column_max(sq, col)[col]),
        torch.log(diag[row] / diag[col]).clamp(-10, 10), entry(col, row)[0] / diag[col], deg[row] / deg[col],
        torch.sign(col - row).double()], 1)


def _mlp_parts(p):
    F, H = diaf.PROP_NFEAT, diaf.PROP_HIDDEN
    cut = np.cumsum([H * F, H, H * H, H, H])
    W1, b1, W2, b2, w3, b3 = (p[a:b] for a, b in zip([0, *cut], [*cut, p.numel()]))
    return W1.reshape(H, F), b1, W2.reshape(H, H), b2, w3, b3


def _exact_mlp(p, x):
    W1, b1, W2, b2, w3, b3 = _mlp_parts(p)
    return torch.relu(torch.relu(x @ W1.T + b1) @ W2.T + b2) @ w3 + b3


def exact(case, seed):
    kind = case["kind"]
    if kind == "sparsified":
        return None  # index lists only
    st = prepare(dict(case, kind="setup") if kind in ("apply", "gmres") else case, seed)
    if kind == "train":
        p = st["params"].double().requires_grad_(True)
        loss = (_exact_mlp(p, st["feat"].double()) - st["target"].double()).square().mean()
        (g,) = torch.autograd.grad(loss, p)
        p = p.detach()
        step = 3e-3 * g / (g.abs() + 1e-8)  # the first step: both moments bias-corrected to g and g^2
        return dict(grad=g, loss=loss.detach().reshape(1), params=p - step, m=0.1 * g, v=1e-3 * g * g)
    A = st["A"]
    if kind == "propose":
        s = _exact_mlp(st["net"].params.double(), _exact_features(A, st["CAND"]))
        return dict(scores=s, colptr=None, rowidx=None)
    W, vc, vr, vv, res = _exact_factor(A, st["PW"], st["spec"], case.get("alg", "S"))
    if kind == "setup" and not case["apply"]:
        return dict(W=None, V_colptr=None, V_rowidx=None, V=None, res=res, flags=None)
    apply = _exact_apply(st["PW"], W, _inverse_v(case, A.n, vc, vr, vv))
    if kind == "setup":
        return dict(W=W, V_colptr=None, V_rowidx=None, V=vv, res=res, flags=None, y=apply(st["x"]))
    if kind == "apply":
        return dict(y=apply(st["x"]))
    b = _spmv(A, torch.ones_like(st["x"]) + 0.1 * st["x"])
    acol = torch.repeat_interleave(torch.arange(A.n, device=DEV), A.colptr.diff().long())
    mv = lambda v: torch.zeros_like(v).index_add_(0, A.rowidx.long(), A.vals * v[acol])  # noqa: E731
    x, rel = _exact_gmres(mv, apply, b, 1e-6, 50, 2000)
    return dict(x=x, iterations=None, relres=rel)
