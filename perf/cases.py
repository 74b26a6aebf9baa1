"""The framework's work as a user's program has it: scalar products, operator and preconditioner applications,
truncated sums and products (the steps of Alg. 5), and whole solves, through the public entry points of
paper_2306_00632_gb300.api.

Operators of the single steps are synthetic (banded matrices with smoothly varying coefficients, the sparsity and
scale of the B-spline ones), so that they need no quadrature; solves use the library's own geometry setup.  Outputs
are what does not depend on the choice of a basis: factors of unrounded tensors with their block scales, rounded
tensors as dense arrays, solutions as the field in single precision (a solve fixes no more digits than its
tolerance).  Tolerances of truncations lie in the middle of a gap of the spectrum near the wanted one: a rank is
then decided by the input and not by the last bit.
"""
import math
import os
from types import SimpleNamespace

# as the benchmark and the server set it: hardware queues for concurrent solves, read when CUDA starts
os.environ.setdefault("CUDA_DEVICE_MAX_CONNECTIONS", "32")

import numpy as np  # noqa: E402
import torch  # noqa: E402

from paper_2306_00632_gb300 import api, lib  # noqa: E402

F64, F32 = "f64", "f32"
CODE = {F64: lib.F64, F32: lib.F32}
TYPE = {F64: torch.float64, F32: torch.float32}
RANK_CAP = 96      # the benchmark's and the server's rank cap (at most n)


def listed():
    return [
        # the smallest call: a scalar product of Alg. 5 on a small problem (n = 32, the unit cube's size)
        {"name": "dot small", "kind": "dot", "n": 32, "r": 6, "dtype": F64},
        # residual f - A x at the large configuration (n = 512, rank 80, 19 terms)
        {"name": "residual 512", "kind": "residual", "n": 512, "p": 3, "R": 19, "r": 80, "dtype": F32},
        # Alg. 4 on a residual of the benchmark size, double precision
        {"name": "precond 128", "kind": "precond", "n": 128, "p": 3, "RP": 12, "r": 44, "dtype": F64},
        # p <- T(z + beta p) on a small problem in double precision
        {"name": "sum small", "kind": "sum", "n": 32, "r": 9, "dtype": F64, "eps": 1e-3},
        # the same inside the FP32 inner solves of the benchmark (k < n: the QR path)
        {"name": "sum 128", "kind": "sum", "n": 128, "r": 54, "dtype": F32, "eps": 0.05},
        # q <- T(A p) inside the FP32 inner solves of the benchmark
        {"name": "product 128", "kind": "product", "n": 128, "p": 3, "R": 19, "r": 36, "dtype": F32, "eps": 0.05},
        # the same in double precision at an odd size, even degree
        {"name": "product 97 f64", "kind": "product", "n": 97, "p": 2, "R": 19, "r": 21, "dtype": F64, "eps": 1e-4},
        # the large configuration's truncated product (Grams above order 128)
        {"name": "product 512", "kind": "product", "n": 512, "p": 3, "R": 19, "r": 40, "dtype": F32, "eps": 0.05},
        # r <- T(f - A x) of the elasticity block system, at a size the server's requests have
        {"name": "elasticity 24", "kind": "elasticity", "n": 24, "p": 2, "R": 8, "r": 10, "dtype": F64, "eps": 1e-3},
        # a whole solve in double precision
        {"name": "solve 32 f64", "kind": "solve", "n": 32, "p": 2, "form": F64, "count": 1},
        # a whole solve of the benchmark problem, mixed form, alone (latency)
        {"name": "solve 128 mixed", "kind": "solve", "n": 128, "p": 3, "form": "mixed", "count": 1},
        # many solves of it at once (throughput)
        {"name": "solves 128 mixed", "kind": "solve", "n": 128, "p": 3, "form": "mixed", "count": 8},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))


def draw(rng):
    kind = rng.choice(["dot", "residual", "precond", "sum", "sum", "product", "product", "elasticity", "solve"])
    if kind == "solve":
        if rng.random() < 0.5:
            return {"kind": kind, "n": rng.randint(24, 36), "p": rng.randint(2, 4), "form": F64, "count": 1}
        return {"kind": kind, "n": rng.randint(40, 128), "p": rng.randint(2, 4), "form": "mixed",
                "count": rng.choice([1, 2, 4])}
    dtype = rng.choice([F64, F32])
    if kind == "elasticity":
        return {"kind": kind, "n": rng.randint(16, 32), "p": rng.randint(2, 3), "R": rng.randint(3, 10),
                "r": rng.randint(5, 14), "dtype": F64, "eps": round(10 ** rng.uniform(-4, -2), 6)}
    eps = round(10 ** (rng.uniform(-1.5, -0.8) if dtype == F32 else rng.uniform(-5, -2)), 7)
    if kind == "sum":
        n = _log(rng, 32, 400) if dtype == F32 else _log(rng, 32, 144)
        return {"kind": kind, "n": n, "r": rng.randint(4, min(60, n // 2)), "dtype": dtype, "eps": eps}
    p = rng.randint(2, 4)
    if kind == "product":
        n = _log(rng, 32, 400) if dtype == F32 else _log(rng, 32, 144)
        return {"kind": kind, "n": n, "p": p, "R": rng.choice([3, 7, 13, 19]), "r": rng.randint(4, min(40, n // 2)),
                "dtype": dtype, "eps": eps}
    n = _log(rng, 32, 512)
    r = rng.randint(2, min(80, n // 2))
    if kind == "dot":
        return {"kind": kind, "n": n, "r": r, "dtype": dtype}
    if kind == "residual":
        return {"kind": kind, "n": n, "p": p, "R": rng.choice([3, 13, 19, 25]), "r": r, "dtype": dtype}
    return {"kind": kind, "n": n, "p": p, "RP": rng.randint(8, 17), "r": min(r, 64), "dtype": dtype}


# ------------------------------------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _smooth(g, n, r):
    """r orthonormal smooth functions on n points: random combinations of decaying sines."""
    m = min(n, r + 8)
    x = torch.arange(1, n + 1, device="cuda", dtype=torch.float64) / (n + 1)
    k = torch.arange(1, m + 1, device="cuda", dtype=torch.float64)
    s = torch.sin(math.pi * x[:, None] * k[None, :]) * k ** -0.5
    return torch.linalg.qr(s @ _randn(g, m, r))[0]


def _tucker(g, n, r, dtype, fall=1e-3):
    """(core, factors), multilinear rank near r, mode singular values falling to `fall`; values of the dtype."""
    ranks = (r, max(1, r - 1), max(1, r - 3))
    rho = fall ** (1.0 / max(r, 2))
    i = [rho ** torch.arange(q, device="cuda", dtype=torch.float64) for q in ranks]
    core = _randn(g, *ranks) * i[0][:, None, None] * i[1][None, :, None] * i[2][None, None, :]
    core = core / core.norm()
    u = [_smooth(g, n, q) for q in ranks]
    if dtype == F32:
        core, u = core.float().double(), [v.float().double() for v in u]
    return core, u


def _bands(g, n, p, R, dtype):
    """(weights, bands[R][3][2p+1][n]): stencils of a mass or a stiffness matrix times a smooth coefficient."""
    d = torch.arange(-p, p + 1, device="cuda", dtype=torch.float64)
    mass = torch.exp(-d * d / (0.35 * p)) / torch.exp(-d * d / (0.35 * p)).sum()
    stiff = -mass.clone()
    stiff[p] -= stiff.sum()
    x = torch.arange(1, n + 1, device="cuda", dtype=torch.float64) / (n + 1)
    which = torch.arange(R, device="cuda")[:, None] % 3 == torch.arange(3, device="cuda")[None, :]
    base = torch.where(which[:, :, None], stiff[None, None, :], mass[None, None, :])
    a = _randn(g, R, 3, 3)
    freq = torch.arange(1, 4, device="cuda", dtype=torch.float64) * math.pi
    coef = 1.0 + 0.25 * torch.einsum("jtq,iq->jti", a, torch.sin(x[:, None] * freq[None, :]))
    b = base[:, :, :, None] * coef[:, :, None, :]
    i = torch.arange(n, device="cuda")[None, :] + d[:, None].long()
    b = b * ((i >= 0) & (i < n))
    w = 0.6 ** torch.arange(R, device="cuda", dtype=torch.float64) * (1.0 + 0.1 * _randn(g, R))
    return w, (b.float().double() if dtype == F32 else b)


def _dense(bands):
    """One banded matrix [2p+1, n] as a dense one: K[i, i + d - p] = bands[d, i]."""
    bw, n = bands.shape
    K = torch.zeros(n, n, device=bands.device, dtype=bands.dtype)
    i = torch.arange(n, device=bands.device)
    for d in range(bw):
        j = i + d - bw // 2
        ok = (j >= 0) & (j < n)
        K[i[ok], j[ok]] = bands[d, ok]
    return K


def _fd_tables(g, n, p, RP):
    """Tables of Alg. 4 with the structure App. B gives them: p - 1 outliers for odd p, p - 2 for even p."""
    n2 = p - 1 if p % 2 else p - 2
    n1 = n - n2
    j = torch.arange(1, n1 + 1, device="cuda", dtype=torch.float64)
    lam = torch.cat([(math.pi * j) ** 2, (4.0 + torch.rand(n2, generator=g, device="cuda", dtype=torch.float64))
                     * (math.pi * n1) ** 2])
    mu = 1.0 - 0.4 * (j / (n1 + 1)) ** 2
    W = torch.zeros(n, n1, dtype=torch.float64)
    s = n2 // 2
    W[torch.arange(n1) + s, torch.arange(n1)] = 1.0
    end = 0.2 * torch.randn(p, p, generator=torch.Generator().manual_seed(int(RP) + n), dtype=torch.float64)
    W[:p, :p] += end
    W[n - p:, n1 - p:] += end.flip(0, 1)
    v2u2 = _randn(g, n, n2) / math.sqrt(n)
    lmin = 3.0 * float(lam.min())
    q = torch.arange(RP, device="cuda", dtype=torch.float64)
    alpha = 4.0 * 0.35 ** q
    omega = 2.0 * alpha
    return SimpleNamespace(n1=n1, n2=n2, lam=lam, mu=mu, W=W, v2u2=v2u2, omega=omega, alpha=alpha, lmin=lmin)


def _host(t):
    return t.detach().cpu().numpy()


def _flat(t):
    """Column-major values of a 2-d or 3-d tensor, on the host."""
    return _host(t.permute(*reversed(range(t.dim()))).contiguous().reshape(-1))


def _problem(n, p, w, bands, rhs, fd, dtype):
    W = fd.W.numpy()
    nz = [np.nonzero(W[i])[0] for i in range(n)]
    ex = {"w": _host(w), "bands": _host(bands).reshape(-1), "lam": _host(fd.lam), "mu": _host(fd.mu),
          "w_rowptr": np.concatenate([[0], np.cumsum([len(q) for q in nz])]), "w_col": np.concatenate(nz),
          "w_val": np.concatenate([W[i, q] for i, q in enumerate(nz)]), "v2u2": _flat(fd.v2u2),
          "omega": _host(fd.omega), "alpha": _host(fd.alpha)}
    info = SimpleNamespace(n=n, p=p, R=len(ex["w"]), n1=fd.n1, n2=fd.n2, RP=len(ex["omega"]), w_nnz=len(ex["w_col"]),
                           lambda_min=fd.lmin, k0=0, k1=0)
    return api.problem_from_export(ex, info, CODE[dtype], pinned=False,
                                   rhs=(_host(rhs[0]), [_host(u) for u in rhs[1]]))


def _upload(t, cap, dtype):
    return api.Tucker.from_numpy(_host(t[0]), [_host(u) for u in t[1]], cap=cap, dtype=CODE[dtype])


def _terms(w, bands, x, sign=1.0):
    """Blocks (scale, core, factors) of sign A x."""
    return [(sign * float(w[j]), x[0], [_dense(bands[j, t]) @ x[1][t] for t in range(3)]) for j in range(len(w))]


def _gap_eps(blocks, eps):
    """The tolerance within a factor 1.4 of eps whose budget is furthest from every mode's tail energies."""
    R = []
    for t in range(3):
        Y = torch.cat([b[2][t] for b in blocks], 1)
        R.append(torch.linalg.qr(Y, mode="r")[1] if Y.shape[1] < Y.shape[0] else Y)
    off, Z = [0, 0, 0], 0
    for s, core, u in blocks:
        part = s * core
        for t in range(3):
            k = u[t].shape[1]
            part = torch.tensordot(part, R[t][:, off[t]:off[t] + k], dims=([0], [1]))
            off[t] += k
        Z = Z + part
    tails = []
    for t in range(3):
        M = Z.movedim(t, 0).reshape(Z.shape[t], -1)
        lam = torch.linalg.eigvalsh(M @ M.T).clamp_min(0)
        c = torch.cumsum(lam, 0) / lam.sum()
        tails.append(torch.log(c[c > 1e-14]))
    tails = torch.cat(tails)
    e = eps * 1.4 ** torch.linspace(-1, 1, 81, device="cuda", dtype=torch.float64)
    far = (torch.log(e * e / 3)[:, None] - tails[None, :]).abs().min(1)[0]
    return float(e[int(far.argmax())])


_inputs_of = {}


def _inputs(case, seed):
    """What the case's call is given, in 64 bits (values of the case's dtype)."""
    c = SimpleNamespace(**case)
    g = _gen(seed)
    if c.kind == "solve":
        return SimpleNamespace(problems=[_solve_tables(c, g, i) for i in range(c.count)])
    s = SimpleNamespace()
    if c.kind == "elasticity":
        s.x = [_tucker(g, c.n, c.r - i, c.dtype) for i in range(3)]
        s.f = [_tucker(g, c.n, 1, c.dtype) for i in range(3)]
        s.A = [[_bands(g, c.n, c.p, c.R if i == j else max(1, c.R // 2), c.dtype) for j in range(3)] for i in range(3)]
        for i in range(3):
            for j in range(3):
                if i != j:
                    s.A[i][j] = (0.3 * s.A[i][j][0], s.A[i][j][1])
        s.fd = _fd_tables(g, c.n, c.p, 8)
        s.blocks = [[(1.0, s.f[i][0], s.f[i][1])] + [b for j in range(3) for b in _terms(*s.A[i][j], s.x[j], -1.0)]
                    for i in range(3)]
        s.eps = [_gap_eps(b, c.eps) for b in s.blocks]
        return s
    s.x = _tucker(g, c.n, c.r, c.dtype)
    if c.kind == "dot":
        # y: x with a tenth of another tensor in its core, as successive iterates are
        s.y = (s.x[0] + 0.1 * _tucker(g, c.n, c.r, c.dtype)[0], s.x[1])
        if c.dtype == F32:
            s.y = (s.y[0].float().double(), s.y[1])
    if c.kind == "sum":
        s.y = _tucker(g, c.n, max(2, c.r - 2), c.dtype)
        s.b = 0.3 + 0.4 * float(torch.rand(1, generator=g, device="cuda"))
        s.blocks = [(1.0, s.x[0], s.x[1]), (s.b, s.y[0], s.y[1])]
    if c.kind in ("residual", "product", "precond"):
        s.fd = _fd_tables(g, c.n, c.p, getattr(c, "RP", 8))
        s.w, s.bands = _bands(g, c.n, c.p, getattr(c, "R", 3), c.dtype)
        s.f = _tucker(g, c.n, 2, c.dtype)
    if c.kind == "product":
        s.blocks = _terms(s.w, s.bands, s.x)
    if c.kind in ("sum", "product"):
        s.eps = _gap_eps(s.blocks, c.eps)
    return s


def _solve_tables(c, g, i):
    """The twisted annulus (amplitudes of the benchmark family; the host setup is made once per geometry), its load
    modulated by a smooth random source: the same operator, another right-hand side."""
    amp = (0.0333, 0.11, 0.19, 0.27)[i % 4]
    key = (c.n, c.p, amp)
    if key not in _inputs_of:
        _inputs_of[key] = api.setup_host(lib.GEOM_TWIST, amp, c.p, c.n)
    h = _inputs_of[key]
    x = np.arange(1, c.n + 1) / (c.n + 1.0)
    a = _host(_randn(g, 3, 3))
    rhs = []
    for t in range(3):
        m = 1.0 + 0.2 * sum(a[t, q] * np.sin((q + 1) * np.pi * x) for q in range(3))
        rhs.append(h["f_U"][t] * m[:, None])
    return SimpleNamespace(h=h, core=h["f_core"], rhs=rhs)


def _ctx(n, cols, dtype):
    cap = min(n, RANK_CAP)
    return api.Ctx(n, max(cols, 2 * cap), cap, dtype)


def prepare(case, seed):
    c = SimpleNamespace(**case)
    s = _inputs(case, seed)
    if c.kind == "solve":
        return _prepare_solves(c, s)
    n, dt = c.n, CODE[c.dtype]
    st = SimpleNamespace(case=c, kind=c.kind)
    cap = min(n, RANK_CAP)
    if c.kind == "elasticity":
        mats = lambda i, j: [(float(s.A[i][j][0][q]), [_host(_dense(s.A[i][j][1][q, t])) for t in range(3)])  # noqa: E731
                             for q in range(len(s.A[i][j][0]))]
        fd = {"lam": _host(s.fd.lam), "mu": _host(s.fd.mu), "W": s.fd.W.numpy(), "v2u2": _host(s.fd.v2u2),
              "omega": _host(s.fd.omega), "alpha": _host(s.fd.alpha), "lambda_min": s.fd.lmin}
        st.e = api.tpcg_elast_create(n, c.p, [[mats(i, j) for j in range(3)] for i in range(3)],
                                     [(_host(f[0]), [_host(u) for u in f[1]]) for f in s.f], fd, 0.3 / 0.52, 1 / 2.6,
                                     dtype=dt)
        st.x = [_upload(x, cap, c.dtype) for x in s.x]
        cols = 1 + 3 * (c.R + 2 * max(1, c.R // 2)) * c.r
        st.y = [api.Tucker(n, cols, cap ** 3, dt) for _ in range(3)]
        st.ctx = _ctx(n, cols, dt)
        st.eps = s.eps
        return st
    st.x = _upload(s.x, cap, c.dtype)
    if c.kind == "dot":
        st.y = _upload(s.y, cap, c.dtype)
        st.ctx = _ctx(n, 2 * cap, dt)
        st.out = torch.zeros(1, dtype=torch.float64, device="cuda")
    elif c.kind == "sum":
        st.y, st.b, st.eps = _upload(s.y, cap, c.dtype), s.b, s.eps
        st.z = api.Tucker(n, 2 * cap, cap ** 3, dt)
        st.ctx = _ctx(n, 2 * cap, dt)
    else:
        st.pb = _problem(n, c.p, s.w, s.bands, s.f, s.fd, c.dtype)
        if c.kind == "precond":
            st.y = api.Tucker(n, c.RP * cap, 1, dt)
            st.ctx = _ctx(n, c.RP * cap, dt)
        else:
            cols = c.R * c.r + 2
            st.y = api.Tucker(n, cols, cap ** 3 if c.kind == "product" else 1, dt)
        if c.kind == "product":
            st.eps, st.ctx = s.eps, _ctx(n, cols, dt)
    return st


def _prepare_solves(c, s):
    dt = lib.MIXED if c.form == "mixed" else lib.F64
    cap = min(c.n, RANK_CAP)
    st = SimpleNamespace(case=c, kind="solve", form=c.form)
    st.pbs = [api.problem_from_export(_export_of(q.h), q.h["info"], dt, pinned=False, rhs=(q.core, q.rhs))
              for q in s.problems]
    st.ctxs = [api.Ctx(c.n, api.max_cols_for(pb.info, cap, dt), cap, dt) for pb in st.pbs]
    st.xs = [api.Tucker(c.n, cap, cap ** 3, dt) for _ in st.pbs]
    st.streams = [api.ctx_stream(x) for x in st.ctxs]
    return st


def _export_of(h):
    ex = {k: h[k] for k in ("w", "lam", "mu", "omega", "alpha", "w_rowptr", "w_col", "w_val")}
    ex["bands"] = h["bands"].reshape(-1)
    ex["v2u2"] = h["v2u2"].reshape(-1, order="F")
    return ex


# ------------------------------------------------------------------------------------------------ the calls
def _parts(y, ranks, nblk):
    """Factors and block scales of an unrounded tensor, as they lie in its buffers."""
    return {"factors": [y.U[t][:ranks[t]] for t in range(3)], "scales": y.desc.view(torch.float64)[8::5][:nblk]}


def _field(y, dtype=None):
    """The dense tensor of a rounded one (indices i3, i2, i1)."""
    _, (r1, r2, r3), _ = y.read_desc()
    core = y.core[:r1 * r2 * r3].view(r3, r2, r1)
    u = [y.U[t][:r] for t, r in enumerate((r1, r2, r3))]
    if dtype is not None:
        core, u = core.to(dtype), [v.to(dtype) for v in u]
    n = y.n
    a = (core.reshape(r3 * r2, r1) @ u[0]).view(r3, r2, n)
    a = torch.matmul(u[1].T, a).view(r3, n * n)
    return (u[2].T @ a).view(n, n, n)


def run(st):
    c = st.case
    if st.kind == "dot":
        out = api.tucker_dot(st.ctx, st.x, st.y, st.out)
        return out if c.dtype == F64 else out.float()
    if st.kind == "residual":
        api.tucker_residual(st.pb, st.x, st.y)
        return _parts(st.y, [_x_rank(2, t) + c.R * _x_rank(c.r, t) for t in range(3)], 1 + c.R)
    if st.kind == "precond":
        api.fd_precond_apply(st.pb, st.ctx, st.x, st.y)
        return _parts(st.y, [c.RP * _x_rank(c.r, t) for t in range(3)], c.RP)
    if st.kind == "sum":
        api.tucker_axpby(1.0, st.x, st.b, st.y, st.z)
        api.tucker_round(st.ctx, st.z, st.eps)
        return _field(st.z)
    if st.kind == "product":
        api.tucker_apply(st.pb, st.x, st.y)
        api.tucker_round(st.ctx, st.y, st.eps)
        return _field(st.y)
    if st.kind == "elasticity":
        api.elast_residual(st.e, st.x, st.y)
        for i in range(3):
            api.tucker_round(st.ctx, st.y[i], st.eps[i])
        return [_field(y) for y in st.y]
    if c.count == 1:
        api.tpcg_solve(st.pbs[0], st.ctxs[0], st.xs[0], stream=st.streams[0], tol=1e-6)
    else:
        api.tpcg_solve_batch(st.pbs, st.ctxs, st.xs, st.streams, tol=1e-6)
    return [_field(x, torch.float32) for x in st.xs]


def _x_rank(r, t):
    return (r, max(1, r - 1), max(1, r - 3))[t]


# ------------------------------------------------------------------------------------------------ the work
def work(case):
    """Inputs read once and outputs written once; of the operations those of the contraction that forms the
    tensor and of its first Gram (a truncation has to look at the whole of it)."""
    c = SimpleNamespace(**case)
    n, e = c.n, 4 if case.get("dtype") == F32 else 8
    if c.kind == "solve":
        # data of a solve; operations of about 30 operator products on full tensors (19 banded terms)
        return {"bytes": c.count * 8.0 * n ** 3, "flops": c.count * 30 * 19 * 3 * 2.0 * (2 * c.p + 1) * n ** 3}
    r = c.r
    if c.kind == "dot":
        return {"bytes": e * 2.0 * (3 * n * r + r ** 3), "flops": 6.0 * n * r * r + 6.0 * r ** 4}
    if c.kind in ("residual", "precond"):
        terms = c.R if c.kind == "residual" else c.RP
        per = 2.0 * (2 * c.p + 1) if c.kind == "residual" else 10.0 * math.log2(n)
        tables = 3.0 * terms * (2 * c.p + 1) * n if c.kind == "residual" else 0.0
        return {"bytes": e * (3.0 * n * r * (1 + terms) + tables), "flops": 3.0 * per * n * r * terms}
    if c.kind == "sum":
        k, terms, fields = min(n, 2 * r), 2, 1
    elif c.kind == "product":
        k, terms, fields = min(n, c.R * r), c.R, 1
    else:
        terms = c.R + 2 * max(1, c.R // 2)
        k, fields = min(n, 1 + terms * r), 3
    form = terms * 2.0 * (k * r ** 3 + k * k * r * r + k ** 3 * r)
    gram = float(k) ** 4
    return {"bytes": fields * e * (3.0 * n * r * terms + terms * r ** 3 + n ** 3),
            "flops": fields * (form + gram + 2.0 * n ** 3 * r)}


# ------------------------------------------------------------------------------------------------ 64-bit values
def _field64(core, u):
    a = torch.tensordot(core, u[0], dims=([0], [1]))       # r2 r3 n
    a = torch.tensordot(a, u[1], dims=([0], [1]))          # r3 n n
    return torch.tensordot(u[2], a, dims=([1], [0])).transpose(1, 2).contiguous()   # i3, i2, i1


def _sthosvd(blocks, eps, cap):
    """ST-HOSVD of the dense sum of the blocks, as a dense tensor (indices i3, i2, i1)."""
    Z = sum(s * _field64(core, u) for s, core, u in blocks).permute(2, 1, 0)
    budget = eps * eps * float((Z * Z).sum()) / 3
    P = []
    Y = Z
    for t in range(3):
        M = Y.movedim(t, 0).reshape(Y.shape[t], -1)
        lam, V = torch.linalg.eigh(M @ M.T)
        tail = torch.cumsum(lam.clamp_min(0), 0)
        drop = min(int((tail <= budget).sum()), len(lam) - 1)
        drop = max(drop, len(lam) - cap)
        V = V[:, drop:]
        P.append(V)
        Y = torch.tensordot(V.T, Y, dims=([1], [t])).movedim(0, t)
    return _field64(Y, P)


def exact(case, seed):
    c = SimpleNamespace(**case)
    s = _inputs(case, seed)
    if c.kind == "dot":
        y = s.y[0]
        for t in range(3):
            y = torch.tensordot(y, s.x[1][t].T @ s.y[1][t], dims=([0], [1]))
        return (s.x[0] * y).sum().reshape(1)
    if c.kind in ("sum", "product"):
        return _sthosvd(s.blocks, s.eps, min(c.n, RANK_CAP))
    if c.kind == "elasticity":
        return [_sthosvd(b, e, min(c.n, RANK_CAP)) for b, e in zip(s.blocks, s.eps)]
    if c.kind == "residual":
        f = [torch.linalg.qr(u) for u in s.f[1]]
        fac = [torch.cat([q * torch.sign(torch.diagonal(r)) for q, r in [f[t]]]
                         + [_dense(s.bands[j, t]) @ s.x[1][t] for j in range(c.R)], 1).T.contiguous() for t in range(3)]
        return {"factors": fac, "scales": torch.cat([torch.ones(1, device="cuda", dtype=torch.float64), -s.w])}
    if c.kind == "precond":
        return _precond64(c, s)
    if c.count > 2:
        return None      # a reference solve takes seconds each
    return [_solve64(c, q) for q in s.problems]


def _precond64(c, s):
    f = s.fd
    i = torch.arange(1, f.n1 + 1, device="cuda", dtype=torch.float64)
    pts = i / (f.n1 + 1) if c.p % 2 else (i - 0.5) / f.n1
    dst = math.sqrt(2.0) * torch.sin(math.pi * pts[:, None] * i[None, :])
    U = torch.cat([f.W.cuda() @ dst / f.mu, f.v2u2], 1)
    fac = []
    for t in range(3):
        z = U.T @ s.x[1][t]
        fac.append(torch.cat([U @ (torch.exp(-a / f.lmin * f.lam)[:, None] * z) for a in f.alpha.tolist()], 1).T.contiguous())
    return {"factors": fac, "scales": f.omega / f.lmin}


def _solve64(c, q):
    """Preconditioned CG on the full tensor; the preconditioner is the exact inverse on the unit cube."""
    bands = torch.as_tensor(q.h["bands"], device="cuda")
    R = bands.shape[0]
    K = [[_dense(bands[j, t]) for t in range(3)] for j in range(R)]
    w = [float(v) for v in q.h["w"]]
    f = _field64(torch.as_tensor(np.ascontiguousarray(q.core), device="cuda"),
                 [torch.as_tensor(u, device="cuda") for u in q.rhs])

    def modes(X, A1, A2, A3):      # X[i3, i2, i1]
        n = X.shape[0]
        X = (X.reshape(n * n, n) @ A1.T).view(n, n, n)
        X = torch.matmul(A2, X)
        return (A3 @ X.reshape(n, n * n)).view(n, n, n)

    def apply(X):
        return sum(w[j] * modes(X, *K[j]) for j in range(R))

    key = ("cube", c.n, c.p)
    if key not in _inputs_of:
        _inputs_of[key] = api.setup_host(lib.GEOM_CUBE, 0.0, c.p, c.n)
    cube = torch.as_tensor(_inputs_of[key]["bands"], device="cuda")
    one = sorted([_dense(cube[j, 0]) for j in range(2 + (cube.shape[0] > 2))], key=lambda m: float(m.norm()))
    M1, K1 = one[0], one[-1]
    L = torch.linalg.cholesky(M1 / M1.norm() * math.sqrt(c.n))
    Li = torch.linalg.inv(L)
    lam, V = torch.linalg.eigh(Li @ K1 @ Li.T)
    V = Li.T @ V
    D = lam[:, None, None] + lam[None, :, None] + lam[None, None, :]

    def prec(X):
        return modes(modes(X, V.T, V.T, V.T) / D, V, V, V)

    x = torch.zeros_like(f)
    r, z = f.clone(), prec(f)
    d, rz, stop = z.clone(), float((f * z).sum()), 1e-11 * float(f.norm())
    for _ in range(400):
        Ad = apply(d)
        a = rz / float((d * Ad).sum())
        x, r = x + a * d, r - a * Ad
        if float(r.norm()) <= stop:
            break
        z = prec(r)
        rz, old = float((r * z).sum()), rz
        d = z + rz / old * d
    return x
