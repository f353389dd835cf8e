"""Measured cases of the ascg solver: what a program calls, over the range it calls it on.

Each case is one call (or one submit-and-drain loop of the solve server)
through the public binding, on device-resident operators and vectors, all in
float64, the library's only data type:

  powers      ascg_matrix_powers: the basis [P(A) p, P(A) r] of one block
  gram        ascg_gram: G = Y^T Y of a basis
  block_step  ascg_block_step: condition estimates, step choice, coordinate CG
  recover     ascg_recover_tc (w >= 9) or ascg_recover: x, r, p of a block
  solve       ascg_solve: a whole solve, classical or adaptive s-step
  batch       ascg_solve_batch: many uneven systems in one call
  serve       ascg_server_*: requests of mixed size and accuracy, drained

The matrices are the families that the tests and the benchmark use (2D and 3D
Poisson, log-normal diffusion, random banded SPD), equilibrated, built on the
GPU from the seed; right-hand sides are uniform on [-1, 1] and normalised.
"""
import math

import numpy as np
import torch

import paper_1701_03989_gb300 as P

F64 = torch.float64
DEV = "cuda"


# --- matrices ----------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) % (1 << 62))


def _uniform(n, g):
    return torch.rand(n, dtype=F64, device=DEV, generator=g) * 2.0 - 1.0


def _rhs(n, g):
    b = _uniform(n, g)
    return b / b.norm()


def _csr(cols, vals, keep):
    """CSR arrays from (n, k) candidate columns (increasing per row), values and a mask, equilibrated."""
    n = cols.shape[0]
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = torch.cumsum(keep.sum(1), 0)
    d = torch.where(keep, vals.abs(), torch.zeros_like(vals)).amax(1).rsqrt()
    vals = vals * (d[:, None] * d[cols.clamp(0, n - 1)])
    return rowptr, cols[keep].to(torch.int32), vals[keep].contiguous()


def _poisson(dim, m):
    n = m ** dim
    i = torch.arange(n, device=DEV)
    shifts = [m ** k for k in range(dim)]  # fastest axis first
    cols, keep, vals = [], [], []
    for s in reversed(shifts):
        cols.append(i - s)
        keep.append((i // s) % m > 0)
    cols.append(i)
    keep.append(torch.ones_like(i, dtype=torch.bool))
    for s in shifts:
        cols.append(i + s)
        keep.append((i // s) % m < m - 1)
    vals = torch.full((n, 2 * dim + 1), -1.0, dtype=F64, device=DEV)
    vals[:, dim] = 2.0 * dim
    return _csr(torch.stack(cols, 1), vals, torch.stack(keep, 1))


def _diffusion(m, g):
    """Cell-centred finite volumes, log-normal coefficients (sigma = 2), harmonic-mean faces, Dirichlet."""
    a = torch.exp(2.0 * torch.randn((m, m), dtype=F64, device=DEV, generator=g))
    fv = 2.0 * a[:-1] * a[1:] / (a[:-1] + a[1:])
    fh = 2.0 * a[:, :-1] * a[:, 1:] / (a[:, :-1] + a[:, 1:])
    v = torch.zeros((m, m, 5), dtype=F64, device=DEV)
    v[1:, :, 0], v[:, 1:, 1], v[:, :-1, 3], v[:-1, :, 4] = -fv, -fh, -fh, -fv
    v[..., 2] = -v.sum(-1)
    v[0, :, 2] += 2.0 * a[0]
    v[-1, :, 2] += 2.0 * a[-1]
    v[:, 0, 2] += 2.0 * a[:, 0]
    v[:, -1, 2] += 2.0 * a[:, -1]
    i = torch.arange(m * m, device=DEV)
    cols = torch.stack([i - m, i - 1, i, i + 1, i + m], 1)
    r, c = i // m, i % m
    keep = torch.stack([r > 0, c > 0, r >= 0, c < m - 1, r < m - 1], 1)
    return _csr(cols, v.reshape(m * m, 5), keep)


def _banded(n, hbw, g):
    """Off-diagonals within the band U[-1, 0], mirrored; diagonal = row sum + 1e-3."""
    hbw = min(hbw, n - 1)
    v = torch.zeros((n, 2 * hbw + 1), dtype=F64, device=DEV)
    for k in range(1, hbw + 1):
        u = -torch.rand(n - k, dtype=F64, device=DEV, generator=g)
        v[: n - k, hbw + k] = u
        v[k:, hbw - k] = u
    v[:, hbw] = v.abs().sum(1) + 1e-3
    cols = torch.arange(n, device=DEV)[:, None] + torch.arange(-hbw, hbw + 1, device=DEV)[None, :]
    return _csr(cols, v, (cols >= 0) & (cols < n))


def _matrix(c, g):
    fam, size = c["family"], int(c["size"])
    if fam == "poisson2d":
        return _poisson(2, size)
    if fam == "poisson3d":
        return _poisson(3, size)
    if fam == "diffusion2d":
        return _diffusion(size, g)
    return _banded(size, int(c["hbw"]), g)


def _rows(c):
    return int(c["size"]) ** {"poisson2d": 2, "poisson3d": 3, "diffusion2d": 2, "banded": 1}[c["family"]]


def _nnz(c):
    n, m = _rows(c), int(c["size"])
    if c["family"] == "banded":
        h = min(int(c["hbw"]), n - 1)
        return n * (2 * h + 1) - h * (h + 1)
    return 7 * n - 6 * m * m if c["family"] == "poisson3d" else 5 * n - 4 * m


def _bounds(c):
    """Extreme eigenvalues: closed form for Poisson, Gershgorin for the rest."""
    if c["family"].startswith("poisson"):
        m = int(c["size"])
        return 1.0 - math.cos(math.pi / (m + 1)), 1.0 + math.cos(math.pi / (m + 1))
    return 1e-4, 2.0


class _Op:
    """An operator handle that its owner frees."""

    def __init__(self, csr):
        rowptr, colind, val = csr
        self.n = rowptr.numel() - 1
        self.h = P.ascg_op_create_csr(self.n, val.numel(), rowptr, colind, val, 1)

    def __del__(self):
        P.ascg_op_destroy(self.h)


# --- the cases -----------------------------------------------------------------

def listed():
    return [
        # one block's basis of a 3D problem, as a program with its own outer loop builds it
        dict(name="powers_cheb16_poisson3d_100", kind="powers", family="poisson3d", size=100, basis="chebyshev", s=16),
        # long rows (81 entries) and an odd size: a banded system of the batched workload
        dict(name="powers_mono10_banded_20011", kind="powers", family="banded", size=20011, hbw=40, basis="monomial", s=10),
        # the Gram matrix of the largest basis of the 128^3 workload
        dict(name="gram_2097152_w33", kind="gram", n=2097152, w=33),
        # and of the smallest workload (32 x 32 grid, s = 8): latency
        dict(name="gram_1024_w17", kind="gram", n=1024, w=17),
        # the small dense work of a block at the largest s: latency
        dict(name="block_step_s16", kind="block_step", s=16, n=4096, eps=1e-10),
        # the end of a block with s = 12, odd number of rows
        dict(name="recover_999999_w25", kind="recover", n=999999, w=25),
        # the smallest workload, a whole solve: launches and latency
        dict(name="solve_poisson2d_32", kind="solve", family="poisson2d", size=32, method="adaptive", basis="monomial", s=8, eps=1e-10),
        # the headline workload, a whole solve
        dict(name="solve_poisson3d_128", kind="solve", family="poisson3d", size=128, method="adaptive", basis="chebyshev", s=16, eps=1e-12),
        # the same problem by classical CG
        dict(name="classical_poisson3d_128", kind="solve", family="poisson3d", size=128, method="classical", basis="monomial", s=1, eps=1e-12),
        # ill-conditioned variable coefficients, Newton basis, odd grid
        dict(name="solve_newton_diffusion_401", kind="solve", family="diffusion2d", size=401, method="adaptive", basis="newton", s=12, eps=1e-10),
        # uneven systems of all families in one call
        dict(name="batch_32", kind="batch", count=32, nmin=1e3, nmax=1e5, s=10),
        # requests of mixed size and accuracy through the solve server
        dict(name="serve_16", kind="serve", count=16, nmin=1e4, nmax=2e5, s=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_matrix(rng, nlo, nhi):
    fam = rng.choice(["poisson2d", "poisson3d", "diffusion2d", "banded"])
    n = _log(rng, nlo, nhi)
    if fam == "poisson3d":
        return dict(family=fam, size=max(4, round(n ** (1 / 3))))
    if fam == "banded":
        return dict(family=fam, size=max(64, n // 8), hbw=rng.randint(8, 64))
    return dict(family=fam, size=max(8, round(n ** 0.5)))


def draw(rng):
    kind = rng.choice(["powers", "gram", "block_step", "recover", "solve", "solve", "batch", "serve"])
    if kind == "powers":
        basis = rng.choice(["monomial", "chebyshev", "newton"])
        return dict(kind=kind, basis=basis, s=rng.randint(1, 16), **_draw_matrix(rng, 1e3, 2e6))
    if kind == "gram":
        return dict(kind=kind, n=_log(rng, 1e3, 4e6), w=2 * rng.randint(1, 16) + 1)
    if kind == "block_step":
        return dict(kind=kind, s=rng.randint(1, 16), n=_log(rng, 512, 65536), eps=10.0 ** -rng.randint(6, 12))
    if kind == "recover":
        return dict(kind=kind, n=_log(rng, 1e3, 4e6), w=2 * rng.randint(1, 16) + 1)
    if kind == "solve":
        c = dict(kind=kind, **_draw_matrix(rng, 1e3, 3e5))
        if rng.random() < 0.3:
            return dict(c, method="classical", basis="monomial", s=1, eps=10.0 ** -rng.randint(6, 12))
        if c["family"] == "diffusion2d":
            return dict(c, method="adaptive", basis="newton", s=rng.randint(4, 12), eps=10.0 ** -rng.randint(6, 10))
        basis = rng.choice(["monomial", "chebyshev"]) if c["family"].startswith("poisson") else "monomial"
        return dict(c, method="adaptive", basis=basis, s=rng.randint(4, 16 if basis == "chebyshev" else 10), eps=10.0 ** -rng.randint(6, 12))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(4, 32), nmin=1e3, nmax=float(_log(rng, 5e3, 1e5)), s=rng.randint(4, 10))
    return dict(kind=kind, count=rng.randint(4, 16), nmin=1e4, nmax=float(_log(rng, 3e4, 2e5)), s=rng.randint(4, 10))


def _members(c, seed):
    """The systems of a batch or request list: sizes log-uniform, families in turn, targets from the seed."""
    r = np.random.default_rng(seed)
    out, q, count = [], 0, int(c["count"])
    for q in range(count):
        # sizes at the quantiles of the log-uniform law, so that every seed costs about the same
        n = math.exp(math.log(c["nmin"]) + (q + 0.5) / count * (math.log(c["nmax"]) - math.log(c["nmin"])))
        fam = ("poisson2d", "banded", "poisson3d")[q % 3]
        size = round(n) if fam == "banded" else round(n ** (0.5 if fam == "poisson2d" else 1.0 / 3.0))
        eps = (1e-8, 1e-12)[q % 2] if c["kind"] == "batch" else (1e-6, 1e-8, 1e-10, 1e-12)[q % 4]
        out.append(dict(family=fam, size=size, hbw=8 + (q * 17) % 57, eps=eps, seed=int(r.integers(1 << 40))))
    return out


def _coefficients(c):
    """theta, sigma, gamma of the basis recurrence (host)."""
    s = int(c["s"])
    lo, hi = _bounds(c)
    if c["basis"] == "chebyshev":
        h = (hi - lo) / 2
        return np.full(s, (hi + lo) / 2), np.full(s, h / 2), np.array([h] + [h / 2] * (s - 1))
    if c["basis"] == "newton":  # Chebyshev points, interleaved from both ends
        t = (hi + lo) / 2 + (hi - lo) / 2 * np.cos(np.pi * (np.arange(s) + 0.5) / s)
        return t[np.argsort(np.arange(s) * 7 % max(s, 1), kind="stable")].copy(), np.zeros(s), np.ones(s)
    return np.zeros(s), np.zeros(s), np.ones(s)


def _basis_like(n, w, g):
    """A matrix of n x w (column-major, columns of differing scale) like an s-step basis."""
    Y = torch.empty((w, n), dtype=F64, device=DEV)
    for k in range(w):
        Y[k] = _uniform(n, g)
        if k >= 2:
            Y[k].mul_(0.5 ** (k // 2)).add_(Y[k - 2], alpha=0.7)
    return Y


def _block_gram(c, seed):
    """G of a Chebyshev basis of a matrix with eigenvalues spread over [lo, hi], and its coefficients."""
    s, n = int(c["s"]), int(c["n"])
    g = _gen(seed)
    lo, hi = 1e-3, 2.0
    mid, h = (hi + lo) / 2, (hi - lo) / 2
    lam = lo + (hi - lo) * torch.rand(n, dtype=F64, device=DEV, generator=g)
    r = _rhs(n, g)
    p = r + 0.5 * _rhs(n, g)
    t = (lam - mid) / h
    Y = torch.empty((2 * s + 1, n), dtype=F64, device=DEV)
    for k in range(2 * s + 1):
        v = (p, r)[k & 1]
        Y[k] = v if k < 2 else (t * Y[k - 2] if k < 4 else 2 * t * Y[k - 2] - Y[k - 4])
    G = Y @ Y.T
    G = ((G + G.T) / 2).contiguous()
    return G, (np.full(s, mid), np.full(s, h / 2), np.array([h] + [h / 2] * (s - 1)))


def _solve_options(c):
    return P.make_options(method=c["method"], basis=c["basis"], s_max=int(c["s"]), eps_target=c["eps"],
                          lam=_bounds(c) if c["basis"] == "chebyshev" else None, max_iters=20000)


def prepare(case, seed):
    c, kind = case, case["kind"]
    g = _gen(seed)
    if kind == "powers":
        op = _Op(_matrix(c, g))
        Y = torch.zeros((2 * int(c["s"]) + 1, op.n), dtype=F64, device=DEV)
        Y[0], Y[1] = _rhs(op.n, g), _rhs(op.n, g)
        return dict(kind=kind, op=op, Y=Y, s=int(c["s"]), coef=_coefficients(c))
    if kind == "gram":
        n, w = int(c["n"]), int(c["w"])
        return dict(kind=kind, n=n, w=w, Y=_basis_like(n, w, g), G=torch.empty((w, w), dtype=F64, device=DEV))
    if kind == "block_step":
        G, coef = _block_gram(c, seed)
        s = int(c["s"])
        return dict(kind=kind, s=s, n=int(c["n"]), eps=c["eps"], G=G, coef=coef,
                    coords=torch.zeros(3 * (2 * s + 1), dtype=F64, device=DEV))
    if kind == "recover":
        n, w = int(c["n"]), int(c["w"])
        ld = (n + 31) // 32 * 32
        Y = torch.zeros((w, ld), dtype=F64, device=DEV)
        Y[:, :n] = _basis_like(n, w, g)
        return dict(kind=kind, n=n, w=w, ld=ld, Y=Y, coords=_uniform(3 * w, g), x=_uniform(n, g),
                    r=torch.empty(n, dtype=F64, device=DEV), p=torch.empty(n, dtype=F64, device=DEV))
    if kind == "solve":
        op = _Op(_matrix(c, g))
        return dict(kind=kind, op=op, b=_rhs(op.n, g), x=torch.zeros(op.n, dtype=F64, device=DEV), opts=_solve_options(c))
    sys = _members(c, seed)
    ops = [_Op(_matrix(m, _gen(m["seed"]))) for m in sys]
    bs = [_rhs(o.n, _gen(m["seed"] + 1)) for o, m in zip(ops, sys)]
    st = dict(kind=kind, ops=ops, bs=bs, xs=[torch.zeros(o.n, dtype=F64, device=DEV) for o in ops],
              eps=[m["eps"] for m in sys],
              opts=P.make_options(method="adaptive", basis="monomial", s_max=int(c["s"]), max_iters=20000))
    if kind == "serve":
        st["srv"] = _Server(st["opts"])
    return st


class _Server:
    """A solve server with the scheduling the benchmark serves with, and an 8 GB budget."""

    def __init__(self, opts):
        self.h = P.ascg_server_create(opts, 8 << 30, 64)
        P.ascg_server_set_policy(self.h, P.ASCG_ADMIT_SHORTEST_FIRST, 1, True)

    def __del__(self):
        P.ascg_server_destroy(self.h)


def run(state):
    st, kind = state, state["kind"]
    if kind == "powers":
        P.ascg_matrix_powers(st["op"].h, st["s"], *st["coef"], st["Y"], st["Y"].shape[1])
        return st["Y"]
    if kind == "gram":
        P.ascg_gram(st["n"], st["w"], st["Y"], st["n"], st["G"])
        return st["G"]
    if kind == "block_step":
        info, hist = P.ascg_block_step(st["s"], st["G"], P.ASCG_ADAPTIVE, *st["coef"], st["n"], st["eps"], 1.0, 1,
                                       100000, 1.0, st["coords"])
        return dict(coords=st["coords"], hist=hist, sqrt_kappa=np.array(info.sqrt_kappa[: st["s"]]),
                    steps=np.array([info.stilde, info.s_k, info.stop]))
    if kind == "recover":
        f = P.ascg_recover_tc if st["w"] >= 9 else P.ascg_recover
        f(st["n"], st["w"], st["Y"], st["ld"], st["coords"], st["x"], st["r"], st["p"])
        return dict(x=st["x"], r=st["r"], p=st["p"])
    if kind == "solve":
        st["x"].zero_()
        res = P.ascg_solve(st["op"].h, st["b"], st["x"], st["opts"])
        return dict(x=st["x"], iters=res.iters)
    for x in st["xs"]:
        x.zero_()
    if kind == "batch":
        res, _ = P.ascg_solve_batch([o.h for o in st["ops"]], st["bs"], st["xs"], st["opts"], st["eps"])
        return dict(x=st["xs"], iters=np.array([r.iters for r in res]))
    srv, iters = st["srv"].h, np.zeros(len(st["ops"]), dtype=np.int64)
    for q, o in enumerate(st["ops"]):
        P.ascg_server_submit(srv, o.h, st["bs"][q], st["xs"][q], st["eps"][q], q)
    while True:
        done, active, pending = P.ascg_server_step(srv)
        for d in done:
            iters[d.tag] = d.result.iters
        if active == 0 and pending == 0:
            return dict(x=st["xs"], iters=iters)


# --- work and exact values ----------------------------------------------------

def _solve_work(c):
    """One read of A and b, one write of x; the flops of the CG iterations a solve takes, about a quarter of
    the Chebyshev bound sqrt(kappa) ln(2 / eps)."""
    n, nnz = _rows(c), _nnz(c)
    lo, hi = _bounds(c)
    it = min(n, 0.25 * math.sqrt(hi / lo) * math.log(2.0 / c["eps"]))
    return 12.0 * nnz + 24.0 * n, it * (2.0 * nnz + 10.0 * n)


def work(case):
    c, kind = case, case["kind"]
    if kind == "powers":
        n, nnz, s = _rows(c), _nnz(c), int(c["s"])
        return dict(bytes=12.0 * nnz + 8.0 * n * (2 * s + 1), flops=(2 * s - 1) * 2.0 * nnz)
    if kind in ("gram", "recover"):
        n, w = int(c["n"]), int(c["w"])
        return dict(bytes=8.0 * n * w + (0 if kind == "gram" else 32.0 * n), flops=n * w * (w + 1.0 if kind == "gram" else 6.0))
    if kind == "block_step":
        w = 2 * int(c["s"]) + 1
        return dict(bytes=8.0 * (w * w + 3 * w), flops=int(c["s"]) * 4.0 * w * w + sum(4.0 / 3.0 * (2 * i + 1) ** 3 for i in range(1, int(c["s"]) + 1)))
    one = [_solve_work(c)] if kind == "solve" else [_solve_work(m) for m in _members(c, 0)]
    return dict(bytes=sum(o[0] for o in one), flops=sum(o[1] for o in one))


def _sines(v, m, dim):
    """Type-I sine transform along every axis."""
    for ax in range(dim):
        z = torch.zeros_like(v.narrow(ax, 0, 1))
        v = torch.fft.fft(torch.cat([z, v, z, -v.flip(ax)], ax), dim=ax).imag.narrow(ax, 1, m) * -0.5
    return v


def _poisson_solution(c, b):
    """x with A x = b, from the sine transform that diagonalises A."""
    m, dim = int(c["size"]), 2 if c["family"] == "poisson2d" else 3
    one = 1.0 - torch.cos(torch.arange(1, m + 1, dtype=F64, device=DEV) * (math.pi / (m + 1)))
    lam = sum(one.reshape([m if a == k else 1 for a in range(dim)]) for k in range(dim)) / dim
    y = _sines(b.reshape([m] * dim), m, dim) / lam
    return (_sines(y, m, dim) * (2.0 / (m + 1)) ** dim).reshape(-1)


def _exact_block(c, seed):
    """The block in numpy: eigenvalues of the leading Gram blocks, the largest acceptable prefix, CG on coordinates."""
    G, (th, sg, gm) = _block_gram(c, seed)
    G, s, eps = G.cpu().numpy(), int(c["s"]), 2.0 ** -53
    w, tol = 2 * s + 1, c["eps"]
    kap = np.zeros(s)
    for i in range(1, s + 1):
        ev = np.linalg.eigvalsh(G[: 2 * i + 1, : 2 * i + 1])
        kap[i - 1] = np.inf if ev[0] <= (2 * i + 1) * math.sqrt(c["n"]) * eps * ev[-1] else math.sqrt(ev[-1] / ev[0])
    ok = kap <= tol / (eps * math.sqrt(G[1, 1]))
    st = max(1, s if ok.all() else int(np.argmin(ok)))
    B = np.zeros((w, w))
    for ch, last in ((0, s), (1, s - 1)):
        for j in range(last):
            B[2 * j + ch, 2 * j + ch] = th[j]
            B[2 * j + 2 + ch, 2 * j + ch] = gm[j]
            if j:
                B[2 * j - 2 + ch, 2 * j + ch] = sg[j - 1]
    x, r, p, hist = np.zeros(w), np.eye(w)[1], np.eye(w)[0], []
    rr, stop = r @ G @ r, 0
    for _ in range(st):
        q = B @ p
        al = rr / (p @ G @ q)
        x, r = x + al * p, r - al * q
        new = r @ G @ r
        p, be, rr = r + new / rr * p, new / rr, new
        nr = math.sqrt(max(rr, 0.0))
        hist.append((al, be, nr))
        if nr <= tol:
            stop = 1
            break
        if kap[st - 1] >= tol / (eps * nr):
            stop = 2
            break
    return dict(coords=torch.from_numpy(np.concatenate([x, r, p])), hist=np.array(hist).reshape(-1, 3), sqrt_kappa=kap,
                steps=np.array([st, len(hist), stop]))


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "block_step":
        return _exact_block(c, seed)
    if kind == "gram":
        Y = _basis_like(int(c["n"]), int(c["w"]), _gen(seed))
        return Y @ Y.T
    g = _gen(seed)
    if kind == "recover":
        n, w = int(c["n"]), int(c["w"])
        Y, k, x = _basis_like(n, w, g), _uniform(3 * w, g), _uniform(n, g)
        v = k.reshape(3, w) @ Y
        return dict(x=x + v[0], r=v[1], p=v[2])
    if kind == "powers":
        rowptr, colind, val = _matrix(c, g)
        n, s = rowptr.numel() - 1, int(c["s"])
        A = torch.sparse_csr_tensor(rowptr, colind.to(torch.int64), val, (n, n), dtype=F64, device=DEV)
        Y = torch.zeros((2 * s + 1, n), dtype=F64, device=DEV)
        Y[0], Y[1] = _rhs(n, g), _rhs(n, g)
        th, sg, gm = _coefficients(c)
        for k in range(2, 2 * s + 1):
            j = k // 2 - 1
            v = torch.mv(A, Y[k - 2]) - float(th[j]) * Y[k - 2]
            if j:
                v = v - float(sg[j - 1]) * Y[k - 4]
            Y[k] = v / float(gm[j])
        return Y
    if kind == "solve":
        if not c["family"].startswith("poisson"):
            return None
        return dict(x=_poisson_solution(c, _rhs(_rows(c), g)), iters=None)
    sys = _members(c, seed)
    return dict(x=[_poisson_solution(m, _rhs(_rows(m), _gen(m["seed"] + 1))) if m["family"].startswith("poisson") else None
                   for m in sys], iters=None)
