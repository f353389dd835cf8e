"""Kernels at the sizes where their tiling has edges: row lengths around the
groups of the row sums, rows around slices, items and CTAs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _banded(n, h, seed):
    """Symmetric, half-bandwidth h (row lengths h .. 2h off the diagonal), diagonal = row sum + 1."""
    rng = np.random.default_rng(seed)
    a = np.zeros((n, n))
    for k in range(1, min(h, n - 1) + 1):
        u = -rng.random(n - k)
        a[np.arange(n - k), np.arange(k, n)] = u
        a[np.arange(k, n), np.arange(n - k)] = u
    a[np.arange(n), np.arange(n)] = np.abs(a).sum(1) + 1.0
    keep = a != 0
    rowptr = np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int64)
    return a, rowptr, np.nonzero(keep)[1].astype(np.int32), a[keep]


@pytest.mark.parametrize("n", [1, 31, 33, 64, 65, 255, 257, 1025])
def test_batch_row_lengths(n):
    """Every row length from 0 to 18 in the items matrix powers: each solution against a dense solve.

    Tolerance: the diagonal exceeds the row sum by 1 and is at most 2h + 1 <= 19, so ||A^-1|| <= 1, ||A|| <= 38 and a
    relative residual of 1e-12 (4x slack for the updated residual's drift) bounds the error by 4e-12 ||b|| <= 152e-12 ||x||.
    """
    import paper_1701_03989_gb300 as P

    sys = [_banded(n, h, 100 * n + h) for h in range(10)]
    rng = np.random.default_rng(n)
    bs = [rng.uniform(-1, 1, n) for _ in sys]
    ops = [P.ascg_op_create_csr(n, len(v), rp, ci, v, 0) for _, rp, ci, v in sys]
    bd = [torch.from_numpy(b).cuda() for b in bs]
    xd = [torch.zeros(n, dtype=torch.float64, device="cuda") for _ in sys]
    res, st = P.ascg_solve_batch(ops, bd, xd, P.make_options(s_max=5, eps_target=1e-12, max_iters=2000))
    for o in ops:
        P.ascg_op_destroy(o)
    assert st == P.ASCG_OK
    for (a, *_), b, x in zip(sys, bs, xd):
        ref = np.linalg.solve(a, b)
        assert np.linalg.norm(x.cpu().numpy() - ref) <= 1.6e-10 * np.linalg.norm(ref)


def _diagonals(n, h, rng):
    """Integer band matrix as diagonals: main[n] in 1..4, off[k-1][n-k] in -2..2 without 0, k = 1..h."""
    main = rng.integers(1, 5, n).astype(np.float64)
    off = [rng.choice([-2.0, -1.0, 1.0, 2.0], max(n - k, 0)) for k in range(1, h + 1)]
    return main, off


def _apply(main, off, v):
    y = main * v
    for k, u in enumerate(off, 1):
        if len(u):
            y[: -k] += u * v[k:]
            y[k:] += u * v[: -k]
    return y


@pytest.mark.parametrize("h", [0, 1, 2, 3, 6, 9])
@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 65536, 65537])
def test_matrix_powers_exact_integers(n, h):
    """Small integers and powers of two: every result is an exact integer, so both kernels (a warp per chain up to 65536
    rows or for long rows, both chains in a thread otherwise) must give numpy's values bit for bit, whatever the order."""
    import paper_1701_03989_gb300 as P

    rng = np.random.default_rng(1000 * h + n)
    h = min(h, n - 1)
    main, off = _diagonals(n, h, rng)
    cols = np.arange(n)[:, None] + np.arange(-h, h + 1)[None, :]
    vals = np.zeros((n, 2 * h + 1))
    vals[:, h] = main
    for k, u in enumerate(off, 1):
        vals[: n - k, h + k] = u
        vals[k:, h - k] = u
    keep = (cols >= 0) & (cols < n)
    rowptr = np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int64)
    op = P.ascg_op_create_csr(n, int(rowptr[-1]), rowptr, cols[keep].astype(np.int32), vals[keep], 0)
    for s, th, sg, gm in ((1, [1.0], [0.0], [1.0]), (4, [0.0] * 4, [0.0] * 4, [1.0] * 4),
                          (4, [1.0, 2.0, 1.0, 3.0], [0.5, 0.5, 0.5, 0.5], [1.0, 0.5, 0.5, 0.5]),
                          (3, [1.0, 0.0, 2.0], [2.0, 4.0, 1.0], [0.5, 0.5, 0.5])):
        Y = np.zeros((2 * s + 1, n))
        Y[0], Y[1] = rng.integers(-3, 4, n), rng.integers(-3, 4, n)
        Yd = torch.from_numpy(Y.copy()).cuda()
        P.ascg_matrix_powers(op, s, np.array(th), np.array(sg), np.array(gm), Yd, n)
        for k in range(2, 2 * s + 1):
            j = k // 2 - 1
            v = _apply(main, off, Y[k - 2]) - th[j] * Y[k - 2]
            if j:
                v = v - sg[j - 1] * Y[k - 4]
            Y[k] = v / gm[j]
        assert np.array_equal(Yd.cpu().numpy(), Y), (s, th)
    P.ascg_op_destroy(op)


def test_scratch_of_concurrent_calls():
    """Single-step calls from several threads on streams of their own: each gives the bits it gives alone."""
    import threading

    import paper_1701_03989_gb300 as P

    g = torch.Generator(device="cuda").manual_seed(5)
    Ys = [torch.rand((w, 2048), dtype=torch.float64, device="cuda", generator=g) for w in (5, 9, 17, 33)]
    Gs = [torch.empty((len(Y), len(Y)), dtype=torch.float64, device="cuda") for Y in Ys]
    alone = []
    for Y, G in zip(Ys, Gs):
        P.ascg_gram(2048, len(Y), Y, 2048, G)
        alone.append(G.cpu())
    bad = []

    def work(k):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            G = torch.empty_like(Gs[k])
            for _ in range(50):
                P.ascg_gram(2048, len(Ys[k]), Ys[k], 2048, G, stream=s)
                if not torch.equal(G.cpu(), alone[k]):
                    bad.append(k)

    threads = [threading.Thread(target=work, args=(k % 4,)) for k in range(8)]
    torch.cuda.synchronize()
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


@pytest.mark.parametrize("s", range(1, 17))
@pytest.mark.parametrize("kind", ["dense", "diagonal"])
def test_condition_estimates_every_order(s, kind):
    """sqrt(kappa(G_{k,i})) for every order 3 .. 33 against numpy's eigenvalues.

    dense: random Gram matrices of condition below 1e8; diagonal: zero off-diagonals (every minor a product, the small ones
    rescaled, exact condition numbers). Tolerance: the multisection leaves relative brackets below 1e-9 for both ends, and
    rounding moves an eigenvalue by at most 64 w eps ||G||, so sqrt(kappa) is within 1e-9 + 32 w eps kappa relatively.
    """
    import paper_1701_03989_gb300 as P

    w, eps = 2 * s + 1, 2.0 ** -53
    rng = np.random.default_rng(s)
    if kind == "dense":
        Y = rng.standard_normal((200, w)) * 10.0 ** rng.uniform(-1.5, 0, w)
        G = Y.T @ Y
    else:
        G = np.diag(10.0 ** rng.uniform(-6, 0, w))
    G = (G + G.T) / 2
    Gd = torch.from_numpy(G.copy()).cuda()
    coords = torch.zeros(3 * w, dtype=torch.float64, device="cuda")
    info, _ = P.ascg_block_step(s, Gd, P.ASCG_ADAPTIVE, np.zeros(s), np.zeros(s), np.ones(s), 200, 1e-8, 1.0, 1, 100, 1.0,
                                coords)
    for i in range(1, s + 1):
        ev = np.linalg.eigvalsh(G[: 2 * i + 1, : 2 * i + 1])
        kappa = ev[-1] / ev[0]
        assert kappa < 1e8
        got = info.sqrt_kappa[i - 1]
        assert abs(got - np.sqrt(kappa)) <= (1e-9 + 32 * w * eps * kappa) * np.sqrt(kappa), (i, got, kappa)


def test_gram_pieces_do_not_change_a_bit():
    """A system's tensor-core Gram alone (its items cut into one-chunk pieces) and beside enough rows that no item is cut:
    the integer sums do not depend on the cut, so x and the iteration count are the same bit for bit."""
    import paper_1701_03989_gb300 as P

    def system(m, seed):
        n = m ** 3
        i = np.arange(n)
        cols, keep = [], []
        for s in (m * m, m, 1, 0, -1, -m, -m * m):
            cols.append(i - s)
            keep.append(np.ones(n, bool) if s == 0 else
                        (((i // abs(s)) % m > 0) if s > 0 else ((i // abs(s)) % m < m - 1)))
        cols, keep = np.stack(cols, 1), np.stack(keep, 1)
        vals = np.full((n, 7), -1.0 / 6)
        vals[:, 3] = 1.0
        rowptr = np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int64)
        op = P.ascg_op_create_csr(n, int(rowptr[-1]), rowptr, cols[keep].astype(np.int32), vals[keep], 0)
        b = np.random.default_rng(seed).uniform(-1, 1, n)
        return op, torch.from_numpy(b).cuda()

    small = [system(m, m) for m in (10, 13, 27, 33)]  # 1, 3, 20 and 36 chunks
    big = [system(103, 7), system(104, 8)]            # 2166 chunks: more than 256 items
    o = P.make_options(s_max=8, eps_target=1e-8, max_iters=60)

    def run(members):
        xs = [torch.zeros_like(b) for _, b in members]
        res, _ = P.ascg_solve_batch([op for op, _ in members], [b for _, b in members], xs, o)
        return [(x.cpu().numpy(), r.iters, r.blocks) for x, r in zip(xs, res)]

    mixed = run(small + big)
    for k, m in enumerate(small):
        x, it, bl = run([m])[0]
        assert (it, bl) == mixed[k][1:] and np.array_equal(x, mixed[k][0])
    for op, _ in small + big:
        P.ascg_op_destroy(op)


@pytest.mark.parametrize("method", ["fixed", "adaptive"])
@pytest.mark.parametrize("n", [1, 33, 131072, 131073])
def test_fp64_recovery_one_pass_and_split(n, method):
    """The FP64 recovery in one launch (up to 131072 rows) and in two, over many short blocks: the solution's true residual.

    Tolerance: the matrix is tridiagonal with diagonal 4 and off-diagonals -1 (condition below 3), so the updated residual,
    below 1e-12 at convergence, and the true one differ by a few hundred rounding errors of the iterates: 4x the target.
    """
    import paper_1701_03989_gb300 as P

    keep = np.ones((n, 3), bool)
    keep[0, 0] = keep[-1, 2] = False
    cols = np.arange(n)[:, None] + np.arange(-1, 2)[None, :]
    vals = np.broadcast_to(np.array([-1.0, 4.0, -1.0]), (n, 3))
    rowptr = np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int64)
    op = P.ascg_op_create_csr(n, int(rowptr[-1]), rowptr, cols[keep].astype(np.int32), vals[keep], 0)
    b = np.random.default_rng(n).uniform(-1, 1, n)
    x = torch.zeros(n, dtype=torch.float64, device="cuda")
    res = P.ascg_solve(op, torch.from_numpy(b).cuda(), x, P.make_options(method=method, s_max=3, eps_target=1e-12,
                                                                          gram_fp64=True, max_iters=500))
    P.ascg_op_destroy(op)
    x = x.cpu().numpy()
    r = b - 4.0 * x
    r[1:] += x[:-1]
    r[:-1] += x[1:]
    assert res.status == P.ASCG_OK and res.blocks >= min(n, 3) / 3
    assert np.linalg.norm(r) <= 4e-12 * np.linalg.norm(b)


@pytest.mark.parametrize("k", [1, 2, 3, 5, 6, 17, 31, 32])
def test_newton_shifts_every_value(k):
    """All k Ritz values (five bisection levels a round, one CTA a value) against numpy's eigenvalues of the tridiagonal.

    Bisection ends at neighbouring doubles of the Sturm count's own tridiagonal, which is within a few eps ||T|| of the
    exact one, as is numpy's: 32 k eps ||T|| covers both.
    """
    import paper_1701_03989_gb300 as P

    rng = np.random.default_rng(k)
    al, be = rng.uniform(0.3, 3.0, k), rng.uniform(0.01, 1.5, max(k - 1, 1))
    d = 1 / al
    d[1:] += be[: k - 1] / al[: k - 1]
    e = np.sqrt(be[: k - 1]) / al[: k - 1]
    ev = np.linalg.eigvalsh(np.diag(d) + np.diag(e, 1) + np.diag(e, -1))
    got = P.ascg_newton_shifts(al, be, k, k)
    assert abs(got[0]) == max(abs(got))
    assert np.max(np.abs(np.sort(got) - ev)) <= 32 * k * 2.0 ** -53 * np.max(np.abs(ev))


@pytest.mark.parametrize("h", [1, 5, 6, 40])
@pytest.mark.parametrize("n", [31, 257, 5000])
def test_classical_row_lengths(n, h):
    """Classical CG with short rows and with rows long enough for the pipelined row sums, against a dense solve (tolerance
    as in test_batch_row_lengths: ||A^-1|| <= 1, ||A|| <= 2 (2h + 1) + 1 <= 163)."""
    import paper_1701_03989_gb300 as P

    if n == 5000 and h != 40:
        pytest.skip("one dense solve of this size is enough")
    a, rp, ci, v = _banded(n, h, n + h)
    b = np.random.default_rng(n).uniform(-1, 1, n)
    op = P.ascg_op_create_csr(n, len(v), rp, ci, v, 0)
    x = torch.zeros(n, dtype=torch.float64, device="cuda")
    res = P.ascg_solve(op, torch.from_numpy(b).cuda(), x, P.make_options(method="classical", eps_target=1e-12, max_iters=5000))
    P.ascg_op_destroy(op)
    ref = np.linalg.solve(a, b)
    assert res.status == P.ASCG_OK
    assert np.linalg.norm(x.cpu().numpy() - ref) <= 4e-12 * 163 * np.linalg.norm(ref)
