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
