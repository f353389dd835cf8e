"""Batches whose systems sum their rows in different ways in one launch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _banded(n, h, seed):
    """Symmetric, half-bandwidth h, diagonal = row sum + 1."""
    rng = np.random.default_rng(seed)
    h = min(h, n - 1)
    vals = np.zeros((n, 2 * h + 1))
    for k in range(1, h + 1):
        u = -rng.random(n - k)
        vals[: n - k, h + k] = u
        vals[k:, h - k] = u
    vals[:, h] = np.abs(vals).sum(1) + 1.0
    cols = np.arange(n)[:, None] + np.arange(-h, h + 1)[None, :]
    keep = (cols >= 0) & (cols < n)
    rowptr = np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int64)
    return rowptr, cols[keep].astype(np.int32), vals[keep]


@pytest.mark.parametrize("s", [1, 3, 8])
def test_each_system_by_its_own_rows(s):
    """Short rows with both chains in a thread beside long rows by chain, at the edges of slices and items (rows 1 .. 129,
    and around 1024 where the Gram takes the tensor cores): x, iterations and blocks are those of each system alone, bit for
    bit (alone every system here but the first is summed by chain)."""
    import paper_1701_03989_gb300 as P

    sizes = [(210001, 1), (1, 0), (31, 25), (33, 30), (64, 1), (65, 21), (127, 22), (129, 40), (1023, 30), (1025, 30), (3000, 33),
             (777, 2), (5001, 1)]
    members = []
    for k, (n, h) in enumerate(sizes):
        rp, ci, v = _banded(n, h, k)
        b = torch.from_numpy(np.random.default_rng(100 + k).uniform(-1, 1, n)).cuda()
        members.append((P.ascg_op_create_csr(n, len(v), rp, ci, v, 0), b))
    o = P.make_options(s_max=s, eps_target=1e-11, max_iters=400)

    def run(group):
        xs = [torch.zeros_like(b) for _, b in group]
        res, st = P.ascg_solve_batch([op for op, _ in group], [b for _, b in group], xs, o)
        assert st == P.ASCG_OK
        return [(x.cpu().numpy(), r.iters, r.blocks) for x, r in zip(xs, res)]

    mixed = run(members)
    for k, m in enumerate(members):
        x, it, bl = run([m])[0]
        assert (it, bl) == mixed[k][1:] and np.array_equal(x, mixed[k][0]), sizes[k]
    for op, _ in members:
        P.ascg_op_destroy(op)
