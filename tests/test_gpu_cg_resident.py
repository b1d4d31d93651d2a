"""The resident CG iterations at the edges of their layout: ragged row counts, every block shape,
uneven rows, more rows than the shared memory holds."""
import numpy as np
import pytest
import torch

from paper_1801_01134_gb300 import inputs, spc5

pytestmark = pytest.mark.gpu


def spd(n, seed, per_row=3):
    """Symmetric, strictly dominant, random pattern: diag > sum of the absolute off-diagonal entries."""
    rng = np.random.default_rng(seed)
    i = np.repeat(np.arange(n), per_row)
    j = rng.integers(0, n, n * per_row)
    keep = i != j
    i, j = i[keep], j[keep]
    key = np.unique(np.minimum(i, j) * n + np.maximum(i, j))
    a, b = key // n, key % n
    v = rng.uniform(-1.0, 1.0, key.size)
    rows, cols, vals = np.concatenate([a, b, np.arange(n)]), np.concatenate([b, a, np.arange(n)]), np.concatenate([v, v, np.zeros(n)])
    off = np.zeros(n)
    np.add.at(off, rows, np.abs(vals))
    vals[2 * key.size:] = off + 1.0 + rng.random(n)
    order = np.lexsort((cols, rows))
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=n))]).astype(np.int64)
    return inputs.CSR(n, n, rowptr, cols[order].astype(np.int32), vals[order])


def arrow(n, hub):
    """A hub row and column of `hub` entries beside a diagonal: rows far too uneven to lie side by side."""
    rows = [[0] + list(range(1, hub))] + [[0, i] if i < hub else [i] for i in range(1, n)]
    rowptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    cols = np.concatenate([np.asarray(r, np.int32) for r in rows])
    row = np.repeat(np.arange(n), np.diff(rowptr))
    vals = np.where(cols == row, np.where(row == 0, 2.0 * hub, 2.0), 0.5)
    return inputs.CSR(n, n, rowptr, cols, vals)


def solve(A, r, c, low=None, reliable=False, **kw):
    d = spc5.upload_csr(A, torch.float64, "cuda")
    M = spc5.convert(d.rowptr, d.colidx, d.values, A.n, A.m, r, c)
    L = None
    if low is not None:
        dl = spc5.upload_csr(A, low, "cuda")
        L = spc5.convert(dl.rowptr, dl.colidx, dl.values, A.n, A.m, r, c)
    b = torch.from_numpy(inputs.vec_uniform(A.n, seed=1)).cuda()
    x, info = spc5.cg(M, b, A_inner=L, tol=1e-10, reliable=reliable, **kw)
    row = torch.repeat_interleave(torch.arange(A.n, device="cuda"), d.rowptr[1:] - d.rowptr[:-1])
    res = b - torch.zeros_like(b).index_add_(0, row, d.values * x[d.colidx.long()])
    return x, info, float(res.norm() / b.norm())


@pytest.mark.parametrize("r,c", spc5.SHAPES)
@pytest.mark.parametrize("n", [1, 31, 33, 511, 1029])
def test_shapes_and_ragged_sizes(cuda_device, r, c, n):
    A = spd(n, seed=n)
    # float64 stops at the recurred norm, which follows the true one to rounding
    for low, reliable in ((None, False), (torch.float32, True), (torch.bfloat16, False)):
        x, info, rel = solve(A, r, c, low, reliable)
        assert info["converged"] and rel <= 1.0001e-10, (low, reliable, rel)


def test_uneven_rows_take_the_separate_kernels(cuda_device):
    A = arrow(40000, 60)
    for low, reliable in ((None, False), (torch.float32, True)):
        x, info, rel = solve(A, 1, 4, low, reliable)
        assert info["converged"] and rel <= 1.0001e-10


def test_more_rows_than_the_shared_memory_holds(cuda_device):
    A = inputs.poisson_shifted(120, 110, 105, seed=4)  # 1.39 million rows: 9 per thread, float64 holds 7
    x, info, rel = solve(A, 1, 4)
    assert info["converged"] and rel <= 1.0001e-10
    y, again, _ = solve(A, 1, 4)
    assert again == info and torch.equal(x, y)


def test_iteration_limit_and_exact_stop(cuda_device):
    A = inputs.poisson_shifted(30, 30, 30, seed=4)
    _, full, _ = solve(A, 2, 4)
    _, cut, rel = solve(A, 2, 4, max_iters=full["iterations"] - 1)
    assert cut["iterations"] == full["iterations"] - 1 and not cut["converged"] and rel > 1e-10
