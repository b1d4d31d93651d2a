"""The CG iterations' routes: what each costs beside the others, and that they agree."""
import time

import numpy as np
import pytest
import torch

from paper_1801_01134_gb300 import inputs, spc5

pytestmark = pytest.mark.gpu


def grid27(N):
    """27-point grid Laplacian with a little on the diagonal (values exact in bfloat16): slow to converge."""
    A = inputs.stencil3d(N, N, N, points=27, normal_values=False)
    row = np.repeat(np.arange(A.n), np.diff(A.rowptr))
    return inputs.CSR(A.n, A.m, A.rowptr, A.colidx, np.where(A.colidx == row, 26.0, -1.0))


def convert(A, dtype, r, c, **kw):
    d = spc5.upload_csr(A, dtype, "cuda")
    return spc5.convert(d.rowptr, d.colidx, d.values, A.n, A.m, r, c, **kw)


def seconds(f, reps=4):
    t = []
    for _ in range(reps):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        f()
        torch.cuda.synchronize()
        t.append(time.perf_counter() - t0)
    return min(t)


def test_bfloat16_rows_cost_no_more_than_float32(cuda_device):
    A = grid27(96)
    M = convert(A, torch.float64, 2, 4)
    b = torch.from_numpy(inputs.vec_uniform(A.n, seed=1)).cuda()
    # 200 iterations: 52 us each in float32, 47 in bfloat16 (85 where every load waited for the last)
    run = {t: seconds(lambda: spc5.cg(M, b, A_inner=L, tol=1e-25, max_iters=200, reliable=True))
           for t in (torch.float32, torch.bfloat16) for L in [convert(A, t, 2, 4)]}
    assert run[torch.bfloat16] <= 1.25 * run[torch.float32]


def scattered(n, per):
    """n rows of `per` entries spread over all columns, the diagonal among them (on the GPU)."""
    g = torch.Generator("cuda").manual_seed(n)
    cols = torch.randint(0, n // per, (n, per), generator=g, device="cuda") + torch.arange(per, device="cuda") * (n // per)
    i = torch.arange(n, device="cuda")
    cols[i, (i // (n // per)).clamp(max=per - 1)] = i
    cols = cols.sort(1).values
    vals = torch.where(cols == i[:, None], per - 1.0 + 1e-4, -1.0).double()
    return torch.arange(n + 1, device="cuda") * per, cols.int().reshape(-1), vals.reshape(-1)


def test_scattered_float64_rows_keep_their_loads_on_the_way(cuda_device):
    n = 2000000
    rowptr, cols, vals = scattered(n, 8)
    M = spc5.convert(rowptr, cols, vals, n, n, 1, 4)
    L = spc5.convert(rowptr, cols, vals.float(), n, n, 1, 4)
    b = torch.rand(n, dtype=torch.float64, device="cuda")
    # an iteration: float32 98 us, float64 122 (208 where its rows left the L1 no room)
    f64 = seconds(lambda: spc5.cg(M, b, tol=1e-25, max_iters=200))
    f32 = seconds(lambda: spc5.cg(M, b, A_inner=L, tol=1e-25, max_iters=200, reliable=True))
    assert f64 <= 1.6 * f32


@pytest.mark.parametrize("nz", [138, 139])  # 3,105,000 and 3,127,500 rows: either side of twenty rows per thread
def test_float64_rows_around_the_change_of_route(cuda_device, nz):
    A = inputs.poisson_shifted(150, 150, nz, seed=4)
    M = convert(A, torch.float64, 1, 4)
    b = torch.from_numpy(inputs.vec_uniform(A.n, seed=1)).cuda()
    x, info = spc5.cg(M, b, tol=1e-10)
    assert info["converged"] and info["rel_residual"] <= 1e-10
    y, again = spc5.cg(M, b, tol=1e-10, use_graph=True)
    assert again == info and torch.equal(x, y)


@pytest.mark.parametrize("inner,reliable,every", [(None, 0, 90), (torch.bfloat16, 0, 90), (torch.float32, 1, 8)])
def test_a_wait_that_runs_out_ends_in_the_separate_kernels(cuda_device, inner, reliable, every):
    import ctypes

    A = inputs.poisson_shifted(50, 50, 50, seed=4)
    M = convert(A, torch.float64, 2, 4)
    L = convert(A, inner, 2, 4) if inner is not None else None
    b = torch.from_numpy(inputs.vec_uniform(A.n, seed=1)).cuda()

    def solve(wait_us):
        x = torch.full_like(b, float("nan"))
        opts, info = spc5.CgOpts(tol=1e-10, check_every=every, reliable=reliable, wait_us=wait_us), spc5.CgInfo()
        status = spc5.load().spc5_cg(M._h, L._h if L else None, b.data_ptr(), x.data_ptr(), ctypes.byref(opts),
                                     ctypes.byref(info), None)
        assert status == spc5.OK and info.converged and info.rel_residual <= 1e-10
        return x, info

    x, info = solve(0)
    _, late = solve(1)
    if not reliable:
        assert info.iterations % every != 0  # the resident kernel stops at the tolerance
        assert late.iterations % every == 0 and late.iterations > 0  # the separate ones are looked at after 90
    y, again = solve(0)  # the library is as it was
    assert torch.equal(x, y) and again.iterations == info.iterations


@pytest.mark.parametrize("inner,reliable", [(None, False), (torch.float32, False), (torch.float32, True), (torch.bfloat16, True)])
def test_graph_and_plain_agree_bitwise_with_long_intervals(cuda_device, inner, reliable):
    # intervals of more than two blocks take the segment path, so the iterations run as separate
    # kernels: captured once and replayed (over all reliable updates), or launched one by one
    A = inputs.poisson_shifted(21, 20, 19, seed=4)
    kw = dict(long_blocks=2, seg_blocks=3)
    M = convert(A, torch.float64, 2, 4, **kw)
    L = convert(A, inner, 2, 4, **kw) if inner is not None else None
    assert M.arrays().nsegments > 0 and (L is None or L.arrays().nsegments > 0)
    b = torch.from_numpy(inputs.vec_uniform(A.n, seed=1)).cuda()
    plain, info = spc5.cg(M, b, A_inner=L, tol=1e-10, reliable=reliable)
    graph, again = spc5.cg(M, b, A_inner=L, tol=1e-10, reliable=reliable, use_graph=True)
    assert info["converged"] and again == info and torch.equal(plain, graph)
    assert not reliable or info["outer"] >= 2


def test_graph_and_plain_agree_bitwise_with_uneven_rows(cuda_device):
    # rows too uneven to lie side by side, none of them long
    n, hub = 40000, 60
    rows = [[0] + list(range(1, hub))] + [[0, i] if i < hub else [i] for i in range(1, n)]
    rowptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    cols = np.concatenate([np.asarray(r, np.int32) for r in rows])
    row = np.repeat(np.arange(n), np.diff(rowptr))
    A = inputs.CSR(n, n, rowptr, cols, np.where(cols == row, np.where(row == 0, 2.0 * hub, 2.0), 0.5))
    b = torch.from_numpy(inputs.vec_uniform(n, seed=1)).cuda()
    for kw in ({}, {"A_inner": convert(A, torch.float32, 1, 4), "reliable": True}):
        M = convert(A, torch.float64, 1, 4)
        assert M.arrays().nsegments == 0
        x, info = spc5.cg(M, b, tol=1e-10, **kw)
        y, again = spc5.cg(M, b, tol=1e-10, use_graph=True, **kw)
        assert info["converged"] and again == info and torch.equal(x, y)


@pytest.mark.parametrize("r,c", [(1, 4), (2, 4), (4, 8)])
def test_block_matrix(cuda_device, r, c):
    # dense 3 x 3 blocks around a band, symmetric and dominant: float64, and both precisions inside
    nb, bs = 700, 3
    rng = np.random.default_rng(5)
    pairs = {(i, i) for i in range(nb)}
    for i in range(nb):
        for j in rng.integers(max(0, i - 30), min(nb, i + 30), 6):
            pairs |= {(i, int(j)), (int(j), i)}
    D = {}
    for i, j in sorted(pairs):
        if i <= j:
            B = rng.uniform(-1, 1, (bs, bs))
            D[i, j], D[j, i] = (B, B.T) if i < j else (B + B.T, B + B.T)
    dense_rows, cols = [[] for _ in range(nb * bs)], [[] for _ in range(nb * bs)]
    for (i, j), B in sorted(D.items()):
        for a in range(bs):
            dense_rows[i * bs + a].extend(B[a])
            cols[i * bs + a].extend(range(j * bs, j * bs + bs))
    rowptr = np.concatenate([[0], np.cumsum([len(x) for x in cols])]).astype(np.int64)
    ci, vals = np.concatenate(cols).astype(np.int32), np.concatenate(dense_rows)
    row = np.repeat(np.arange(nb * bs), np.diff(rowptr))
    off = np.zeros(nb * bs)
    np.add.at(off, row, np.abs(vals))
    vals = np.where(ci == row, off[row] + 1.0, vals)
    A = inputs.CSR(nb * bs, nb * bs, rowptr, ci, vals)
    b = inputs.vec_uniform(A.n, seed=1)
    bd = torch.from_numpy(b).cuda()
    M = convert(A, torch.float64, r, c)
    for kw in ({}, {"A_inner": convert(A, torch.float32, r, c), "reliable": True}, {"A_inner": convert(A, torch.bfloat16, r, c)}):
        x, info = spc5.cg(M, bd, tol=1e-10, **kw)
        res = b - np.bincount(row, vals * x.cpu().numpy()[ci], A.n)
        assert info["converged"] and np.linalg.norm(res) <= 1.0001e-10 * np.linalg.norm(b)
