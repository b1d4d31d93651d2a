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
