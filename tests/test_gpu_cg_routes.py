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
