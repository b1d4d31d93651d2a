"""The library's memory pools beside other users of the device's memory."""
import pytest
import torch

from paper_1801_01134_gb300 import spc5

pytestmark = pytest.mark.gpu
GB = 1 << 30


def tridiagonal(n):
    """Rowptr, columns and values (2.5 and -1) of an n x n tridiagonal matrix, on the GPU."""
    i = torch.arange(n, device="cuda", dtype=torch.int32)
    cols = torch.stack([i - 1, i, i + 1], 1).reshape(-1)[1:-1].contiguous()
    vals = torch.tensor([-1.0, 2.5, -1.0], dtype=torch.float64, device="cuda").repeat(n)[1:-1].contiguous()
    rowptr = (torch.arange(n + 1, device="cuda") * 3 - 1).clamp(min=0)
    rowptr[n] -= 1
    return rowptr, cols, vals


@pytest.fixture
def clean(cuda_device):
    def sweep():
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        spc5.pool_trim()

    sweep()
    yield
    sweep()


def test_a_solve_gives_its_workspace_back(clean):
    n = 30000000
    rowptr, cols, vals = tridiagonal(n)
    M = spc5.convert(rowptr, cols, vals, n, n, 1, 4)
    L = spc5.convert(rowptr, cols, vals.float(), n, n, 1, 4)
    del rowptr, cols, vals
    b = torch.ones(n, dtype=torch.float64, device="cuda")
    x = torch.empty_like(b)
    spc5.pool_trim()
    free = torch.cuda.mem_get_info()[0]
    # four vectors of 240 MB, five of 120, 90 million unpacked entries of 8 bytes: over 2.2 GB
    _, info = spc5.cg(M, b, A_inner=L, x=x, tol=1e-8, reliable=True)
    assert info["converged"]
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] <= GB + GB // 8  # what the pool may keep, and some
    spc5.pool_trim()
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] <= GB // 8
