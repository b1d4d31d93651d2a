"""CSR -> beta(r,c) for r > 1 where intervals go from the tiles to the list, bit for bit against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_1801_01134_gb300 import inputs, spc5

pytestmark = pytest.mark.gpu


def csr(lengths, m, seed, run=1):
    rng = np.random.default_rng(seed)
    rows = []
    for k in lengths:
        starts = np.sort(rng.choice(m // run, size=-(-k // run), replace=False)) * run
        rows.append((starts[:, None] + np.arange(run)).reshape(-1)[:k])
    rowptr = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    cols = np.concatenate(rows + [np.zeros(0, np.int64)]).astype(np.int32)
    return inputs.CSR(len(lengths), m, rowptr, cols, rng.standard_normal(cols.size))


CASES = {
    # intervals of exactly 512 and 1024 entries for each r, and one more
    "limits": lambda: csr([256] * 8 + [257, 255, 3, 256] + [128] * 8 + [129] + [64] * 7 + [127, 128, 130, 128] * 2 + [0] * 5, 3000, 1),
    # long means: a few intervals, down to one, per thread block
    "rows_of_90": lambda: csr([90 + k % 3 for k in range(300)], 2000, 2),
    "rows_of_200": lambda: csr([200 + k % 5 for k in range(101)], 2500, 3, run=2),
    # short rows, more than a thread block's intervals; listed ones first, last and between
    "among_short": lambda: csr([700] + [2, 0, 1] * 120 + [600, 600] + [3] * 37 + [900], 5000, 4),
    "all_listed": lambda: csr([530] * 33, 4000, 5, run=3),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("r,c", [s for s in spc5.SHAPES if s[0] > 1])
@pytest.mark.parametrize("dtype", [torch.float64, torch.bfloat16])
def test_bit_exact(cuda_device, name, r, c, dtype):
    A = CASES[name]()
    B = oracle.beta_convert(A, r, c)
    d = spc5.upload_csr(A, dtype, "cuda")
    M = spc5.convert(d.rowptr, d.colidx, d.values, A.n, A.m, r, c, long_blocks=50, seg_blocks=7)
    got = M.export()
    assert np.array_equal(got["block_rowptr"], B.block_rowptr) and np.array_equal(got["block_colidx"], B.block_colidx)
    assert np.array_equal(got["block_masks"], B.block_masks)
    raw = np.int64 if dtype == torch.float64 else np.int16
    want = torch.from_numpy(B.values).to(dtype).view(torch.int64 if dtype == torch.float64 else torch.int16).numpy()
    assert np.array_equal(got["values_raw"].view(raw), want)
    if dtype == torch.float64:  # the segments' first values, too
        x = inputs.vec_uniform(A.m, seed=1)
        y = M.spmv(torch.from_numpy(x).cuda()).cpu().numpy()
        ref, S = oracle.csr_spmv_dot2(A, x)
        assert np.all(np.abs(y - ref) <= 1e-13 * S)


@pytest.mark.parametrize("r", [2, 4])
def test_rows_of_600_entries_do_not_wait_for_one_another(cuda_device, r):
    # against the r = 1 conversion of the same matrix, whose work per entry is the least: about 5 times its
    # time; walked a few intervals at a time by 157 thread blocks, 47 times (r = 2) and 270 times (r = 4)
    n, k = 20000, 600
    rowptr = torch.arange(n + 1, device="cuda") * k
    cols = (torch.arange(n * k, device="cuda") % k * 160 + torch.randint(0, 160, (n * k,), device="cuda")).int()
    vals = torch.ones(n * k, device="cuda")

    def ms(r):
        t = []
        for _ in range(4):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            spc5.convert(rowptr, cols, vals, n, k * 160, r, 4).destroy()
            e[1].record()
            torch.cuda.synchronize()
            t.append(e[0].elapsed_time(e[1]))
        return min(t)

    assert ms(r) <= 20 * ms(1)
