"""CSR -> beta(r,c) for r > 1 at the edges of the shared-memory tiles, bit for bit against the oracle."""
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
    "one_row": lambda: csr([7], 30, 1),
    "ragged": lambda: csr(list(np.random.default_rng(2).integers(0, 40, 1031)), 900, 2, run=2),
    # eight rows of 4096 entries together, one more, and hubs among short rows
    "full_tile": lambda: csr([512] * 8 + [3] * 5, 3000, 3),
    "over_a_tile": lambda: csr([512] * 7 + [513] + [3] * 13, 3000, 4),
    "hubs": lambda: csr([2, 9000, 0, 5] + [6] * 700 + [4000, 4200, 1, 0, 2], 20000, 5),
    "dense": lambda: csr([300] * 150, 300, 6),
    "empty": lambda: csr([0] * 130, 10, 7),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("r,c", [s for s in spc5.SHAPES if s[0] > 1])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32, torch.bfloat16])
def test_bit_exact(cuda_device, name, r, c, dtype):
    A = CASES[name]()
    B = oracle.beta_convert(A, r, c)
    d = spc5.upload_csr(A, dtype, "cuda")
    M = spc5.convert(d.rowptr, d.colidx, d.values, A.n, A.m, r, c, long_blocks=50, seg_blocks=7)
    got = M.export()
    assert np.array_equal(got["block_rowptr"], B.block_rowptr) and np.array_equal(got["block_colidx"], B.block_colidx)
    assert np.array_equal(got["block_masks"], B.block_masks)
    want = torch.from_numpy(B.values).to(dtype)
    raw = {8: torch.int64, 4: torch.int32, 2: torch.int16}[want.element_size()]
    assert np.array_equal(got["values_raw"].view(np.int64 if raw == torch.int64 else np.int32 if raw == torch.int32 else np.int16),
                          want.view(raw).numpy())
    x = inputs.vec_uniform(A.m, seed=1)
    if dtype == torch.float64:  # the segments' first values, too
        y = M.spmv(torch.from_numpy(x).cuda()).cpu().numpy()
        ref, S = oracle.csr_spmv_dot2(A, x)
        assert np.all(np.abs(y - ref) <= 1e-13 * S)


@pytest.mark.parametrize("r", [2, 4, 8])
def test_bad_csr_is_named(cuda_device, r):
    for spoil, status in ((lambda c, p: c.__setitem__(p, c[p - 1]), spc5.EDUP), (lambda c, p: c.__setitem__(p, -1), spc5.ERANGE),
                          (lambda c, p: c.__setitem__(p, c[p - 1] - 1), spc5.EUNSORTED)):
        A = CASES["hubs"]()
        for row in (1, 500):  # a hub walked in global memory, a row in a tile
            cols = A.colidx.copy()
            spoil(cols, int(A.rowptr[row]) + 3)
            d = spc5.upload_csr(inputs.CSR(A.n, A.m, A.rowptr, cols, A.values), torch.float64, "cuda")
            with pytest.raises(spc5.Spc5Error) as e:
                spc5.convert(d.rowptr, d.colidx, d.values, A.n, A.m, r, 4)
            assert e.value.status == status and f"row {row}:" in str(e.value)
