"""Block counts at the column limit, against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_1801_01134_gb300 import inputs, spc5

pytestmark = pytest.mark.gpu

TOP = 2**31 - 1  # the largest m: the last column is TOP - 1


def csr(rows, m):
    rowptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    cols = np.concatenate([np.asarray(r, np.int32) for r in rows] + [np.zeros(0, np.int32)])
    return inputs.CSR(len(rows), m, rowptr, cols, np.ones(cols.size))


LIMIT = {
    # a row's only entry, every distance from the last column; single entries and runs
    "alone": lambda: csr([[TOP - 1 - k] for k in range(40)], TOP),
    "first_of_a_run": lambda: csr([[TOP - 40 + k, TOP - 3] for k in range(30)], TOP),
    "last_sixteen": lambda: csr([np.arange(TOP - 16, TOP)] * 9 + [[]] + [[0, TOP - 1]] * 3, TOP),
    # a group of several steps whose last column is the limit
    "hub": lambda: csr([np.arange(TOP - 9000 - k, TOP, 3) for k in range(8)], TOP),
}


@pytest.mark.parametrize("name", sorted(LIMIT))
def test_columns_up_to_the_limit(cuda_device, name):
    A = LIMIT[name]()
    d = spc5.upload_csr(A, torch.float64, "cuda")
    got = spc5.count_blocks(d.rowptr, d.colidx, A.n, A.m)
    assert list(got) == [oracle.beta_count(A, r, c)[1] for r, c in spc5.SHAPES]


def still_works():
    A = LIMIT["hub"]()
    d = spc5.upload_csr(A, torch.float64, "cuda")
    assert list(spc5.count_blocks(d.rowptr, d.colidx, A.n, A.m)) == [oracle.beta_count(A, r, c)[1] for r, c in spc5.SHAPES]


def test_row_pointers_that_fall_back(cuda_device):
    # every second 128 rows fall back to 0: the others, valid by themselves, hold four
    # times nnz entries in long groups, more ranges than a valid CSR can have
    nnz = 200000
    rowptr = np.zeros(128 * 8 + 1, np.int64)
    for piece in range(0, 8, 2):
        rowptr[128 * piece + 1:128 * (piece + 1) + 1] = nnz
    A = inputs.CSR(rowptr.size - 1, nnz, rowptr, np.arange(nnz, dtype=np.int32), np.ones(nnz))
    d = spc5.upload_csr(A, torch.float32, "cuda")
    spc5.count_blocks(d.rowptr, d.colidx, A.n, A.m)
    spc5.features(d)
    with pytest.raises(spc5.Spc5Error) as e:
        spc5.tune(d)
    assert e.value.status == spc5.EINVAL and "row 128:" in str(e.value)
    still_works()


def test_hubs_with_columns_out_of_order(cuda_device):
    # the cuts of such a group do not ascend: a range can end before it starts in one row
    # and hold thousands of entries in another
    rng = np.random.default_rng(0)
    rows = [rng.permutation(2_000_000)[:k] for k in (30000, 30000, 5, 2, 20000, 3, 9, 1)]
    rows += [rng.permutation(50_000)[:k] for k in (9, 0, 7000, 6000, 5000, 4000, 3000, 2500)]
    A = csr(rows + [np.arange(40)] * 5, 2_000_000)
    d = spc5.upload_csr(A, torch.float32, "cuda")
    spc5.count_blocks(d.rowptr, d.colidx, A.n, A.m)
    spc5.features(d)
    with pytest.raises(spc5.Spc5Error) as e:
        spc5.tune(d)
    assert e.value.status == spc5.EUNSORTED and "row 0:" in str(e.value)
    still_works()
