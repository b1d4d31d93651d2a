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
