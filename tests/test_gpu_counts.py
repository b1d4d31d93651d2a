"""Block counts of the twelve shapes at the edges of the counting steps, against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_1801_01134_gb300 import inputs, spc5

pytestmark = pytest.mark.gpu


def csr(rows, m):
    rowptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    cols = np.concatenate([np.asarray(r, np.int32) for r in rows] + [np.zeros(0, np.int32)])
    return inputs.CSR(len(rows), m, rowptr, cols, np.ones(cols.size))


def random_rows(lengths, m, seed):
    rng = np.random.default_rng(seed)
    return [np.sort(rng.choice(m, size=k, replace=False)) for k in lengths]


CASES = {
    # eight rows of exactly a step's entries, and one entry more
    "full_step": lambda: csr(random_rows([256] * 16, 5000, 1), 5000),
    "over_a_step": lambda: csr(random_rows([256] * 7 + [257] + [3] * 9, 5000, 2), 5000),
    # hubs among short rows, a last group of five rows, empty rows between
    "hubs": lambda: csr(random_rows([0, 4, 9000, 2, 0, 7, 3000, 1] + [5] * 130 + [0] * 40 + [6000, 3, 1, 2, 8], 40000, 3), 40000),
    # long rows without a gap of 16: no column where the group can be cut
    "dense_hub": lambda: csr([np.arange(k % 3, 7000 + k) for k in range(8)] + random_rows([3] * 5, 8000, 4), 8000),
    # and with one cut in the middle
    "dense_halves": lambda: csr([np.concatenate([np.arange(0, 2500), np.arange(2516 + k, 6000)]) for k in range(9)], 6000),
    # runs of every length and gap around 4, 8 and 16
    "gaps": lambda: csr([np.cumsum(np.tile([1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17], 12)[i:i + 90]) for i in range(29)], 4000),
    # equal columns in all rows of a group; the last column of a wide matrix
    "equal_rows": lambda: csr([np.array([0, 5, 21, 2**31 - 20, 2**31 - 3, 2**31 - 2])] * 11, 2**31 - 1),
    "one_row": lambda: csr([np.arange(0, 9000, 3)], 9000),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_counts_match_oracle(cuda_device, name):
    A = CASES[name]()
    d = spc5.upload_csr(A, torch.float64, "cuda")
    got = spc5.count_blocks(d.rowptr, d.colidx, A.n, A.m)
    want = [oracle.beta_count(A, r, c)[1] for r, c in spc5.SHAPES]
    assert list(got) == want
    f = spc5.features(d)
    lens = np.diff(A.rowptr)
    assert f[12] == lens.mean() and f[14] == lens.max()
    assert abs(f[13] - lens.std()) <= 1e-9 * max(1.0, lens.std())
