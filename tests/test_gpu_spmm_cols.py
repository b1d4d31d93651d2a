"""SpMM with column groups, whole aligned tiles (packed multiply-adds, unrolled blocks, segments four
blocks at a time, sorted order) and partial or unaligned ones, against the oracle, column by column."""
import numpy as np
import pytest
import torch

import oracle
from paper_1801_01134_gb300 import inputs, spc5

pytestmark = pytest.mark.gpu


def csr(lengths, m, seed, run=1):
    """Rows of the given lengths at random columns, in runs of `run` adjacent ones."""
    rng = np.random.default_rng(seed)
    rows = []
    for k in lengths:
        starts = np.sort(rng.choice(m // run, size=-(-k // run), replace=False)) * run
        rows.append((starts[:, None] + np.arange(run)).reshape(-1)[:k])
    rowptr = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    cols = np.concatenate(rows + [np.zeros(0, np.int64)]).astype(np.int32)
    return inputs.CSR(len(lengths), m, rowptr, cols, rng.standard_normal(cols.size))


def uneven(seed):
    rng = np.random.default_rng(seed)
    return list(np.where(rng.random(700) < 0.4, 0, rng.geometric(0.08, 700)))


CASES = {
    # (matrix, conversion options): one row; rows of 2048 entries and more; rows of a few dozen
    "one": (lambda: csr([5], 50, 1), {}),
    "full_step": (lambda: csr([2048] + [1] * 130 + [2047, 3], 3000, 2), {"long_blocks": 4096, "long_values": 2048}),
    "over_a_step": (lambda: csr([2049, 4], 3000, 3), {"long_blocks": 4096, "long_values": 4000}),
    "many_steps": (lambda: csr([60, 61, 0, 64] * 70, 2000, 4, run=4), {}),
    # empty rows, short rows, hubs in between, a last block of a few rows
    "uneven": (lambda: csr(uneven(5) + [900, 0, 0, 3, 1500] + uneven(6) + [0] * 3, 4000, 7), {}),
    "segments": (lambda: csr(uneven(8), 900, 9, run=3), {"long_blocks": 3, "seg_blocks": 33}),
    "sorted": (lambda: csr(uneven(11) + [900], 4000, 12), {"variant": 10, "order_window": 256}),
    "all_empty": (lambda: csr([0] * 300, 40, 10), {}),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("r,c", [(1, 4), (1, 8), (1, 16), (2, 4), (4, 8), (8, 16)])
@pytest.mark.parametrize("k,ktile,pad", [(4, 8, 0), (8, 8, 0), (13, 8, 1), (20, 16, 4), (32, 32, 0), (35, 32, 1)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32, torch.bfloat16])
def test_column_groups(cuda_device, name, r, c, k, ktile, pad, dtype):
    make, opts = CASES[name]
    A = make()
    rnd = {torch.float64: lambda a: a, torch.float32: oracle.round_f32, torch.bfloat16: oracle.round_bf16}[dtype]
    A = inputs.CSR(A.n, A.m, A.rowptr, A.colidx, rnd(A.values))
    X = inputs.vec_uniform(A.m * k, seed=k).reshape(A.m, k)
    if dtype != torch.float64:
        X = oracle.round_f32(X)
    Yref, S = oracle.csr_spmm_dot2(A, X)
    d = spc5.upload_csr(A, dtype, "cuda")
    M = spc5.convert(d.rowptr, d.colidx, d.values, A.n, A.m, r, c, **opts)
    xdt = torch.float64 if dtype == torch.float64 else torch.float32
    Xd = torch.zeros(A.m, k + pad, dtype=xdt, device="cuda")
    Xd[:, :k] = torch.from_numpy(X)
    Yd = torch.full((A.n, k + pad), float("nan"), dtype=xdt, device="cuda")
    M.spmm(Xd[:, :k], Yd[:, :k], ktile=ktile)
    Y = Yd.double().cpu().numpy()
    assert np.isnan(Y[:, k:]).all()
    u = 2.0**-53 if dtype == torch.float64 else 2.0**-24
    L = np.diff(A.rowptr).astype(np.float64)[:, None]
    # any order of the sums, one rounding per step (the oracle's own error is far below)
    assert np.all(np.abs(Y[:, :k] - Yref) <= (L + 1) * u / (1 - (L + 1) * u) * S + 1e-45)
    Y2 = torch.empty_like(Yd)
    M.spmm(Xd[:, :k], Y2[:, :k], ktile=ktile)
    assert torch.equal(Yd[:, :k], Y2[:, :k])
