"""SpMM where the column-group kernels change over with the blocks' fill: the same bits on either side."""
import numpy as np
import pytest
import torch

from paper_1801_01134_gb300 import inputs, spc5

pytestmark = pytest.mark.gpu


def blocks(fill, r, c, seed, groups=60, per=7):
    """`per` blocks of r x c in each of `groups` block rows, block q with fill[q] values (the corner among them)."""
    rng = np.random.default_rng(seed)
    m = 4 * c * per
    rows = [[] for _ in range(groups * r - 1)]  # a last interval that is not whole
    for g in range(groups):
        for q in range(per):
            want = min(fill[(g * per + q) % len(fill)], r * c)
            cells = np.concatenate([[0], 1 + rng.permutation(r * c - 1)[: want - 1]])
            for cell in cells:
                if g * r + cell // c < len(rows):
                    rows[g * r + cell // c].append(4 * c * q + cell % c)
    rowptr = np.concatenate([[0], np.cumsum([len(x) for x in rows])]).astype(np.int64)
    cols = np.concatenate([np.sort(np.asarray(x, np.int32)) for x in rows]).astype(np.int32)
    return inputs.CSR(len(rows), m, rowptr, cols, rng.standard_normal(cols.size))


# values per block: one, just below and at two, below and at half of an 8 x 8 and an 8 x 16 block, all
FILLS = {"one": [1], "below_two": [1, 3, 1, 3, 1, 2], "two": [2], "below_half": [31, 32, 31], "half_of_64": [32, 33],
         "half_of_128": [64, 65], "all": [128]}


@pytest.mark.parametrize("fill", sorted(FILLS))
@pytest.mark.parametrize("r,c", spc5.SHAPES)
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_same_bits_as_unaligned(cuda_device, fill, r, c, dtype):
    A = blocks(FILLS[fill], r, c, seed=r * c)
    d = spc5.upload_csr(A, dtype, "cuda")
    for variant in (0, 13):  # natural and sorted order
        M = spc5.convert(d.rowptr, d.colidx, d.values, A.n, A.m, r, c, variant=variant)
        assert M.arrays().nsegments == 0
        for k, tile in ((8, 8), (12, 16), (32, 32), (36, 32)):
            X = torch.randn(A.m, k + 1, generator=torch.Generator("cuda").manual_seed(k), device="cuda")[:, :k]
            # an odd leading dimension takes the general kernel; the sums are the same
            assert torch.equal(M.spmm(X.contiguous(), ktile=tile), M.spmm(X, ktile=tile))


def test_scattered_values_are_not_slower_in_a_fixed_shape(cuda_device):
    # 7-point grid, k = 32: beta(1,4) beside beta(1,8) (unrolled 1.4 times its time, bit by bit 1.0),
    # beta(8,8) beside beta(4,8) (column by column 1.5, value by value 1.1)
    A = inputs.stencil3d(100, 100, 100, points=7)
    d = spc5.upload_csr(A, torch.float32, "cuda")
    X, Y = torch.rand(A.m, 32, device="cuda"), torch.empty(A.n, 32, device="cuda")

    def us(r, c):
        M = spc5.convert(d.rowptr, d.colidx, d.values, A.n, A.m, r, c)
        t = []
        for _ in range(7):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            M.spmm(X, Y)
            e[1].record()
            torch.cuda.synchronize()
            t.append(e[0].elapsed_time(e[1]) * 1e3)
        return min(t)

    assert us(1, 4) <= 1.2 * us(1, 8)
    assert us(8, 8) <= 1.3 * us(4, 8)
