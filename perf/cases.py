"""Workloads of the library, through the calls a program makes.

Each case is one pass of something a user of the library does again and again
on a matrix that is already on the GPU: a product in the form the tuner picked
for the matrix, a product with many right-hand sides, a batch of small
products, a solve, a conversion, a choice of format. The matrices are the
synthetic families the library's benchmark and tests are built on (stencils,
block-FEM, R-MAT graphs, uniform and banded rows), generated on the GPU from a
seed.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

import paper_1801_01134_gb300 as _pkg
from paper_1801_01134_gb300 import spc5

DEV = "cuda"
_DT = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
_SIZE = {"f64": 8, "f32": 4, "bf16": 2}
_MODEL = os.path.join(os.path.dirname(os.path.abspath(_pkg.__file__)), "models", "selector_gb300.npz")


# ------------------------------------------------------------------- cases
def listed():
    return [
        # the first thing a user runs: a small 2D Laplacian in a fixed shape with the
        # default kernel; a solver on a small grid is bound by the cost of a call
        {"name": "spmv_laplacian_f64", "op": "spmv", "family": "stencil2d", "nx": 128, "ny": 128, "dtype": "f64",
         "r": 2, "c": 4},
        # structured 3D grid, single precision: equal rows, runs of three
        {"name": "spmv_stencil_f32", "op": "spmv", "family": "stencil3d", "nx": 128, "ny": 128, "nz": 128,
         "points": 27, "dtype": "f32", "r": 0, "c": 0},
        # large finite-element matrix, the paper's double precision
        {"name": "spmv_fem_f64", "op": "spmv", "family": "fem", "nb": 1000000, "bs": 3, "bmin": 9, "bmax": 27,
         "band": 0.05, "dtype": "f64", "r": 0, "c": 0},
        # finite elements at an odd size with bfloat16 values (an inner matrix of a mixed-precision solver)
        {"name": "spmv_fem_bf16", "op": "spmv", "family": "fem", "nb": 333331, "bs": 3, "bmin": 5, "bmax": 21,
         "band": 0.01, "dtype": "bf16", "r": 0, "c": 0},
        # power-law graph in double precision: hub rows, random columns
        {"name": "spmv_rmat_f64", "op": "spmv", "family": "rmat", "scale": 22, "edges": 16, "dtype": "f64",
         "r": 0, "c": 0},
        # circuit-like matrix: short rows, scattered columns, a prime number of rows
        {"name": "spmv_uniform_f32", "op": "spmv", "family": "uniform", "n": 999983, "per_row": 8, "dtype": "f32",
         "r": 0, "c": 0},
        # block solver or smoothing of many vectors on a grid
        {"name": "spmm_stencil_f32_k32", "op": "spmm", "family": "stencil3d", "nx": 128, "ny": 128, "nz": 128,
         "points": 27, "dtype": "f32", "k": 32},
        # feature propagation over a graph
        {"name": "spmm_rmat_f32_k8", "op": "spmm", "family": "rmat", "scale": 22, "edges": 16, "dtype": "f32", "k": 8},
        # many uneven small systems stepped together
        {"name": "batch_f32", "op": "batch", "count": 256, "dtype": "f32"},
        # a whole solve: mixed-precision CG with reliable updates on a 3D grid
        {"name": "cg_reliable", "op": "cg", "nx": 96, "ny": 96, "nz": 96, "inner": "f32", "reliable": True},
        # a new matrix enters: CSR to the form that suits grids
        {"name": "convert_stencil_f64", "op": "convert", "family": "stencil3d", "nx": 128, "ny": 128, "nz": 128,
         "points": 27, "dtype": "f64", "r": 4, "c": 8},
        # a new matrix enters: the learned selector names its shape
        {"name": "select_rmat", "op": "select", "family": "rmat", "scale": 20, "edges": 16, "dtype": "f32"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


_RANDOM = ("fem", "rmat", "uniform", "banded")


def _draw_matrix(rng, most=1.0, families=("stencil2d", "stencil3d") + _RANDOM):
    """A family and a size; `most` scales the largest size down."""
    f = rng.choice(families)
    if f == "stencil2d":
        n = _log(rng, 1e4, 1.5e6 * most)
        nx = max(2, int(math.sqrt(n) * rng.uniform(0.5, 2.0)))
        return {"family": f, "nx": nx, "ny": max(2, n // nx)}
    if f == "stencil3d":
        s = _log(rng, 1e4, 2e6 * most) ** (1 / 3)
        return {"family": f, "nx": max(2, int(s * rng.uniform(0.8, 1.25))), "ny": max(2, int(s)), "nz": max(2, int(s * 0.8)),
                "points": rng.choice((7, 27))}
    if f == "fem":
        bs = rng.choice((2, 3, 4, 6))
        bmin = rng.randint(3, 9)
        return {"family": f, "nb": max(64, int(_log(rng, 1e4, 1.5e6 * most) / bs)), "bs": bs, "bmin": bmin,
                "bmax": bmin + rng.randint(1, 12), "band": round(10 ** rng.uniform(-3, -1), 5)}
    if f == "rmat":
        return {"family": f, "scale": rng.randint(14, 22 if most >= 1 else 20), "edges": rng.randint(4, 16)}
    if f == "uniform":
        return {"family": f, "n": _log(rng, 1e4, 1.5e6 * most), "per_row": rng.randint(2, 30)}
    return {"family": f, "n": _log(rng, 1e4, 1.5e6 * most), "half_bw": rng.randint(2, 48), "density": round(rng.uniform(0.1, 0.95), 3)}


def draw(rng):
    op = rng.choice(("spmv",) * 5 + ("spmm",) * 2 + ("batch", "cg", "convert", "select"))
    if op == "spmv":
        # the tuner's choice three times of four, otherwise a shape the caller fixed with the default kernel
        r, c = (0, 0) if rng.random() < 0.75 else (rng.choice((1, 2, 4, 8)), rng.choice((4, 8, 16)))
        return {"op": op, **_draw_matrix(rng), "dtype": rng.choice(("f64", "f32", "bf16")), "r": r, "c": c}
    if op == "spmm":
        return {"op": op, **_draw_matrix(rng, 0.5), "dtype": rng.choice(("f32", "f32", "bf16", "f64")),
                "k": rng.choice((2, 4, 5, 8, 13, 16, 24, 32))}
    if op == "batch":
        return {"op": op, "count": _log(rng, 8, 256), "dtype": rng.choice(("f32", "f64"))}
    if op == "cg":
        s = _log(rng, 2e4, 8e5) ** (1 / 3)
        return {"op": op, "nx": int(s * rng.uniform(0.8, 1.2)), "ny": int(s), "nz": int(s * 0.9),
                **rng.choice(({"inner": "", "reliable": False}, {"inner": "f32", "reliable": True},
                              {"inner": "f32", "reliable": False}))}
    if op == "convert":
        return {"op": op, **_draw_matrix(rng), "dtype": rng.choice(("f64", "f32", "bf16")),
                "r": rng.choice((1, 1, 2, 4, 8)), "c": rng.choice((4, 8, 16))}
    # a grid's structure is its size; the others' has to be looked at
    return {"op": op, **_draw_matrix(rng, families=_RANDOM), "dtype": "f32"}


# ---------------------------------------------------------------- matrices
class _Csr:
    """CSR structure. The column indices lie at the start of a longer buffer, as they do where a
    program carves its arrays from a pool that it keeps."""

    SLACK = 4096

    def __init__(self, n, m, rowptr, colidx=None):
        self.n, self.m, self.rowptr = n, m, rowptr
        if colidx is not None:
            self.set_columns(colidx)

    def set_columns(self, colidx):
        room = torch.zeros(colidx.numel() + self.SLACK, dtype=torch.int32, device=DEV)
        self.colidx = room[: colidx.numel()].copy_(colidx)

    def rows(self):
        return torch.repeat_interleave(torch.arange(self.n, device=DEV), self.rowptr[1:] - self.rowptr[:-1])


def _ptr(counts):
    p = torch.zeros(counts.numel() + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(counts, 0, out=p[1:])
    return p


def _from_mask(cols, ok, m):
    """Rows of sorted candidate columns and which of them are there."""
    return _Csr(cols.shape[0], m, _ptr(ok.sum(1)), cols[ok])


def _stencil(nx, ny, nz, points):
    n = nx * ny * nz
    i = torch.arange(n, device=DEV, dtype=torch.int32)
    x, y, z = i % nx, (i // nx) % ny, i // (nx * ny)
    cols, ok = [], []
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                if abs(dx) + abs(dy) + abs(dz) > (1 if points in (5, 7) else 3) or (points == 5 and dz):
                    continue
                cols.append(i + (dx + nx * (dy + ny * dz)))
                ok.append((x + dx >= 0) & (x + dx < nx) & (y + dy >= 0) & (y + dy < ny) & (z + dz >= 0) & (z + dz < nz))
    return _from_mask(torch.stack(cols, 1), torch.stack(ok, 1), n)


def _distinct(cols):
    """Sorted rows and a mask that leaves out repeated columns."""
    cols = cols.sort(1).values
    ok = torch.ones_like(cols, dtype=torch.bool)
    ok[:, 1:] = cols[:, 1:] != cols[:, :-1]
    return cols, ok


def _fem(nb, bs, bmin, bmax, band, g):
    """Dense bs x bs blocks: per block row the diagonal and bmin..bmax - 1 others within the band."""
    w = max(bmax, int(band * nb))
    i = torch.arange(nb, device=DEV, dtype=torch.int32).unsqueeze(1)
    cols = i + torch.randint(-w, w + 1, (nb, bmax), generator=g, device=DEV, dtype=torch.int32)
    cols[:, 0] = i[:, 0]
    cols = torch.where(cols < 0, -cols, cols)
    cols = torch.where(cols >= nb, 2 * (nb - 1) - cols, cols).clamp_(0, nb - 1)
    count = torch.randint(bmin, bmax + 1, (nb, 1), generator=g, device=DEV, dtype=torch.int32)
    cols = torch.where(torch.arange(bmax, device=DEV).unsqueeze(0) < count, cols, i)  # the rest repeat the diagonal
    cols, ok = _distinct(cols)
    per = ok.sum(1)
    start, bc = _ptr(per), cols[ok]
    rowptr = _ptr(torch.repeat_interleave(per * bs, bs))
    n = nb * bs
    A = _Csr(n, n, rowptr)
    row = A.rows()
    pos = torch.arange(row.numel(), device=DEV) - rowptr[row]
    A.set_columns(bc[start[row // bs] + pos // bs] * bs + (pos % bs))
    return A


def _rmat(scale, edges, g):
    n, e = 1 << scale, edges << scale
    src = torch.zeros(e, dtype=torch.int64, device=DEV)
    dst = torch.zeros_like(src)
    for _ in range(scale):
        u = torch.rand(e, generator=g, device=DEV)
        src = 2 * src + (u >= 0.76)
        dst = 2 * dst + (((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
    p = torch.randperm(n, generator=g, device=DEV)
    key = torch.unique(p[src] * n + p[dst])
    return _Csr(n, n, _ptr(torch.bincount(key // n, minlength=n)), key % n)


def _matrix(c, g):
    f = c["family"]
    if f == "stencil2d":
        return _stencil(c["nx"], c["ny"], 1, 5)
    if f == "stencil3d":
        return _stencil(c["nx"], c["ny"], c["nz"], c["points"])
    if f == "fem":
        return _fem(c["nb"], c["bs"], c["bmin"], c["bmax"], c["band"], g)
    if f == "rmat":
        return _rmat(c["scale"], c["edges"], g)
    n = c["n"]
    if f == "uniform":
        return _from_mask(*_distinct(torch.randint(0, n, (n, c["per_row"]), generator=g, device=DEV, dtype=torch.int32)), n)
    w = c["half_bw"]
    cols = torch.arange(n, device=DEV, dtype=torch.int32).unsqueeze(1) + torch.arange(-w, w + 1, device=DEV, dtype=torch.int32)
    ok = torch.rand(n, 2 * w + 1, generator=g, device=DEV) < c["density"]
    ok[:, w] = True
    return _from_mask(cols, ok & (cols >= 0) & (cols < n), n)


def _batch_matrices(count, g):
    """Uneven small matrices: n lognormal in [1k, 64k], 3 to 60 per row; stencils, bands and random rows."""
    sizes = np.random.RandomState(count)  # the systems' sizes belong to the case, their patterns to the seed
    u, z = sizes.rand(count, 2), sizes.randn(count)
    for q in range(count):
        n = int(min(65536, max(1024, round(8192.0 * math.exp(float(z[q]))))))
        per, kind = 3 + int(u[q, 0] * 58), int(u[q, 1] * 4)
        if kind == 0:
            if per < 8:
                side = int(math.sqrt(n))
                yield _matrix({"family": "stencil2d", "nx": side, "ny": n // side}, g)
            else:
                s = max(2, round(n ** (1 / 3)))
                yield _matrix({"family": "stencil3d", "nx": s, "ny": s, "nz": s, "points": 27 if per > 16 else 7}, g)
        elif kind == 1:
            w = max(1, per // 2)
            yield _matrix({"family": "banded", "n": n, "half_bw": w, "density": min(0.95, per / (2.0 * w + 1))}, g)
        else:
            yield _matrix({"family": "uniform", "n": n, "per_row": per}, g)


def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _values(A, dtype, g):
    return torch.randn(A.colidx.numel(), generator=g, device=DEV, dtype=torch.float32).to(_DT[dtype])


def _vector(shape, dtype, g):
    t = torch.float64 if dtype == "f64" else torch.float32
    return torch.rand(shape, generator=g, device=DEV, dtype=t) * 2 - 1


def _poisson(c, g):
    """7-point Poisson matrix, its diagonal raised by a uniform [0, 1) per row, and a right-hand side."""
    A = _stencil(c["nx"], c["ny"], c["nz"], 7)
    row = A.rows()
    shift = torch.rand(A.n, generator=g, device=DEV, dtype=torch.float64)
    val = torch.where(A.colidx == row, 6.0 + shift[row], torch.tensor(-1.0, dtype=torch.float64, device=DEV))
    return A, val, _vector(A.n, "f64", g)


# ------------------------------------------------------------------ passes
class _View:
    """A device array of a handle, which it keeps alive."""

    def __init__(self, M, ptr, count, typestr):
        self.M = M
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": (count,), "typestr": typestr, "version": 3}


def _csr(A, val):
    return spc5.DeviceCSR(A.n, A.m, A.rowptr, A.colidx, val)


def _tuned(A, val):
    """The matrix in the shape and kernel that the library's tuner picks for it."""
    t = spc5.tune(_csr(A, val))
    return spc5.convert(A.rowptr, A.colidx, val, A.n, A.m, t["r"], t["c"], variant=t["variant"])


def prepare(case, seed):
    g, op = _generator(seed), case["op"]
    if op == "cg":
        A, val, b = _poisson(case, g)
        # the shape the selector names for 7-point grids, both precisions alike
        M = spc5.convert(A.rowptr, A.colidx, val, A.n, A.m, 1, 4)
        L = spc5.convert(A.rowptr, A.colidx, val.to(_DT[case["inner"]]), A.n, A.m, 1, 4) if case["inner"] else None
        return {"op": op, "M": M, "L": L, "b": b, "x": torch.empty_like(b), "reliable": case["reliable"]}
    model = None
    if op in ("batch", "select"):
        z = np.load(_MODEL)
        model = {"mlp_params": torch.from_numpy(z["mlp_params"]).to(DEV), "feat_mean": z["feat_mean"],
                 "feat_scale": z["feat_scale"]}
    if op == "batch":
        # each system in the shape the learned selector names and the kernel that is fastest on it
        mats, vecs = [], []
        for A in _batch_matrices(case["count"], g):
            val = _values(A, case["dtype"], g)
            r, c, _ = spc5.select(_csr(A, val), spc5.SELECT_MLP, **model)
            mats.append(spc5.convert(A.rowptr, A.colidx, val, A.n, A.m, r, c))
            vecs.append(_vector(A.m, case["dtype"], g))
            mats[-1].autotune(vecs[-1], torch.empty(A.n, dtype=vecs[-1].dtype, device=DEV), reps=3)
        y = torch.empty(sum(M.n for M in mats), dtype=vecs[0].dtype, device=DEV)
        B = spc5.Batch(mats, vecs, list(y.split([M.n for M in mats])))
        return {"op": op, "B": B, "y": y}
    # a conversion's outputs have the structure's sizes, so that belongs to the case: the seed gives the values
    A = _matrix(case, _generator(1) if op == "convert" else g)
    val = _values(A, case["dtype"], g)
    if op == "select":
        return {"op": op, "d": _csr(A, val), "model": model}
    if op == "convert":
        return {"op": op, "A": A, "val": val, "r": case["r"], "c": case["c"]}
    if op == "spmm":
        t = spc5.tune(_csr(A, val), k_spmm=case["k"], reps=3)
        M = spc5.convert(A.rowptr, A.colidx, val, A.n, A.m, t["spmm_r"], t["spmm_c"], variant=t["spmm_variant"])
        X = _vector((A.m, case["k"]), case["dtype"], g)
        return {"op": op, "M": M, "X": X, "Y": torch.empty((A.n, case["k"]), dtype=X.dtype, device=DEV), "tile": t["ktile"]}
    if case["r"]:
        M = spc5.convert(A.rowptr, A.colidx, val, A.n, A.m, case["r"], case["c"])
    else:
        M = _tuned(A, val)
    x = _vector(A.m, case["dtype"], g)
    return {"op": op, "M": M, "x": x, "y": torch.empty(A.n, dtype=x.dtype, device=DEV)}


def run(s):
    op = s["op"]
    if op == "spmv":
        return s["M"].spmv(s["x"], s["y"])
    if op == "spmm":
        return s["M"].spmm(s["X"], s["Y"], ktile=s["tile"])
    if op == "batch":
        s["B"].run()
        return s["y"]
    if op == "cg":
        x, _ = spc5.cg(s["M"], s["b"], A_inner=s["L"], x=s["x"], tol=1e-11, reliable=s["reliable"])
        return x
    if op == "convert":
        A = s["A"]
        M = spc5.convert(A.rowptr, A.colidx, s["val"], A.n, A.m, s["r"], s["c"])
        a = M.arrays()
        vals = _View(M, a.values_d, a.nnz, {spc5.SPC5_F64: "<f8", spc5.SPC5_F32: "<f4", spc5.SPC5_BF16: "<i2"}[a.dtype])
        views = (_View(M, a.block_rowptr_d, a.nintervals + 1, "<i4"), _View(M, a.block_colidx_d, a.nblocks, "<i4"),
                 _View(M, a.block_masks_d, a.nblocks * a.mask_bytes, "|u1"), vals,
                 _View(M, a.valptr_d, a.nintervals + 1, "<i8"))
        return [torch.as_tensor(v, device=DEV) for v in views]
    r, c, scores = spc5.select(s["d"], spc5.SELECT_MLP, **s["model"])
    return [r, c, scores]


# ----------------------------------------------------------- what is needed
def _shape_of(c):
    """(rows, entries, runs of adjacent columns) of a case's matrix, without building it."""
    f = c["family"]
    if f in ("stencil2d", "stencil3d"):
        nx, ny, nz = c["nx"], c["ny"], c.get("nz", 1)
        n = nx * ny * nz
        if f == "stencil3d" and c["points"] == 27:
            return n, (3 * nx - 2) * (3 * ny - 2) * (3 * nz - 2), nx * (3 * ny - 2) * (3 * nz - 2)
        nnz = n + 2 * ((nx - 1) * ny * nz + nx * (ny - 1) * nz + nx * ny * (nz - 1))
        return n, nnz, nnz - 2 * (nx - 1) * ny * nz
    if f == "fem":
        blocks = c["nb"] * 0.5 * (c["bmin"] + c["bmax"])
        return c["nb"] * c["bs"], blocks * c["bs"] ** 2, blocks * c["bs"]
    if f == "rmat":
        nnz = 0.96 * (c["edges"] << c["scale"])
        return 1 << c["scale"], nnz, nnz
    if f == "uniform":
        return c["n"], c["n"] * c["per_row"], c["n"] * c["per_row"]
    nnz = c["n"] * (1 + 2 * c["half_bw"] * c["density"])
    return c["n"], nnz, max(c["n"], nnz * (1 - c["density"]))


def work(case):
    """Values once, a column and a mask byte for each run of adjacent entries, vectors once, a row pointer."""
    op = case["op"]
    if op == "batch":
        n, nnz, runs = 12000.0 * case["count"], 31.5 * 12000.0 * case["count"], 20.0 * 12000.0 * case["count"]
        s = _SIZE[case["dtype"]]
        return {"bytes": nnz * s + runs * 5 + n * (2 * s + 12), "flops": 2 * nnz}
    if op == "cg":
        # about 60 iterations, each with one product and the passes over x, r, p and q
        n = case["nx"] * case["ny"] * case["nz"]
        s = _SIZE[case["inner"] or "f64"]
        return {"bytes": 60 * (7 * n * s + 5 * 5 * n + 12 * n + 9 * n * s), "flops": 60 * (14 * n + 12 * n)}
    n, nnz, runs = _shape_of(case)
    s = _SIZE[case["dtype"]]
    sx = max(4, s)
    if op == "select":
        return {"bytes": 4 * nnz + 8 * (n + 1), "flops": 12 * nnz}
    if op == "convert":
        return {"bytes": nnz * (4 + 2 * s) + 5 * runs + 20 * n, "flops": 0}
    k = case.get("k", 1)
    return {"bytes": nnz * s + runs * 5 + 12 * n + 2 * k * n * sx, "flops": 2.0 * k * nnz}


# --------------------------------------------------------------- reference
def _product(A, val, x):
    """A x in 64 bits: products gathered, then added row by row."""
    return torch.zeros(A.n, dtype=torch.float64, device=DEV).index_add_(0, A.rows(), val.double() * x.double()[A.colidx])


def exact(case, seed):
    g, op = _generator(seed), case["op"]
    if op == "cg":
        A, val, b = _poisson(case, g)
        row = A.rows()

        def mul(p):
            return torch.zeros_like(p).index_add_(0, row, val * p[A.colidx])

        # plain conjugate gradients, carried on past what 64 bits resolve
        x, r = torch.zeros_like(b), b.clone()
        p, rho = r.clone(), r @ r
        for _ in range(400):
            if float(rho) <= 1e-30 * float(b @ b):
                break
            q = mul(p)
            alpha = rho / (p @ q)
            x, r = x + alpha * p, r - alpha * q
            new = r @ r
            p, rho = r + (new / rho) * p, new
        return x
    if op in ("convert", "select"):
        return None
    if op == "batch":
        ys = []
        for A in _batch_matrices(case["count"], g):
            val = _values(A, case["dtype"], g)
            ys.append(_product(A, val, _vector(A.m, case["dtype"], g)))
        return torch.cat(ys)
    A = _matrix(case, g)
    val = _values(A, case["dtype"], g)
    if op == "spmv":
        return _product(A, val, _vector(A.m, case["dtype"], g))
    X = _vector((A.m, case["k"]), case["dtype"], g)
    return torch.stack([_product(A, val, X[:, j]) for j in range(case["k"])], 1)
