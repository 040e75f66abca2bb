"""The forms of the kernels for many blocks, and for mostly zero ones, at the numbers of blocks where
each begins, against plain FP64 (NumPy) or the oracle."""
import numpy as np
import pytest

from oracle import clr_oracle as co
from paper_1509_00309_gb300 import workloads as wl
from tests import clr_pack
from tests.test_gpu_product import _check_product

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def ctx():
    from paper_1509_00309_gb300 import build, clr
    build.build()
    return clr.Context(0, precision="fp64", eps_lr=1e-8)


# 676 tiles: each CTA takes its own (all with low-rank work, sums concatenated and accumulated
# densely), or clusters do (few with work)
@pytest.mark.parametrize("p_zero,p_dense,max_rank", [(0.1, 0.2, None), (0.7, 0.02, 2), (0.94, 0.02, 2)])
def test_low_rank_products_of_many_tiles(ctx, p_zero, p_dense, max_rank):
    sizes = [16, 1, 7, 33, 2, 20, 9, 3, 40, 12, 5, 8, 25] * 2
    rng = np.random.default_rng(int(100 * p_zero))
    a, b = (co.from_blocks(sizes, sizes, wl.random_blocks_spec(
        rng, sizes, sizes, p_zero=p_zero, p_dense=p_dense, max_rank=max_rank)) for _ in range(2))
    gc = ctx.multiply(clr_pack.to_library(ctx, a), clr_pack.to_library(ctx, b))
    _check_product(ctx, a, b, 1e-8, gc)


# 529 and 484 dense tiles: a CTA a tile, or clusters; 1 x 1 tiles among them
@pytest.mark.parametrize("nb", [22, 23])
def test_norms_of_many_dense_tiles(ctx, nb):
    sizes = ([40, 1, 17, 9, 64] * 5)[:nb]
    n = sum(sizes)
    rng = np.random.default_rng(nb)
    a, b = rng.standard_normal((n, n)), rng.standard_normal((n, n))
    norms = ctx.multiply(ctx.from_dense(a, sizes), ctx.from_dense(b, sizes)).get_blocks(pool=False)[2]
    off = np.concatenate([[0], np.cumsum(sizes)])
    ab, mag = a @ b, np.abs(a) @ np.abs(b)
    for i in range(nb):
        for j in range(nb):
            box = (slice(off[i], off[i + 1]), slice(off[j], off[j + 1]))
            # n products and additions an entry on either side, m n <= 4096 squares
            bound = 2.0 * (n + 4096) * U * np.linalg.norm(mag[box])
            assert abs(norms[i, j] - np.linalg.norm(ab[box])) <= bound, (i, j)


# clusters of eight up to 1024 blocks, four up to 3072, two, one beyond 16384 (a scaled copy: beyond
# 3072)
@pytest.mark.parametrize("nb,p_zero", [(32, 0.3), (33, 0.3), (56, 0.5), (129, 0.97)])
def test_linear_combination_of_many_blocks(ctx, nb, p_zero):
    sizes = ([3, 1, 20, 9, 12, 2, 33] * 19)[:nb]
    rng = np.random.default_rng(nb)
    x, y = (co.from_blocks(sizes, sizes, wl.random_blocks_spec(rng, sizes, sizes, p_zero=p_zero,
                                                               p_dense=0.5 * (1 - p_zero)))
            for _ in range(2))
    gx, gy = clr_pack.to_library(ctx, x), clr_pack.to_library(ctx, y)
    n, dx, dy = sum(sizes), x.to_dense(), y.to_dense()
    off = x.row_off
    for a, b, diag in ((-1.25, 0.375, 1.875), (0.75, 0.0, 0.0), (0.0, 0.5, 0.0)):
        out = ctx.lincomb(a, gx, b, gy, diag)
        got, want = out.to_dense(), a * dx + b * dy + diag * np.eye(n)
        norms = out.get_blocks(pool=False)[2]
        # truncation at 1e-8 a block (none in a copy); 33 squares and products of entries of order 10
        eps = 1e-8 if a != 0.0 and b != 0.0 else 0.0
        for i in range(nb):
            for j in range(nb):
                box = (slice(off[i], off[i + 1]), slice(off[j], off[j + 1]))
                w = np.linalg.norm(want[box])
                tol = eps * (1 + 1e-6) + 1e-11
                assert np.linalg.norm(got[box] - want[box]) <= tol, (a, i, j)
                assert abs(norms[i, j] - w) <= tol, (a, i, j)


# two CTAs a block-row from 229 on; more blocks in a row than 32 a CTA looks at at once (64 and 256)
@pytest.mark.parametrize("nr,nc,p_zero", [(229, 70, 0.9), (229, 5, 0.2), (3, 300, 0.97), (2, 513, 0.5)])
def test_matvec_of_many_blocks(ctx, nr, nc, p_zero):
    import torch
    rng = np.random.default_rng(nr + nc)
    rows, cols = ([3, 40, 1, 17, 70] * 46)[:nr], ([5, 1, 33, 9] * 129)[:nc]
    a = co.from_blocks(rows, cols, wl.random_blocks_spec(rng, rows, cols, p_zero=p_zero,
                                                         p_dense=0.5 * (1 - p_zero)))
    da = a.to_dense()
    mag = np.zeros(da.shape)
    for (i, j), b in a.blocks.items():
        mag[a.row_off[i]:a.row_off[i + 1], a.col_off[j]:a.col_off[j + 1]] = (
            np.abs(b.d) if b.kind == co.KIND_DENSE else np.abs(b.x) @ np.abs(b.w).T)
    x = rng.standard_normal(sum(cols))
    y = torch.empty(sum(rows), dtype=torch.float64, device="cuda")
    ctx.matvec(clr_pack.to_library(ctx, a), torch.from_numpy(x).cuda(), y)
    # ranks of at most 35, n terms, on either side
    bound = 2.0 * (sum(cols) + 35) * U * (mag @ np.abs(x))
    assert (np.abs(y.cpu().numpy() - da @ x) <= bound).all()


# one part a block and more blocks than CTAs; two, four and eight parts; mostly zero
@pytest.mark.parametrize("sizes,p_zero", [
    ([1, 20, 7] * 34, 0.3), ([70, 61, 66] * 11, 0.3), ([100, 93, 130] * 11, 0.6), ([256, 40] * 3, 0.1),
    ([1, 20, 7] * 110, 0.999),
])
def test_transposes_of_many_blocks(ctx, sizes, p_zero):
    rng = np.random.default_rng(len(sizes))
    a = co.from_blocks(sizes, sizes, wl.random_blocks_spec(rng, sizes, sizes, p_zero=p_zero,
                                                           p_dense=0.5 * (1 - p_zero)))
    ga = clr_pack.to_library(ctx, a)
    gt = ctx.transpose(ga)
    assert np.array_equal(gt.to_dense(), ga.to_dense().T)
    for x, y in zip(ga.get_blocks(pool=False)[:3], gt.get_blocks(pool=False)[:3]):
        assert np.array_equal(x.T, y)


# 64 x 64 tiles from 4097 tiles on, 32 x 32 below; warps whose columns lie in one block and in
# several, all zero, and ragged edges
@pytest.mark.parametrize("big,sizes", [
    (False, [256, 1, 100, 7, 33]), (True, [256, 200, 31, 1, 180, 64, 3] * 6 + [97]),
    (True, [5, 1, 3, 17, 8, 2, 33, 9] * 53 + [63]),
])
def test_reconstruction_by_either_tile(ctx, big, sizes):
    n = sum(sizes)
    assert (((n + 63) // 64) ** 2 > 4096) == big
    rng = np.random.default_rng(n)
    many = len(sizes) > 100
    a = co.from_blocks(sizes, sizes, wl.random_blocks_spec(
        rng, sizes, sizes, p_zero=0.6 if many else 0.2, p_dense=0.2))
    got = clr_pack.to_library(ctx, a).to_dense()
    zero = np.ones((n, n), bool)
    for (i, j), b in a.blocks.items():
        box = (slice(a.row_off[i], a.row_off[i + 1]), slice(a.col_off[j], a.col_off[j + 1]))
        zero[box] = False
        if b.kind == co.KIND_DENSE:
            assert np.array_equal(got[box], b.d)
        else:
            # ranks of at most 128
            assert (np.abs(got[box] - b.x @ b.w.T)
                    <= 2.0 * 130 * U * (np.abs(b.x) @ np.abs(b.w).T)).all()
    assert (got[zero] == 0.0).all()
