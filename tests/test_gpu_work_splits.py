"""The ways the kernels share out their work -- sub-tile edges, clusters of CTAs per tile,
teams, register and shared-memory forms -- at the sizes where each begins, ends or leaves a
remainder, against plain FP64 (NumPy) or the oracle."""
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


def _abs_dense(c):
    """sum over the blocks of |D| or |X| |W|^T: what bounds the rounding of reconstructions."""
    out = np.zeros(c.shape)
    for (i, j), b in c.blocks.items():
        v = np.abs(b.d) if b.kind == co.KIND_DENSE else np.abs(b.x) @ np.abs(b.w).T
        out[c.row_off[i]:c.row_off[i + 1], c.col_off[j]:c.col_off[j + 1]] = v
    return out


# the FP64 tile products' sub-tile edge is the largest of 64, 32, 16 that gives every SM six
# sub-tiles; with more than 1024 tiles it is 64
@pytest.mark.parametrize("sizes", [
    [1, 15, 16, 17],                       # 16, the smallest
    [256, 255, 33],                        # 16, the largest clusters
    [200] * 6 + [31],                      # 32: 49 tiles, 1849 sub-tiles
    [250] * 7 + [255, 65, 63],             # 64: 100 tiles, 1156 sub-tiles
    [1, 63, 64, 65, 16, 48, 47] * 4 + [33] * 5,   # 64, numbered without a prefix sum
])
def test_fp64_dense_tiles_at_every_sub_tile_edge(ctx, sizes):
    n = sum(sizes)
    rng = np.random.default_rng(n)
    a, b = rng.standard_normal((n, n)), rng.standard_normal((n, n))
    got = ctx.multiply(ctx.from_dense(a, sizes), ctx.from_dense(b, sizes)).to_dense()
    # n products and additions on either side
    assert (np.abs(got - a @ b) <= 2.0 * (n + 1) * U * (np.abs(a) @ np.abs(b))).all()


# clusters of eight CTAs a tile up to 64 tiles, of four beyond; rows fewer than the CTAs; ranks that
# fill the concatenation (QR) and that exceed it (dense accumulation)
@pytest.mark.parametrize("nb,max_rank", [(3, None), (8, 5), (9, 5), (9, None)])
def test_low_rank_products_by_clusters(ctx, nb, max_rank):
    sizes = [256, 1, 7, 65, 2, 30, 129, 3, 40][:nb]
    rng = np.random.default_rng(100 * nb + (max_rank or 0))
    a, b = (co.from_blocks(sizes, sizes, wl.random_blocks_spec(
        rng, sizes, sizes, p_zero=0.1, p_dense=0.2, max_rank=max_rank)) for _ in range(2))
    gc = ctx.multiply(clr_pack.to_library(ctx, a), clr_pack.to_library(ctx, b))
    _check_product(ctx, a, b, 1e-8, gc)


# block-rows of one to eight row groups and fewer blocks than CTAs; 9, 1089 and 4225 blocks take
# eight, four and one CTA in the transposition
@pytest.mark.parametrize("rows,cols", [
    ([256, 1, 33], [200, 31, 64]),
    ([1, 2, 31, 32, 33, 5, 97, 161, 7, 225], [256] + [3, 40] * 10),
    ([9, 1, 4] * 11, [2, 17, 33] * 11),
    ([3, 1, 6, 2, 8] * 13, [2, 5, 1, 4, 7] * 13),
])
def test_matvec_transpose_and_reconstruction(ctx, rows, cols):
    import torch
    rng = np.random.default_rng(len(rows) + len(cols))
    a = co.from_blocks(rows, cols, wl.random_blocks_spec(rng, rows, cols))
    ga = clr_pack.to_library(ctx, a)
    da, aa = a.to_dense(), _abs_dense(a)
    n = sum(cols)
    got = ga.to_dense()
    assert (np.abs(got - da) <= 2.0 * 130 * U * aa).all()   # ranks of at most 128
    for (i, j), b in a.blocks.items():
        if b.kind == co.KIND_DENSE:
            assert np.array_equal(got[a.row_off[i]:a.row_off[i + 1],
                                      a.col_off[j]:a.col_off[j + 1]], b.d)
    assert np.array_equal(ctx.transpose(ga).to_dense(), got.T)
    x = rng.standard_normal(n)
    y = torch.empty(sum(rows), dtype=torch.float64, device="cuda")
    ctx.matvec(ga, torch.from_numpy(x).cuda(), y)
    # W^T x, X t and the blocks' sums on the one side; the reconstruction and n terms on the other
    bound = 2.0 * (n + 130) * U * (aa @ np.abs(x))
    assert (np.abs(y.cpu().numpy() - da @ x) <= bound).all()


def _graded(rng, m, n, r, common):
    """An m x n block of rank r whose column space lies in `common` (m x >= r)."""
    x = common[:, :r] @ rng.standard_normal((r, r))
    return x * np.logspace(0, -3, r), rng.standard_normal((n, r))


# sums of two low-rank blocks by QR of the factors: at most 76 tiles take a pair of CTAs each, more
# one; R up to 32 or 64 columns and up to 128, 192 or 256 rows stay in registers
@pytest.mark.parametrize("sizes,r_top", [
    ([256, 193], 64), ([256, 192, 129, 128, 17, 4], 30), ([256, 130, 200], 20),
    ([256, 64, 192, 129, 128, 40, 33, 8, 4], 32),
])
def test_low_rank_sums_by_pairs_and_single_ctas(ctx, sizes, r_top):
    rng = np.random.default_rng(sum(sizes) + r_top)
    specs = [[], []]
    for m in sizes:
        rows = [[], []]
        for n in sizes:
            r = max(1, min(r_top, min(m, n) // 4))
            common = np.linalg.qr(rng.standard_normal((m, r)))[0]
            for row in rows:
                row.append((2, _graded(rng, m, n, r, common)))
        for s, row in zip(specs, rows):
            s.append(row)
    x, y = (co.from_blocks(sizes, sizes, s) for s in specs)
    eps = 1e-8
    g = clr_pack.from_library(ctx.lincomb(0.75, clr_pack.to_library(ctx, x), -1.5,
                                          clr_pack.to_library(ctx, y)))
    want = co.lincomb(0.75, x, -1.5, y, 0.0, eps)
    exact, mag = 0.75 * x.to_dense() - 1.5 * y.to_dense(), _abs_dense(x) + _abs_dense(y)
    assert np.array_equal(g.kinds(), want.kinds())
    assert np.abs(g.ranks().astype(int) - want.ranks().astype(int)).max() <= 1
    for i in range(len(sizes)):
        for j in range(len(sizes)):
            box = (slice(x.row_off[i], x.row_off[i + 1]), slice(x.row_off[j], x.row_off[j + 1]))
            d = np.linalg.norm(g.block_dense(i, j) - exact[box])
            assert d <= eps * (1 + 1e-6) + 1e-13 * mag[box].sum(), (i, j, d)


def test_linear_combination_of_largest_blocks(ctx):
    sizes = [256, 1, 100]
    rng = np.random.default_rng(8)
    x, y = (co.from_blocks(sizes, sizes, wl.random_blocks_spec(rng, sizes, sizes, p_zero=0.2))
            for _ in range(2))
    out = ctx.lincomb(-1.25, clr_pack.to_library(ctx, x), 0.375, clr_pack.to_library(ctx, y),
                      1.875)
    exact = -1.25 * x.to_dense() + 0.375 * y.to_dense() + 1.875 * np.eye(sum(sizes))
    mag = 2.0 * np.linalg.norm(_abs_dense(x) + _abs_dense(y)) + 2.0 * np.sqrt(sum(sizes))
    # nine tiles truncated at eps, sums of at most 256 terms
    assert np.linalg.norm(out.to_dense() - exact) <= 3e-8 + 300 * 2 * U * mag
    norms = out.get_blocks(pool=False)[2]
    g = clr_pack.from_library(out)
    for i in range(3):
        for j in range(3):
            w = np.linalg.norm(g.block_dense(i, j))
            assert abs(norms[i, j] - w) <= 1e-8 + 1e-12 * w


# 16 blocks: teams of four CTAs a block; 169: the same kernel, a block per CTA; 324: the kernel
# without clusters
@pytest.mark.parametrize("sizes", [
    [256, 97, 16, 200], [120, 33, 64, 8, 90, 1, 48, 70, 2, 100, 25, 60, 5],
    [40, 17, 64, 5, 33, 1, 90, 12, 50] * 2,
])
def test_build_by_teams_and_single_ctas(ctx, sizes):
    n = sum(sizes)
    rng = np.random.default_rng(n)
    r = 0.02 * np.arange(n) + rng.uniform(-0.004, 0.004, n)
    a = np.exp(-(r[:, None] - r[None, :]) ** 2 / 2.0) + 1e-3 * np.eye(n)
    eps = 1e-8
    g = clr_pack.from_library(ctx.from_dense(a, sizes, eps_lr=eps))
    want = co.build(a, sizes, sizes, eps)
    gk, wk, gr, wr = g.kinds(), want.kinds(), g.ranks(), want.ranks()
    for i in range(len(sizes)):
        for j in range(len(sizes)):
            blk = a[want.row_off[i]:want.row_off[i + 1], want.col_off[j]:want.col_off[j + 1]]
            if gk[i, j] != wk[i, j]:
                # only at the threshold between dense and low rank
                assert max(gr[i, j], wr[i, j]) >= co.dense_rank_limit(sizes[i], sizes[j])
            elif gk[i, j] == co.KIND_LR:
                assert abs(int(gr[i, j]) - int(wr[i, j])) <= 1
            d = np.linalg.norm(g.block_dense(i, j) - blk)
            assert d <= (0.0 if gk[i, j] == co.KIND_DENSE
                         else eps * (1 + 1e-6) + 1e-14 * np.linalg.norm(blk)), (i, j, d)


def _slow_tail(rng, m, n, lead, decay, top):
    """U diag(s) V^T: `lead` singular values from 1 to 1e-4, then a tail from `top` falling by
    `decay` each."""
    k = min(m, n)
    u, v = (np.linalg.qr(rng.standard_normal((d, k)))[0] for d in (m, n))
    s = np.concatenate([np.logspace(0, -4, lead), top * decay ** np.arange(k - lead)])
    return (u * s) @ v.T


# a team of four CTAs and a CTA alone do the same arithmetic: QR ranks of ~235 (sweeps on a copy in
# global memory), ~190 (on the FP32 triangular factor, in global memory) and ~60 (in shared memory)
@pytest.mark.parametrize("decay", [0.999, 0.985, 0.93])
def test_teams_and_single_ctas_give_the_same_bits(ctx, decay):
    rng = np.random.default_rng(int(1000 * decay))
    big = [256, 240]
    eps = 1e-8
    a = np.zeros((496, 496))
    for i, m in enumerate(big):
        for j, n in enumerate(big):
            # the tail's norm is 0.9 eps: the rank is the leading part's
            tail = 0.9 * eps * np.sqrt(1.0 - decay ** 2)
            a[256 * i:256 * i + m, 256 * j:256 * j + n] = _slow_tail(rng, m, n, 20, decay, tail)
    team = ctx.from_dense(a, big, eps_lr=eps)
    pad = np.zeros((514, 514))
    pad[:496, :496] = a
    alone = ctx.from_dense(pad, big + [1] * 18, eps_lr=eps)   # 400 blocks: no clusters of CTAs
    kt, rt = team.get_blocks()[:2]
    ka, ra = alone.get_blocks()[:2]
    assert np.array_equal(kt, ka[:2, :2]) and np.array_equal(rt, ra[:2, :2])
    assert (np.abs(rt - 20) <= 1).all()
    assert np.array_equal(team.to_dense(), alone.to_dense()[:496, :496])
    for i, m in enumerate(big):
        for j, n in enumerate(big):
            box = (slice(256 * i, 256 * i + m), slice(256 * j, 256 * j + n))
            assert np.linalg.norm(team.to_dense()[box] - a[box]) <= eps * (1 + 1e-6) + 1e-13


def test_leading_tiles_by_teams(ctx):
    # 169 tiles whose costs differ by 1000: the largest take teams, by their size at first and by
    # their measured cost when the product is repeated into the same matrix, with the same bits
    sizes = [256, 230] + [40, 25, 33, 48, 7, 60, 22, 37, 51, 1, 44]
    n = sum(sizes)
    rng = np.random.default_rng(3)
    r = 0.02 * np.arange(n) + rng.uniform(-0.004, 0.004, n)
    a = np.exp(-(r[:, None] - r[None, :]) ** 2 / 2.0) + 1e-3 * np.eye(n)
    s = ctx.from_dense(a, sizes, eps_lr=1e-10)
    ctx.set_opts(recompress_dense=1)
    try:
        c = ctx.multiply(s, s)
        first = c.to_dense()
        for _ in range(2):
            ctx.multiply_into(s, s, c)
            assert np.array_equal(c.to_dense(), first)
    finally:
        ctx.set_opts(recompress_dense=0)
    # 169 tiles truncated at 1e-8, their operands at 1e-10
    tol = 13 * 1e-8 + 2 * 13 * 1e-10 * np.linalg.norm(a, 2) + 2 * n * U * np.linalg.norm(a) ** 2
    assert np.linalg.norm(first - a @ a) <= tol
