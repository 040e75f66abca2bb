"""Truncation at an eps near the FP64 noise floor of a block, where columns of the FP32 sweeps'
rounding exceed eps: ranks as the singular values give them."""
import numpy as np
import pytest

from oracle import clr_oracle as co
from tests import clr_pack
from tests.test_gpu_work_splits import _slow_tail

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1509_00309_gb300 import build, clr
    build.build()
    return clr.Context(0, precision="fp64", eps_lr=1e-8)


# sums of two blocks of the same column space: the core has twice the rank that its values have
@pytest.mark.parametrize("eps,spread", [(1e-13, 3), (1e-13, 8), (1e-12, 8), (1e-12, 13)])
def test_rank_of_sums_near_the_noise_floor(ctx, eps, spread):
    sizes = [256, 130, 64]
    rng = np.random.default_rng(7)
    specs = [[], []]
    for m in sizes:
        rows = [[], []]
        for n in sizes:
            r = min(24, min(m, n) // 4)
            common = np.linalg.qr(rng.standard_normal((m, r)))[0]
            for row in rows:
                x = common @ np.linalg.qr(rng.standard_normal((r, r)))[0]
                w = np.linalg.qr(rng.standard_normal((n, r)))[0]
                row.append((2, (x * np.logspace(0, -spread, r), w)))
        for spec, row in zip(specs, rows):
            spec.append(row)
    x, y = (co.from_blocks(sizes, sizes, spec) for spec in specs)
    ctx.set_opts(eps_lr=eps)
    try:
        g = clr_pack.from_library(ctx.lincomb(0.75, clr_pack.to_library(ctx, x), -1.5,
                                              clr_pack.to_library(ctx, y)))
    finally:
        ctx.set_opts(eps_lr=1e-8)
    want = co.lincomb(0.75, x, -1.5, y, 0.0, eps)
    assert np.abs(g.ranks().astype(int) - want.ranks().astype(int)).max() <= 1
    # nine tiles truncated at eps; rounding of factors of norm at most ~5
    assert (np.linalg.norm(g.to_dense() - 0.75 * x.to_dense() + 1.5 * y.to_dense())
            <= 3 * eps * (1 + 1e-6) + 3e-14)


# the SVD of whole blocks, without the pivoted QR in front: FP32 copies cached by L1 (a cluster above
# 156) or in shared memory, one pass of the orthonormalisation or two
@pytest.mark.parametrize("m,n", [(256, 240), (157, 90), (156, 130)])
@pytest.mark.parametrize("eps", [1e-13, 1e-12, 1e-11])
def test_rank_of_whole_blocks_near_the_noise_floor(ctx, eps, m, n):
    rng = np.random.default_rng(5)
    decay = 0.985
    a = _slow_tail(rng, m, n, 20, decay, 0.9 * eps * np.sqrt(1.0 - decay ** 2))
    ctx.set_opts(svd_no_prereduce=1)
    try:
        m = ctx.from_dense(a, [m], [n], eps_lr=eps)
    finally:
        ctx.set_opts(svd_no_prereduce=0)
    kinds, ranks = m.get_blocks()[:2]
    # the tail's norm is 0.9 eps, the smallest of the kept singular values 1e-4
    assert kinds[0, 0] == co.KIND_LR and abs(int(ranks[0, 0]) - 20) <= 1
    assert np.linalg.norm(m.to_dense() - a) <= eps * (1 + 1e-6) + 3e-14
