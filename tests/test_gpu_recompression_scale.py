"""Recompression of blocks far from norm 1: the FP32 sweeps see the same numbers whatever the
scale, so a matrix and eps multiplied by the same power of two give the same kinds and ranks."""
import numpy as np
import pytest

from oracle import clr_oracle as co
from tests import clr_pack
from tests.test_gpu_work_splits import _abs_dense, _graded, _slow_tail

pytestmark = pytest.mark.gpu

# 9e-19 and 7e-46 (squares, then the entries themselves, below the FP32 range), 7e19 and 2e60
SCALES = [2.0 ** -60, 2.0 ** -150, 2.0 ** 66, 2.0 ** 200]


@pytest.fixture(scope="module")
def ctx():
    from paper_1509_00309_gb300 import build, clr
    build.build()
    return clr.Context(0, precision="fp64", eps_lr=1e-8)


# eps = 1e-8: the right factor from the kept columns; 1e-12, less than 1000 times the noise floor:
# V is accumulated.  Without the pivoted QR every block takes the SVD of all its columns, and a
# block of independent entries is certified dense after the first stage.
@pytest.mark.parametrize("prereduce", [True, False])
@pytest.mark.parametrize("eps", [1e-8, 1e-12])
def test_build_at_any_scale(ctx, eps, prereduce):
    sizes = [256, 100]
    rng = np.random.default_rng(5)
    a = rng.standard_normal((356, 356))
    for i, j in ((0, 0), (0, 1), (1, 0)):
        decay = 0.93
        a[256 * i:256 * i + sizes[i], 256 * j:256 * j + sizes[j]] = _slow_tail(
            rng, sizes[i], sizes[j], 20, decay, 0.9 * eps * np.sqrt(1.0 - decay ** 2))
    off = [0, 256, 356]
    ctx.set_opts(svd_no_prereduce=0 if prereduce else 1)
    try:
        for s in [1.0] + SCALES:
            m = ctx.from_dense(s * a, sizes, eps_lr=s * eps)
            kinds, ranks = m.get_blocks()[:2]
            assert kinds[1, 1] == co.KIND_DENSE
            # the tail's norm is 0.9 eps: the rank is the leading part's (of the kept singular
            # values the smallest is 1e-4)
            lr = [(0, 0), (0, 1), (1, 0)]
            assert all(kinds[ij] == co.KIND_LR for ij in lr), (s, kinds)
            assert all(abs(int(ranks[ij]) - 20) <= 1 for ij in lr), (s, ranks)
            if s == 1.0:
                want = ranks
            assert np.array_equal(ranks, want), (s, ranks)
            d = m.to_dense() / s - a
            for i, j in lr:
                err = np.linalg.norm(d[off[i]:off[i + 1], off[j]:off[j + 1]])
                assert err <= eps * (1 + 1e-6) + 1e-13, (s, i, j, err)
    finally:
        ctx.set_opts(svd_no_prereduce=0)


def test_low_rank_sum_at_any_scale(ctx):
    sizes, r = [256, 130, 64], 24
    rng = np.random.default_rng(6)
    specs = [[], []]
    for m in sizes:
        rows = [[], []]
        for n in sizes:
            k = min(r, min(m, n) // 4)
            common = np.linalg.qr(rng.standard_normal((m, k)))[0]
            for row in rows:
                row.append(_graded(rng, m, n, k, common))
        for spec, row in zip(specs, rows):
            spec.append(row)
    eps, want = 1e-8, None
    try:
        for s in [1.0] + SCALES:
            x, y = (co.from_blocks(sizes, sizes, [[(2, (s * b[0], b[1])) for b in row]
                                                  for row in spec]) for spec in specs)
            ctx.set_opts(eps_lr=s * eps)
            g = clr_pack.from_library(ctx.lincomb(0.75, clr_pack.to_library(ctx, x), -1.5,
                                                  clr_pack.to_library(ctx, y)))
            if want is None:
                want = g.ranks()
            assert (g.kinds() == co.KIND_LR).all() and np.array_equal(g.ranks(), want), s
            exact = 0.75 * x.to_dense() - 1.5 * y.to_dense()
            mag = np.linalg.norm(_abs_dense(x) + _abs_dense(y))
            # nine blocks truncated at s eps
            assert np.linalg.norm(g.to_dense() - exact) <= 3 * s * eps * (1 + 1e-6) + 1e-13 * mag
    finally:
        ctx.set_opts(eps_lr=eps)
