"""Which tiles of a recompression take a team of CTAs: all of a few, the leading ones of more whose
costs differ, none of equal ones; and that the tiles a product hands over from teams to single CTAs
have the same bits as by single CTAs alone."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1509_00309_gb300 import build, clr
    build.build()
    return clr.Context(0, precision="fp64", eps_lr=1e-8)


def _kernel(sizes):
    n = sum(sizes)
    rng = np.random.default_rng(n)
    r = 0.02 * np.arange(n) + rng.uniform(-0.004, 0.004, n)
    return np.exp(-(r[:, None] - r[None, :]) ** 2 / 2.0) + 1e-3 * np.eye(n)


def _team_tiles(ctx, run):
    ctx.profile_enable(True)
    try:
        run()
        return ctx.profile_team_tiles()
    finally:
        ctx.profile_enable(False)


def _ctas():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count // 4 * 4


def test_teams_take_all_of_few_blocks(ctx):
    sizes = [256, 97, 16, 200]
    a = _kernel(sizes)
    assert 2 * len(sizes) ** 2 <= _ctas()
    assert _team_tiles(ctx, lambda: ctx.from_dense(a, sizes, eps_lr=1e-8)) == 16


def test_teams_take_the_leading_of_many_tiles(ctx):
    # more tiles than half the CTAs, fewer than twice as many
    nb = math.isqrt(_ctas()) + 1
    assert _ctas() < 2 * nb ** 2 and nb ** 2 <= 2 * _ctas()
    ctx.set_opts(recompress_dense=1)
    try:
        for sizes, some in (([256, 230] + ([40, 25, 33, 48, 7, 60, 22, 37, 51, 1, 44] * 3)[:nb - 2], True),
                            ([64] * nb, False)):
            s = ctx.from_dense(_kernel(sizes), sizes, eps_lr=1e-10)
            # by the sizes in a new matrix, then by the costs measured in it
            out = []
            n = _team_tiles(ctx, lambda: out.append(ctx.multiply(s, s)))
            assert 0 < n < nb ** 2 if some else n == 0, n
            first = out[0].to_dense()
            n = _team_tiles(ctx, lambda: ctx.multiply_into(s, s, out[0]))
            assert not some or 0 < n < nb ** 2, n
            assert np.array_equal(out[0].to_dense(), first)
    finally:
        ctx.set_opts(recompress_dense=0)
