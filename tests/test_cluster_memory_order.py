"""The order of accesses to memory that the CTAs of a cluster share, read from the sources: a store
to (or load from) another CTA's shared memory is undefined before that CTA is known to have started,
which only a cluster barrier shows.  A violation is a race that may never show in a result, so it
is looked for in the text and not by running the kernels."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1509_00309_gb300", "csrc")


def _function(file, name):
    """The body of function `name`, without comments."""
    with open(os.path.join(CSRC, file)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    start = text.index("{", re.search(r"\b%s\(" % name, text).end())
    depth = 0
    for i in range(start, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[start:i + 1]
    raise AssertionError(name)


@pytest.mark.parametrize("file,kernel,barrier,access", [
    ("k_lowrank.cu", "lr_products_kernel", "cluster.sync()", "map_shared_rank("),
    ("k_ns.cu", "lincomb_apply_kernel", "cluster.sync()", "map_shared_rank("),
    ("k_ns.cu", "matvec_kernel", "cluster.sync()", "map_shared_rank("),
    ("k_dense64.cu", "dense_tile_norms_kernel", "cluster.sync()", "map_shared_rank("),
    ("k_svd.cu", "compress_dense_body", "if (team) tm.sync()", "tm.put("),
])
def test_a_cluster_barrier_precedes_the_first_access_to_a_peer(file, kernel, barrier, access):
    body = _function(file, kernel)
    assert 0 <= body.index(barrier) < body.index(access)


def test_the_series_powers_in_a_teams_scratch_are_dealt_over_the_team():
    # F and F^2 lie in one global scratch for all CTAs of a team where they do not fit shared
    # memory: each entry is then written by one thread of the team, and read behind its barrier
    share = _function("k_svd.cu", "FloatShare")
    assert "t0 = own ? (int)threadIdx.x : tm.tid" in share and "own ? kThreads : tm.nt" in share
    for name, stores in (("small_series", ["f"]), ("orthonormalise_fp64", ["f", "w"])):
        # (a store by every CTA for itself only under fs.own)
        body = _function("k_svd.cu", name).replace("if (fs.own) f[x] = v;", "")
        loop = body.index("for (int x = fs.t0; x < q * q; x += fs.step)")
        for m in stores:
            assert body.count(m + "[x] =") == 1 and body.index(m + "[x] =") > loop
        assert loop < body.index("tm.sync();", loop) < body.index("cta_gemm_auto(")
