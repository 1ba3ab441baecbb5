"""The one-launch build's bounded wait, made to run out by its poll limit (a wait of two polls is over before the last
block arrives): the call, the replay and what follows them on the same context return the right counts."""
import numpy as np
import pytest

import gen
from tests.gpu_util import assert_match, gpu_count, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1911_03545_gb300 as cf
    c = cf.cf_create(0, torch.cuda.current_stream())
    yield c
    cf.cf_destroy(c)


@pytest.mark.parametrize("late", ["new", "used"])
@pytest.mark.parametrize("periodic", [True, False])
def test_a_call_whose_build_gives_up(ctx, late, periodic):
    import paper_1911_03545_gb300 as cf
    cat = gen.uniform_box(20_000, 100.0, 1, np.float32)
    edges, kw = gen.log_edges(0.1, 9.0, 8), dict(autocorr=True, periodic=periodic, box=100.0)
    exp = None
    if late == "used":
        exp = gpu_count(ctx, "r", edges, cat, **kw)
        assert cf.cf_get_stats(ctx)["kernel_launches"] <= 4          # the one-launch build
    cf.cf_set_option(ctx, cf.CF_OPT_ITER_LIMIT, 1)
    got = gpu_count(ctx, "r", edges, cat, **kw)
    assert cf.cf_get_stats(ctx)["kernel_launches"] > 4               # the general one
    cf.cf_set_option(ctx, cf.CF_OPT_ITER_LIMIT, 0)
    cf.cf_set_option(ctx, cf.CF_OPT_BLOCK_PRUNE, 1)
    want = gpu_count(ctx, "r", edges, cat, **kw)
    assert_match(got, want)
    if exp is not None:
        assert_match(exp, want)


def test_a_replay_whose_build_gives_up(ctx):
    import torch

    import paper_1911_03545_gb300 as cf
    cats = [gen.uniform_box(n, 100.0, n, np.float32) for n in (20_000, 5_001, 1)]
    edges = gen.log_edges(0.1, 9.0, 8)
    p = cf.params(kind="r", edges=edges, autocorr=True, periodic=True, box=100.0)
    pts = [cf.points(*to_dev(c, "cuda:0", False)) for c in cats]
    other = cf.cf_create(0, torch.cuda.current_stream())
    try:
        cf.cf_set_option(other, cf.CF_OPT_BLOCK_PRUNE, 1)
        want = [gpu_count(other, "r", edges, c, autocorr=True, periodic=True, box=100.0) for c in cats]
    finally:
        cf.cf_destroy(other)

    def check(outs):
        for got, exp in zip(outs, want):
            assert_match(got, exp)

    cf.cf_batch_capture(ctx, p, pts)
    check(cf.cf_batch_replay(ctx, p, 3))
    cf.cf_set_option(ctx, cf.CF_OPT_ITER_LIMIT, 1)
    check(cf.cf_batch_replay(ctx, p, 3))                             # gives up, and is counted without the graph
    assert cf.cf_get_stats(ctx)["kernel_launches"] > 5
    with pytest.raises(cf.CfError, match="no captured batch"):
        cf.cf_batch_replay(ctx, p, 3)
    cf.cf_batch_capture(ctx, p, pts)
    for _ in range(2):
        check(cf.cf_batch_replay(ctx, p, 3))
    check(cf.cf_batch_count(ctx, p, pts))
