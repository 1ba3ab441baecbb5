"""The work list of cell pairs of many items: every tile pair of a cell with itself (the triangle) and with
another cell exactly once, at the edges of tiles and ranges and with the smallest of both."""
import numpy as np
import pytest

import gen
from tests.gpu_util import gpu_count

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [32, 33, 64, 65, 97, 1000, 4097, 30_001])
def test_every_pair_of_a_cell_once(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1911_03545_gb300 as cf
    ctx = cf.cf_create(0, torch.cuda.current_stream())
    try:
        a, b = gen.uniform_box(n, 1.0, 1, np.float32), gen.uniform_box(n // 3 + 1, 1.0, 2, np.float32)
        edges = [0.0, 1.0, 2.0]          # every pair of the unit box counts
        for tile, jchunk in ((0, 0), (32, 32), (64, 128)):
            cf.cf_set_option(ctx, cf.CF_OPT_TILE, tile)
            cf.cf_set_option(ctx, cf.CF_OPT_JCHUNK, jchunk)
            for refine in (1, 2):
                kw = dict(periodic=False, refine=(refine,) * 3)
                auto = gpu_count(ctx, "r", edges, a, autocorr=True, **kw)
                assert int(np.asarray(auto["npairs"]).astype(np.uint64).sum()) == n * n       # the points themselves too
                cross = gpu_count(ctx, "r", edges, a, b, autocorr=False, **kw)
                assert int(np.asarray(cross["npairs"]).astype(np.uint64).sum()) == n * (n // 3 + 1)
    finally:
        cf.cf_destroy(ctx)


def test_a_list_that_does_not_fit_takes_larger_items():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1911_03545_gb300 as cf
    n = 60_000
    cat = gen.uniform_box(n, 100.0, 1, np.float32)
    edges, kw = gen.log_edges(0.1, 10.0, 8), dict(autocorr=True, periodic=True, box=100.0)
    free, capped = (cf.cf_create(0, torch.cuda.current_stream()) for _ in range(2))
    try:
        exp = gpu_count(free, "r", edges, cat, **kw)
        fine = cf.cf_get_stats(free)["work_items"]
        used = 0
        for cap in range(1 << 21, 1 << 25, 1 << 18):
            cf.cf_set_option(capped, cf.CF_OPT_MEM_CAP, cap)
            try:
                got = gpu_count(capped, "r", edges, cat, **kw)
            except cf.CfError as e:
                assert "cap" in str(e)
                continue
            used = cf.cf_get_stats(capped)["work_items"]
            break
        assert 0 < used < fine
        np.testing.assert_array_equal(got["npairs"], exp["npairs"])
        again = gpu_count(capped, "r", edges, cat, **kw)
        np.testing.assert_array_equal(again["npairs"], exp["npairs"])
    finally:
        cf.cf_destroy(free)
        cf.cf_destroy(capped)


@pytest.mark.parametrize("n,m,large", [(420_000, 5_000, True), (5_000, 420_000, False), (300_000, 5_000, False)])
def test_few_j_points_per_cell_take_large_tiles(n, m, large):
    """Counts of the pinned tile, and the number of items that the open one makes."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1911_03545_gb300 as cf
    cats = [gen.uniform_box(k, 200.0, s, np.float32) for s, k in ((1, n), (2, m))]
    edges = gen.log_edges(0.1, 12.0, 7)
    ctx = cf.cf_create(0, torch.cuda.current_stream())
    try:
        outs, items = [], []
        for tile in (0, 64, 128):
            cf.cf_set_option(ctx, cf.CF_OPT_TILE, tile)
            outs.append(gpu_count(ctx, "r", edges, *cats, autocorr=False, periodic=True, box=200.0))
            items.append(cf.cf_get_stats(ctx)["work_items"])
        assert items[0] == items[2 if large else 1]
        for o in outs[1:]:
            np.testing.assert_array_equal(o["npairs"], outs[0]["npairs"])
    finally:
        cf.cf_destroy(ctx)


@pytest.mark.parametrize("n,m,box,small", [(660, 7_700, 8.0, True), (2_000, 0, 8.0, True), (8_000, 0, 8.0, False),
                                           (30_000, 0, 41.0, True)])
def test_small_dense_calls_take_small_items(n, m, box, small):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1911_03545_gb300 as cf
    cats = [gen.uniform_box(k, box, s, np.float32) for s, k in ((1, n), (2, max(m, 1)))]
    edges = gen.log_edges(0.1, 10.0, 7)
    ctx = cf.cf_create(0, torch.cuda.current_stream())
    try:
        outs, items = [], []
        for tile, jchunk in ((0, 0), (64, 128), (128, 512)):
            cf.cf_set_option(ctx, cf.CF_OPT_TILE, tile)
            cf.cf_set_option(ctx, cf.CF_OPT_JCHUNK, jchunk)
            outs.append(gpu_count(ctx, "r", edges, cats[0], cats[1] if m else None, autocorr=not m, periodic=False,
                                  refine=(1, 1, 1)))
            items.append(cf.cf_get_stats(ctx)["work_items"])
        assert items[1] != items[2] and items[0] == items[1 if small else 2]
        for o in outs[1:]:
            np.testing.assert_array_equal(o["npairs"], outs[0]["npairs"])
    finally:
        cf.cf_destroy(ctx)
