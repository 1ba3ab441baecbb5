"""Sparse catalogues, whose cells the plan widens: the counts must be those of the grid with cells as wide
as the largest separation (pinned by the refinement factor 1) bit for bit, the sums to 1e-6."""
import numpy as np
import pytest

import gen
from tests.gpu_util import assert_match, gpu_count

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,auto,periodic,dtype", [
    ("r", True, True, np.float32), ("r", False, False, np.float64), ("rppi", True, True, np.float64),
    ("rppi", False, True, np.float32), ("wp", True, False, np.float32), ("theta", True, False, np.float32),
    ("mocks", False, False, np.float32)])
def test_widened_cells_keep_results(kind, auto, periodic, dtype):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1911_03545_gb300 as cf
    n = 60_001
    edges = gen.log_edges(0.1, 6.0, 9)
    kw = dict(autocorr=auto, periodic=periodic, box=200.0, weighted=True, ravg=True)
    if kind in ("rppi", "wp", "mocks"):
        kw.update(pimax=9.0, npibins=6)
    if kind == "theta":
        edges = gen.log_edges(0.02, 0.5, 9)
        cats = [gen.sphere_patch(n, 0.0, 180.0, -60.0, 60.0, s) for s in (1, 2)]
    elif kind == "mocks":
        edges = gen.log_edges(0.5, 6.0, 9)
        cats = [gen.survey_cone(n, 0.0, 90.0, 0.0, 60.0, 300.0, 420.0, s) for s in (1, 2)]
    else:
        cats = [gen.uniform_box(n, 200.0, s, dtype) for s in (1, 2)]
    for s, c in enumerate(cats):
        c.w = gen.uniform_weights(n, 0.5, 1.5, 10 + s).astype(c.x.dtype)
    ctx = cf.cf_create(0, torch.cuda.current_stream())
    try:
        d2 = None if auto else cats[1]
        got = gpu_count(ctx, kind, edges, cats[0], d2, **kw)
        wide = cf.cf_get_stats(ctx)["cells"]
        exp = gpu_count(ctx, kind, edges, cats[0], d2, refine=(1, 1, 1), **kw)
        assert wide < cf.cf_get_stats(ctx)["cells"]
        assert int(np.asarray(got["npairs"]).sum()) > 1000
        assert_match(got, exp, True, True)
    finally:
        cf.cf_destroy(ctx)


@pytest.mark.parametrize("kind,auto,periodic,n", [
    ("r", True, True, 33_000), ("r", False, False, 60_001), ("rppi", True, True, 60_001), ("wp", False, True, 40_003),
    ("mocks", False, False, 40_003)])
def test_halved_cells_keep_results(kind, auto, periodic, n):
    """Dense catalogues, whose cells the plan halves: counts of the grid with whole cells, bit for bit."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1911_03545_gb300 as cf
    box = 60.0 if kind in ("r", "mocks") else 50.0
    edges = gen.log_edges(0.1, 15.0, 9)
    kw = dict(autocorr=auto, periodic=periodic, box=box if periodic else 0.0, weighted=True, ravg=True)
    if kind in ("rppi", "wp", "mocks"):
        kw.update(pimax=15.0 if kind != "mocks" else 9.0, npibins=6)
    cats = [gen.uniform_box(m, box, s, np.float32) for s, m in ((1, n), (2, n // 2))]
    for s, c in enumerate(cats):
        if kind == "mocks":
            for a in (c.x, c.y, c.z):
                a += np.float32(300.0)
        c.w = gen.uniform_weights(len(c.x), 0.5, 1.5, 10 + s).astype(c.x.dtype)
    ctx = cf.cf_create(0, torch.cuda.current_stream())
    try:
        d2 = None if auto else cats[1]
        got = gpu_count(ctx, kind, edges, cats[0], d2, **kw)
        st = cf.cf_get_stats(ctx)
        exp = gpu_count(ctx, kind, edges, cats[0], d2, refine=(1, 1, 1), **kw)
        assert st["refine"] == [2, 2, 2] and st["cells"] == 8 * cf.cf_get_stats(ctx)["cells"]
        assert_match(got, exp, True, True)
    finally:
        cf.cf_destroy(ctx)


@pytest.mark.parametrize("kind,sizes,auto,halved", [
    ("r", (2_000, 100_000), False, False), ("r", (100_000, 2_000), False, False), ("r", (60_000, 100_000), False, False),
    ("r", (70_000, 100_000), False, True), ("r", (100_000, 3_000, 40_000), True, False),
    ("r", (60_000,) + (100,) * 20, True, False), ("r", (100_000, 60_000), True, False), ("r", (100_000, 70_000), True, True),       # 480 and 560 per cell
    ("rppi", (2_000, 100_000), False, False), ("rppi", (20_000, 100_000), False, True),
    ("mocks", (500, 100_000), False, False), ("mocks", (5_000, 100_000), False, True)])
def test_unequal_sets_are_not_halved(kind, sizes, auto, halved):
    """Cells are halved where both sets of every pair fill them: a few points against dense ones, or small catalogues
    beside a large one, keep whole cells, which the small ones do not widen either."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1911_03545_gb300 as cf
    from tests.gpu_util import to_dev
    box, edges = 60.0, gen.log_edges(0.1, 12.0, 7)
    kw = dict(kind=kind, edges=edges, autocorr=auto, periodic=kind != "mocks", box=box)
    if kind != "r":
        kw.update(pimax=12.0 if kind == "rppi" else 6.0, npibins=5)
    cats = [gen.uniform_box(n, box, 3 + i, np.float32) for i, n in enumerate(sizes)]
    if kind == "mocks":
        for c in cats:
            for a in (c.x, c.y, c.z):
                a += np.float32(300.0)
    pts = [cf.points(*to_dev(c, "cuda:0", False)) for c in cats]
    ctx = cf.cf_create(0, torch.cuda.current_stream())
    try:
        outs, cells = [], []
        for refine in ((0, 0, 0), (1, 1, 1)):
            p = cf.params(refine=refine, **kw)
            outs.append(cf.cf_batch_count(ctx, p, pts) if auto else [cf.cf_count(ctx, p, *pts)])
            want = 2 if halved and refine[0] == 0 else 1
            assert cf.cf_get_stats(ctx)["refine"] == [want] * 3
            cells.append(cf.cf_get_stats(ctx)["cells"])
        assert cells[0] == (8 if halved else 1) * cells[1]
        for got, exp in zip(*outs):
            assert_match(got, exp)
    finally:
        cf.cf_destroy(ctx)


@pytest.mark.parametrize("n,cells", [(3, 97), (40_000, 90), (5_003, 41), (20_000, 60)])
def test_boxes_of_mostly_empty_cells(n, cells):
    """Grids of more cells than the boxes' pass has warps for one each (a warp then takes up to 32), and one of just
    more: counts of the call that uses no boxes."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1911_03545_gb300 as cf
    box = 10.0 * cells
    cat = gen.uniform_box(n, box, 5, np.float32)
    for a in (cat.x, cat.y, cat.z):
        a[n // 2:] = a[: n - n // 2] + np.float32(0.3)       # pairs, one of them in the next cell here and there
        np.minimum(a, np.float32(box), out=a)
    edges = gen.log_edges(0.1, 10.0, 7)
    ctx = cf.cf_create(0, torch.cuda.current_stream())
    try:
        outs = []
        for prune in (0, 1):
            cf.cf_set_option(ctx, cf.CF_OPT_CELL_PRUNE, prune)
            outs.append(gpu_count(ctx, "r", edges, cat, autocorr=True, periodic=True, box=box, refine=(1, 1, 1)))
            assert cf.cf_get_stats(ctx)["cells"] > 65_536
        assert int(np.asarray(outs[0]["npairs"]).sum()) > n // 2
        assert_match(outs[0], outs[1])
    finally:
        cf.cf_destroy(ctx)
