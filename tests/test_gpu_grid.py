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
