"""What a context counted before, or was limited to before, decides neither the grid nor the work list of a call."""
import numpy as np
import pytest

import gen
from tests.gpu_util import assert_match, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture
def make():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1911_03545_gb300 as cf
    made = []

    def new(**opts):
        made.append(cf.cf_create(0, torch.cuda.current_stream()))
        for k, v in opts.items():
            cf.cf_set_option(made[-1], getattr(cf, k), v)
        return made[-1]
    yield new
    for c in made:
        cf.cf_destroy(c)


@pytest.mark.parametrize("cap", [0, 1 << 30])
def test_the_number_of_sets_is_part_of_the_plan(make, cap):
    """64,000 points of one catalogue or of 32 in the same box: the cells' width goes by their number."""
    import paper_1911_03545_gb300 as cf
    p = cf.params(kind="r", edges=gen.log_edges(0.1, 5.0, 7), autocorr=True, periodic=True, box=200.0)
    whole = gen.uniform_box(64_000, 200.0, 1, np.float32)
    one = [cf.points(*to_dev(whole, "cuda:0", False))]
    many = [cf.points(*to_dev(gen.uniform_box(2_000, 200.0, 5 + i, np.float32), "cuda:0", False)) for i in range(32)]
    cells = {}
    for name, first, second in (("one", many, one), ("many", one, many)):
        fresh, used = make(CF_OPT_MEM_CAP=cap), make(CF_OPT_MEM_CAP=cap)
        exp = cf.cf_batch_count(fresh, p, second)
        cells[name] = cf.cf_get_stats(fresh)["cells"]
        cf.cf_batch_count(used, p, first)
        got = cf.cf_batch_count(used, p, second)
        assert cf.cf_get_stats(used)["cells"] == cells[name]
        for g, e in zip(got, exp):
            assert_match(g, e)
    assert cells["many"] < cells["one"]


def test_a_larger_cap_gives_the_small_items_back(make):
    """A list that did not fit is made with the largest items; once the cap is raised the shape is open again."""
    import paper_1911_03545_gb300 as cf
    p = cf.params(kind="r", edges=gen.log_edges(0.1, 10.0, 8), autocorr=True, periodic=True, box=100.0)
    pts = cf.points(*to_dev(gen.uniform_box(60_000, 100.0, 1, np.float32), "cuda:0", False))
    exp = cf.cf_count(make(CF_OPT_MEM_CAP=1 << 30), p, pts)
    wide = make(CF_OPT_MEM_CAP=1 << 30)
    cf.cf_count(wide, p, pts)
    fine = cf.cf_get_stats(wide)["work_items"]
    ctx = make()
    for cap in range(1 << 21, 1 << 25, 1 << 18):
        cf.cf_set_option(ctx, cf.CF_OPT_MEM_CAP, cap)
        try:
            assert_match(cf.cf_count(ctx, p, pts), exp)
        except cf.CfError as e:
            assert "cap" in str(e)
            continue
        break
    assert cf.cf_get_stats(ctx)["work_items"] < fine
    cf.cf_set_option(ctx, cf.CF_OPT_MEM_CAP, 1 << 30)
    assert_match(cf.cf_count(ctx, p, pts), exp)
    assert cf.cf_get_stats(ctx)["work_items"] == fine


def _fits(cf, make, cap, *calls):
    """Whether the calls (params, points) all pass in turn, twice each, in a new context with that cap."""
    ctx = make(CF_OPT_MEM_CAP=int(cap))
    try:
        for p, pts in calls:
            for _ in range(2):
                cf.cf_count(ctx, p, pts)
    except cf.CfError as e:
        assert "cap" in str(e)
        return False
    return True


@pytest.mark.parametrize("n,box", [(10_000, 100.0), (60_000, 100.0)])
def test_a_larger_cap_never_refuses_what_a_smaller_one_takes(make, n, box):
    import paper_1911_03545_gb300 as cf
    p = cf.params(kind="r", edges=gen.log_edges(0.1, 10.0, 10), autocorr=True, periodic=True, box=box)
    pts = cf.points(*to_dev(gen.uniform_box(n, box, 1, np.float32), "cuda:0", False))
    took = [_fits(cf, make, cap, (p, pts)) for cap in range(16_000_000, 28_000_000, 250_000)]
    assert True in took and False in took
    assert took == sorted(took)


def test_a_call_that_fits_alone_fits_after_another(make):
    """Dense points make a long list; the cap then has to hold more points with a short one."""
    import paper_1911_03545_gb300 as cf
    dense = (cf.params(kind="r", edges=gen.log_edges(0.1, 12.0, 8), autocorr=True, periodic=True, box=60.0, refine=(2, 2, 2)),
             cf.points(*to_dev(gen.uniform_box(150_000, 60.0, 1, np.float32), "cuda:0", False)))
    wide = (cf.params(kind="r", edges=gen.log_edges(0.1, 2.0, 8), autocorr=True, periodic=True, box=200.0),
            cf.points(*to_dev(gen.uniform_box(400_000, 200.0, 2, np.float32), "cuda:0", False)))
    lo, hi = 1 << 20, 1 << 28
    while hi - lo > 1 << 17:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if _fits(cf, make, mid, wide) else (mid, hi)
    ctx = make(CF_OPT_MEM_CAP=hi)
    try:
        cf.cf_count(ctx, *dense)
    except cf.CfError as e:
        assert "cap" in str(e)
    assert_match(cf.cf_count(ctx, *wide), cf.cf_count(make(), *wide))


def test_a_queue_that_does_not_fit_is_forgotten(make):
    """A lattice whose separations all lie on edges needs a queue past the cap; the next call does not."""
    import paper_1911_03545_gb300 as cf
    k = np.arange(40, dtype=np.float32)
    x, y, z = (np.ascontiguousarray(a.ravel()) for a in np.meshgrid(k, k, k, indexing="ij"))
    grid = gen.Catalogue(x, y, z, None)
    p = cf.params(kind="r", edges=[1.0, 2.0, 3.0, 4.0], autocorr=True, periodic=True, box=40.0)
    small = (cf.params(kind="r", edges=gen.log_edges(0.1, 10.0, 10), autocorr=True, periodic=True, box=100.0),
             cf.points(*to_dev(gen.uniform_box(10_000, 100.0, 1, np.float32), "cuda:0", False)))
    ctx = make(CF_OPT_MEM_CAP=28_000_000)
    for _ in range(2):
        with pytest.raises(cf.CfError, match="cap"):
            cf.cf_count(ctx, p, cf.points(*to_dev(grid, "cuda:0", False)))
        assert_match(cf.cf_count(ctx, *small), cf.cf_count(make(), *small))
