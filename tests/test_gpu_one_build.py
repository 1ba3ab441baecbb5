"""The one-launch build of small calls against the general build (taken with group pruning on): the counts bit
for bit, at the edges of its ranges (points, sort keys, sub-cells), one context through all sizes in turn."""
import numpy as np
import pytest

import gen
from tests.gpu_util import assert_match, gpu_count

pytestmark = pytest.mark.gpu

# (points, box, largest separation, refinement, sub-cells per axis, whether one launch builds it)
SIZES = [(262_144, 100.0, 4.0, 0, 0, True), (1, 100.0, 9.0, 1, 0, True), (262_145, 100.0, 4.0, 0, 0, False),
         (20_000, 108.5, 3.0, 1, 0, True),         # 36^3 cells: the most that fit the keys
         (20_000, 111.5, 3.0, 1, 0, False),        # 37^3 cells
         (5_003, 82.0, 9.0, 1, 4, True), (5_003, 91.0, 10.0, 1, 1, True), (5_003, 200.0, 9.0, 1, 4, False),
         (257, 30.0, 9.0, 2, 2, True)]


def test_one_launch_build_keeps_counts():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1911_03545_gb300 as cf
    one, gen_ctx = (cf.cf_create(0, torch.cuda.current_stream()) for _ in range(2))
    cf.cf_set_option(gen_ctx, cf.CF_OPT_BLOCK_PRUNE, 1)
    try:
        for turn in range(2):
            for n, box, rmax, refine, sub, small in SIZES[::1 if turn == 0 else -1]:
                cat = gen.uniform_box(n, box, 3 + turn, np.float32)
                kw = dict(autocorr=True, periodic=True, box=box, refine=(refine,) * 3)
                edges = gen.log_edges(0.1, rmax, 8)
                got = []
                for ctx in (one, gen_ctx):
                    cf.cf_set_option(ctx, cf.CF_OPT_CELL_ORDER, sub)
                    gpu_count(ctx, "r", edges, cat, None, **kw)
                    got.append(gpu_count(ctx, "r", edges, cat, None, **kw))
                launches = cf.cf_get_stats(one)["kernel_launches"]
                assert (launches <= 4) == small, (n, box, launches)
                assert_match(got[0], got[1])
    finally:
        cf.cf_destroy(one)
        cf.cf_destroy(gen_ctx)


@pytest.mark.parametrize("refine,whole,small", [(2, 12, True), (2, 14, False), (3, 6, True), (3, 10, False)])
def test_refined_grids_of_many_cells_take_the_general_build(refine, whole, small):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1911_03545_gb300 as cf
    cat = gen.uniform_box(9_001, 10.0 * whole, 4, np.float32)
    edges = gen.log_edges(0.1, 10.0, 8)
    kw = dict(autocorr=True, periodic=True, box=10.0 * whole)
    ctx = cf.cf_create(0, torch.cuda.current_stream())
    try:
        for _ in range(2):
            got = gpu_count(ctx, "r", edges, cat, None, refine=(refine,) * 3, **kw)
            assert cf.cf_get_stats(ctx)["cells"] == (refine * whole) ** 3
            assert (cf.cf_get_stats(ctx)["kernel_launches"] <= 4) == small
        assert_match(got, gpu_count(ctx, "r", edges, cat, None, refine=(1, 1, 1), **kw))
    finally:
        cf.cf_destroy(ctx)
