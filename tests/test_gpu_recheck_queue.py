"""The FP64 recheck on queues short and long, for tables that fit its shared counters and one that does not
(the audit option queues every pair): counts equal to the oracle's, points on a lattice so that values fall
on edges."""
import numpy as np
import pytest

import gen
from tests.gpu_util import assert_match, gpu_count, oracle_count

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,nb,npi", [("r", 1, 0), ("r", 14, 0), ("wp", 14, 40), ("rppi", 12, 40), ("rppi", 20, 120),
                                         ("mocks", 14, 42)])
def test_recheck_of_short_and_long_queues(kind, nb, npi):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1911_03545_gb300 as cf
    ctx = cf.cf_create(0, torch.cuda.current_stream())
    cf.cf_set_option(ctx, cf.CF_OPT_AUDIT, 1)
    try:
        for n in (40, 127, 130, 700):         # 130 points: more than 8192 pairs
            r = np.random.Generator(np.random.PCG64(n))
            p = (r.integers(0, 40, (3, n)) * 0.25 + (60.0 if kind == "mocks" else 0.0)).astype(np.float64)
            cat = gen.Catalogue(p[0].copy(), p[1].copy(), p[2].copy(), r.uniform(0.5, 1.5, n))
            edges = np.linspace(0.0 if kind == "r" else 0.25, 8.0, nb + 1)
            kw = dict(autocorr=True, periodic=False, weighted=True, ravg=True)
            if npi:
                kw.update(pimax=8.0, npibins=npi)
            got = gpu_count(ctx, kind, edges, cat, **kw)
            exp = oracle_count(kind, edges, cat, None, mode="brute", **kw)
            assert_match(got, exp, True, True)
    finally:
        cf.cf_destroy(ctx)
