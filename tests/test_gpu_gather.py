"""The pair kernel's gathering step at the sizes where it can go wrong: group and block edges (32), the
padding to a multiple of four, ranges of which nothing or everything is within reach, cells paired with
themselves, every kind, counts only and with sums (counts bit-exact, sums to 1e-6 as everywhere)."""
import numpy as np
import pytest

import gen
from tests.gpu_util import assert_match, gpu_count, oracle_count

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1911_03545_gb300 as cf
    c = cf.cf_create(0, torch.cuda.current_stream())
    yield c
    cf.cf_destroy(c)


def _groups(n, seed, centre, dtype):
    """n points in each of three tight groups: two within reach of each other, one in the next cell but
    mostly out of reach, interleaved so that kept and dropped points alternate along a cell."""
    r = np.random.Generator(np.random.PCG64(seed))
    c = np.array(centre)[:, None] + np.array([[0.0, 3.0, 7.5], [0.0, 1.0, 6.0], [0.0, -2.0, 5.0]])
    p = c[:, None, :] + r.normal(0.0, 0.6, size=(3, n, 3))
    p = p.reshape(3, -1).astype(dtype)
    w = r.uniform(0.5, 1.5, p.shape[1]).astype(dtype)
    return gen.Catalogue(p[0].copy(), p[1].copy(), p[2].copy(), w)


@pytest.mark.parametrize("n", [1, 3, 4, 5, 31, 32, 33, 63, 65, 100, 171])
@pytest.mark.parametrize("kind", ["r", "rppi", "wp", "theta", "mocks"])
def test_gathered_blocks(ctx, kind, n):
    for sums, dtype in ((False, np.float32), (True, np.float32), (True, np.float64)):
        edges = gen.log_edges(0.05, 8.0, 9)
        kw = dict(periodic=False, weighted=sums, ravg=sums)
        centre = (20.0, 20.0, 20.0)
        if kind == "theta":
            edges = gen.log_edges(0.2, 14.0, 9)
        if kind == "mocks":
            centre = (70.0, 60.0, 80.0)
        if kind in ("rppi", "wp"):
            kw.update(periodic=True, box=40.0)
        if kind in ("rppi", "wp", "mocks"):
            kw.update(pimax=6.0, npibins=7)
        d1, d2 = _groups(n, 100 + n, centre, dtype), _groups(2 * n + 1, 200 + n, centre, dtype)
        if kind == "theta":
            for d in (d1, d2):
                r = np.sqrt(d.x.astype(np.float64) ** 2 + d.y.astype(np.float64) ** 2 + d.z.astype(np.float64) ** 2)
                d.x, d.y, d.z = ((v / r).astype(dtype) for v in (d.x, d.y, d.z))
        for auto in (True, False):
            got = gpu_count(ctx, kind, edges, d1, None if auto else d2, autocorr=auto, **kw)
            exp = oracle_count(kind, edges, d1, None if auto else d2, autocorr=auto, mode="brute", **kw)
            assert_match(got, exp, sums, sums)


@pytest.mark.parametrize("n", [2, 8, 9, 16, 17, 24, 36, 40, 48])
@pytest.mark.parametrize("kind", ["r", "rppi", "wp", "theta", "mocks"])
def test_groups_that_share_the_warp(ctx, kind, n):
    """Last groups of up to 4, 8 and 16 points, which have several lanes per point."""
    test_gathered_blocks(ctx, kind, n)


@pytest.mark.parametrize("kind,box,rmax,pimax", [
    ("r", (20.0, 20.0, 20.0), 9.99, 0.0),           # one or two cells on every axis, almost to half the side
    ("r", (90.0, 20.0, 33.0), 9.0, 0.0),            # cells on x and z, explicit on y
    ("rppi", (40.0, 40.0, 25.0), 4.0, 12.5),        # explicit along the line of sight, to half the side
    ("wp", (16.0, 50.0, 30.0), 7.0, 8.0)])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("sums", [False, True])
def test_gathering_across_an_explicit_minimum_image(kind, box, rmax, pimax, dtype, sums):
    """Groups near and across the faces of a box whose axes have fewer than three cells: clumps on the corners, points
    on the faces themselves and on a lattice of half the side.  An explicit minimum image rounds the unwrapped difference,
    and the side, at the side's magnitude, so a pair's separation is off by up to 2 sqrt(3) 2^-24 L besides."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1911_03545_gb300 as cf
    rng = np.random.default_rng(11)
    L = np.array(box)
    pts = [rng.uniform(0.0, 1.0, (900, 3)) * L, (rng.normal(0.0, 0.4, (700, 3)) % L),
           (L / 2 + rng.normal(0.0, 0.4, (700, 3))), rng.integers(0, 3, (200, 3)) * (L / 2)]
    x = np.concatenate(pts).astype(dtype)
    x = np.minimum(np.maximum(x, 0), L.astype(dtype))
    cats = []
    for part in (x, x[::3] * dtype(0.5)):
        c = gen.uniform_box(len(part), 1.0, 1, dtype)
        c.x, c.y, c.z = (np.ascontiguousarray(part[:, a]) for a in range(3))
        c.w = gen.uniform_weights(len(part), 0.5, 1.5, 2).astype(dtype)
        cats.append(c)
    edges = gen.log_edges(0.05, rmax, 9)
    ctx = cf.cf_create(0, torch.cuda.current_stream())
    try:
        for auto in (True, False):
            kw = dict(autocorr=auto, periodic=True, box=box, weighted=sums, ravg=sums)
            if pimax:
                kw.update(pimax=pimax, npibins=5)
            d2 = None if auto else cats[1]
            got = gpu_count(ctx, kind, edges, cats[0], d2, **kw)
            exp = oracle_count(kind, edges, cats[0], d2, **kw)
            assert_match(got, exp, sums)
            if sums:
                tol = 1e-6 * np.asarray(exp["ravg"]) + 2.0 * 3.0 ** 0.5 * 2.0 ** -24 * max(box)
                assert np.all(np.abs(got["ravg"] - exp["ravg"]) <= tol)
    finally:
        cf.cf_destroy(ctx)


@pytest.mark.parametrize("kind,npi", [("rppi", 3), ("wp", 1), ("rppi", 1)])
@pytest.mark.parametrize("pimax,step", [(2.5e-39, 1e-39), (4e20, 1.7e20)])
def test_pi_limits_at_the_ends_of_float32(ctx, kind, npi, pimax, step):
    """Limits along the line of sight whose inverse, or whose square, does not fit float32."""
    rng = np.random.default_rng(4)
    n = 700
    c = gen.uniform_box(n, 10.0, 3, np.float32)
    c.z = (rng.integers(0, 6, n) * step).astype(np.float32)
    edges, kw = gen.log_edges(0.1, 5.0, 5), dict(autocorr=True, periodic=False, pimax=pimax, npibins=npi)
    got = gpu_count(ctx, kind, edges, c, None, **kw)
    exp = oracle_count(kind, edges, c, None, mode="brute", **kw)
    assert 0 < int(np.asarray(got["npairs"]).sum()) < n * n
    assert_match(got, exp)
