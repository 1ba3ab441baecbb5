"""Work items of a cell pair, counted past 32 bits: the header's own functions, compiled for the host, against exact
integers at the sizes where a product of 32 bits wraps, and the calls that reach such counts."""
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1911_03545_gb300", "csrc")
PROG = """
#include <cstdio>
#include <cstdlib>
#include "cf_internal.h"
int main(int c, char **v)
{
    const uint32_t n = strtoul(v[1], 0, 10), m = strtoul(v[2], 0, 10);
    printf("%llu %llu\\n", (unsigned long long)cfi_item_count(n, n, true), (unsigned long long)cfi_item_count(n, m, false));
    for (int i = 3; i < c; i++) {
        uint32_t a, b;
        cfi_tile_pair(n, (uint32_t)strtoull(v[i], 0, 10), a, b);
        printf("%u %u\\n", a, b);
    }
}
"""


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    d = tmp_path_factory.mktemp("items")
    (d / "p.cpp").write_text(PROG)
    exe = str(d / "p")
    subprocess.run(["g++", "-O1", "-I" + CSRC, "-I" + os.path.join(os.path.dirname(os.path.dirname(CSRC)), "include"),
                    str(d / "p.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("n", [1, 2, 3, 257, 65_535, 65_536, 65_537, 65_625, 92_681])
def test_counts_and_tile_pairs(prog, n):
    total = n * (n + 1) // 2
    rows = sorted({0, 1, n // 3, n // 2, n - 2, n - 1} & set(range(n)))
    want = []       # (place, a, b): the first, second and last pair of some rows
    for a in rows:
        first = a * n - a * (a - 1) // 2
        want += [(first + b - a, a, b) for b in sorted({a, min(a + 1, n - 1), n - 1})]
    out = subprocess.run([prog, str(n), str(3 * n + 1)] + [str(k) for k, _, _ in want], check=True,
                         capture_output=True, text=True).stdout.split("\n")
    assert out[0] == f"{total} {n * (3 * n + 1)}"
    assert [tuple(map(int, s.split())) for s in out[1:len(want) + 1]] == [(a, b) for _, a, b in want]


def _count(ctx, cf, edges, sets, **kw):
    import torch
    p = cf.params(kind="r", edges=edges, **kw)
    pts = [cf.points(*[torch.from_numpy(a).to("cuda:0") for a in s]) for s in sets]
    return cf.cf_count(ctx, p, *pts)


@pytest.mark.gpu
def test_a_cell_of_more_tile_pairs_than_32_bits_hold():
    """4.2 million points in one cell of a sparse grid are 2,153,353,125 items: they do not fit the cap, and the call
    has to say so instead of counting a few of them."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1911_03545_gb300 as cf
    rng = np.random.default_rng(1)
    s = [rng.uniform(0.1, 0.9, 4_200_000).astype(np.float32) for _ in range(3)]
    for a in s:
        a[0], a[1] = 0.0, 24.99          # the box, 24 cells on a side
    ctx = cf.cf_create(0, torch.cuda.current_stream())
    try:
        cf.cf_set_option(ctx, cf.CF_OPT_MEM_CAP, 2 << 30)
        with pytest.raises(cf.CfError, match="cap"):
            _count(ctx, cf, [0.01, 0.1, 1.0], [s], autocorr=True)
        few = [a[:40_000] for a in s]
        assert int(_count(ctx, cf, [0.0, 1.0, 50.0], [few], autocorr=True)["npairs"].astype(np.uint64).sum()) == 40_000 ** 2
    finally:
        cf.cf_destroy(ctx)


@pytest.mark.gpu
@pytest.mark.parametrize("prune", [0, 1])
def test_a_cell_pair_of_more_items_than_32_bits_hold(prune):
    """Items of 32 x 1 points pinned: 372,000 x 372,000 points of one cell are 4,324,500,000 of them, past the limit."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1911_03545_gb300 as cf
    rng = np.random.default_rng(2)
    sets = [[rng.uniform(0.0, 1.0, 372_000).astype(np.float32) for _ in range(3)] for _ in range(2)]
    ctx = cf.cf_create(0, torch.cuda.current_stream())
    try:
        cf.cf_set_option(ctx, cf.CF_OPT_CELL_PRUNE, prune)
        cf.cf_set_option(ctx, cf.CF_OPT_REFINE, 1)
        cf.cf_set_option(ctx, cf.CF_OPT_TILE, 32)
        cf.cf_set_option(ctx, cf.CF_OPT_JCHUNK, 1)
        with pytest.raises(cf.CfError, match="work list"):
            _count(ctx, cf, [0.01, 0.1, 2.0], sets, autocorr=False)
        few = [[a[:500] for a in s] for s in sets]
        out = _count(ctx, cf, [0.0, 1.0, 2.0], few, autocorr=False)
        assert int(out["npairs"].astype(np.uint64).sum()) == 500 ** 2
    finally:
        cf.cf_destroy(ctx)
