"""Performance cases of the pair counter: what a user has it count, through the public entry points.

A case is a dict of plain values (see `_case`).  `prepare` draws a catalogue on the GPU and keeps what
a user's program keeps (the parameters, the point sets and one context per program, which counts one
catalogue after another); `run` is one `cf_count` (or one `cf_batch_count` over several catalogues).

Catalogues follow the recipes of this repository's benchmark: clusters of normally distributed members
around uniform centres (topped up with uniform points to the exact size), uniform boxes, a patch of the
sphere as unit vectors, and a survey cone seen from the origin.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1911_03545_gb300 as cf

DEV = "cuda:0"
# footprints of the angular and the observed catalogues (RA, DEC in degrees, comoving distance)
SPHERE = (0.0, 90.0, -10.0, 30.0)
CONE = (0.0, 90.0, 0.0, 60.0, 300.0, 1000.0)

_ctx = None


def _context():
    """The program's one context, on its current stream."""
    global _ctx
    if _ctx is None:
        _ctx = cf.cf_create(0, torch.cuda.current_stream())
    return _ctx


def _case(name=None, **kw):
    c = {"kind": "r", "auto": True, "n": 0, "n2": 0, "ncat": 1, "f64": False, "periodic": True, "box": 0.0,
         "members": 0, "sigma": 0.0, "rmin": 0.1, "rmax": 20.0, "nbins": 20, "pimax": 0.0, "npi": 0,
         "weighted": False, "ravg": False}
    c.update(kw)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # one small mock or a subsample of one (the smallest size of the scaling sweep): launches and
        # latency are most of the call
        _case("r_10k", n=10_000, box=90.5, members=100, sigma=1.0),
        # the small correctness configuration: uniform float64 positions in a periodic box
        _case("uniform_r_20k_f64", n=20_000, f64=True, box=250.0, rmax=25.0),
        # wp(rp) of a galaxy sample of an odd size
        _case("wp_100k", kind="wp", n=100_003, box=368.4, members=50, sigma=2.0, rmax=25.0, nbins=14, pimax=40.0,
              npi=40),
        # a survey-like sample in float64 without a periodic box, weights and mean separations
        _case("r_200k_f64_wr", n=200_003, f64=True, periodic=False, box=245.6, members=25, sigma=2.0, weighted=True,
              ravg=True),
        # many small mocks counted in one call
        _case("batch_32_rppi", kind="rppi", n=20_000, ncat=32, box=250.0, members=50, sigma=1.0, rmax=20.0, nbins=14,
              pimax=40.0, npi=40),
        # xi(r) of a million clustered points with weights and mean separations: the benchmark's headline
        _case("r_1m_wr", n=1_000_000, box=420.0, members=100, sigma=1.0, weighted=True, ravg=True),
        # the same catalogue to twice the separation, counts only: dense cells (the scaling sweep's Rmax series)
        _case("r_1m_rmax40", n=1_000_000, box=420.0, members=100, sigma=1.0, rmax=40.0),
        # DD(rp, pi) of two million clustered points
        _case("rppi_2m", kind="rppi", n=2_000_000, box=1000.0, members=100, sigma=2.0, rmax=25.0, nbins=14, pimax=40.0,
              npi=40),
        # DD(rp, pi) with weights and mean separations, an odd size
        _case("rppi_700k_wr", kind="rppi", n=700_001, box=704.7, members=100, sigma=2.0, rmax=25.0, nbins=14,
              pimax=40.0, npi=40, weighted=True, ravg=True),
        # DR(rp, pi): data against twice as many randoms, the largest of the benchmark's counts
        _case("rppi_dr_2m_4m", kind="rppi", auto=False, n=2_000_000, n2=4_000_000, box=1000.0, members=100, sigma=2.0,
              rmax=25.0, nbins=14, pimax=40.0, npi=40),
        # w(theta) of a million directions
        _case("theta_1m", kind="theta", n=1_000_000, periodic=False, rmin=0.001, rmax=1.0),
        # DR(rp, pi) of observed galaxies against randoms at ten times their density
        _case("mocks_dr_200k_2m", kind="mocks", auto=False, n=200_000, n2=2_000_000, periodic=False, members=100,
              sigma=2.0, rmin=0.5, rmax=42.0, nbins=14, pimax=42.0, npi=42),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _cost(c):
    """Pairs in reach of each other's cells, about (unordered for an auto-correlation)."""
    n2 = c["n"] if c["auto"] else c["n2"]
    if c["kind"] == "theta":
        density = n2 / _volume(c)
        return 0.5 * c["n"] * density * (3.0 * c["rmax"]) ** 2
    reach = 27.0 * c["rmax"] ** 3
    if c["kind"] in ("rppi", "wp"):
        reach = 27.0 * c["rmax"] ** 2 * c["pimax"]
    elif c["kind"] == "mocks":
        reach = 27.0 * (c["rmax"] ** 2 + c["pimax"] ** 2) ** 1.5
    return (0.5 if c["auto"] else 1.0) * c["ncat"] * c["n"] * n2 * reach / _volume(c)


def draw(rng):
    """One more case: the same kinds, sizes over three decades, densities, reaches, options."""
    kind = rng.choice(["r", "r", "r", "rppi", "rppi", "wp", "theta", "mocks", "batch"])
    n = int(_log_uniform(rng, 5_000, 2_000_000))
    wr = rng.random() < 0.35
    c = _case(kind=kind, n=n)
    if kind == "theta":
        c.update(n=min(n, 1_500_000), periodic=False, rmin=0.001, rmax=round(_log_uniform(rng, 0.3, 2.0), 3),
                 nbins=rng.randint(8, 25))
        limit = 3e9
    elif kind == "mocks":
        n = int(_log_uniform(rng, 5_000, 200_000))
        c.update(auto=False, n=n, n2=n * rng.randint(5, 10) + rng.randint(0, 9), periodic=False, members=100,
                 sigma=round(rng.uniform(1.0, 3.0), 2), rmin=0.5, rmax=round(rng.uniform(20.0, 42.0), 1), nbins=14,
                 pimax=40.0, npi=40)
        limit = 6e9
    elif kind == "batch":
        c.update(kind="rppi", n=int(_log_uniform(rng, 2_000, 40_000)), ncat=rng.randint(8, 32), box=250.0, members=50,
                 sigma=1.0, rmax=round(rng.uniform(15.0, 25.0), 1), nbins=14, pimax=40.0, npi=40)
        limit = 2e9
    else:
        density = (0.0135 if kind == "r" else 0.002) * _log_uniform(rng, 0.4, 2.0)
        clustered = rng.random() < 0.75
        c.update(box=round((n / density) ** (1.0 / 3.0), 1), members=rng.randint(20, 120) if clustered else 0,
                 sigma=round(rng.uniform(1.0, 3.0), 2) if clustered else 0.0, f64=rng.random() < 0.25,
                 periodic=rng.random() < 0.75, weighted=wr, ravg=wr, nbins=rng.randint(8, 25))
        c["rmax"] = round(rng.uniform(10.0, 30.0), 1)
        if kind != "r":
            c.update(pimax=40.0, npi=40)
            if kind == "rppi" and rng.random() < 0.4:
                c.update(auto=False, n2=2 * n + rng.randint(0, 99))
        limit = 1.5e9 if wr else 4e9
    while _cost(c) > limit:
        for k in ("n", "n2"):
            c[k] = int(c[k] * 0.8)
    if c["box"] and kind != "batch" and c["n"] < n:
        c["box"] = round(c["box"] * (c["n"] / n) ** (1.0 / 3.0), 1)
    return c


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _uniform(g, lo, hi, n):
    return torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * (hi - lo) + lo


def _spread(g, centres, n, members, sigma):
    """n points: `members` normal ones around each centre in turn (the centres given are enough)."""
    idx = torch.arange(n, device=DEV) // max(1, members)
    return [c[idx] + sigma * torch.randn(n, generator=g, device=DEV, dtype=torch.float64) for c in centres]


def _in_box(g, c, n, clustered):
    L = c["box"]
    if not clustered or not c["members"]:
        p = [_uniform(g, 0.0, L, n) for _ in range(3)]
    else:
        m = c["members"]
        nc = n // m
        p = [_uniform(g, 0.0, L, max(1, nc)) for _ in range(3)]
        q = _spread(g, p, nc * m, m, c["sigma"])
        rest = n - nc * m
        p = [torch.cat([torch.remainder(a, L), _uniform(g, 0.0, L, rest)]) for a in q]
    return p


def _on_sphere(g, n):
    ra = _uniform(g, math.radians(SPHERE[0]), math.radians(SPHERE[1]), n)
    sd = _uniform(g, math.sin(math.radians(SPHERE[2])), math.sin(math.radians(SPHERE[3])), n)
    cd = torch.sqrt(1.0 - sd * sd)
    return [cd * torch.cos(ra), cd * torch.sin(ra), sd]


def _in_cone(g, c, n, clustered):
    m = c["members"] if clustered else 1
    nc = -(-n // m)
    ra = _uniform(g, math.radians(CONE[0]), math.radians(CONE[1]), nc)
    sd = _uniform(g, math.sin(math.radians(CONE[2])), math.sin(math.radians(CONE[3])), nc)
    cd = torch.sqrt(1.0 - sd * sd)
    d = _uniform(g, CONE[4] ** 3, CONE[5] ** 3, nc) ** (1.0 / 3.0)
    p = [d * cd * torch.cos(ra), d * cd * torch.sin(ra), d * sd]
    return _spread(g, p, n, m, c["sigma"]) if clustered and m > 1 else p


def _set(g, c, n, clustered):
    """[x, y, z(, w)] of one point set in the case's type, in a catalogue's arbitrary order."""
    if c["kind"] == "theta":
        p = _on_sphere(g, n)
    elif c["kind"] == "mocks":
        p = _in_cone(g, c, n, clustered)
    else:
        p = _in_box(g, c, n, clustered)
    dt = torch.float64 if c["f64"] else torch.float32
    p = [a.to(dt) for a in p]
    if c["box"]:
        p = [torch.where(a >= c["box"], torch.zeros_like(a), a) for a in p]     # a value rounded up to the side
    if c["weighted"]:
        p.append(_uniform(g, 0.5, 1.5, n).to(dt))
    return [a.contiguous() for a in p]


def _sizes(c):
    """Sizes of a batch's catalogues: from a twentieth of n to n, evenly in the logarithm."""
    k = c["ncat"]
    return [int(c["n"] * 20.0 ** (-i / max(1, k - 1))) for i in range(k)] if k > 1 else [c["n"]]


def _sets(c, seed):
    g = _gen(seed)
    s = [_set(g, c, n, True) for n in _sizes(c)]
    if not c["auto"]:
        s.append(_set(g, c, c["n2"], False))
    return s


def _edges(c):
    e = np.geomspace(c["rmin"], c["rmax"], c["nbins"] + 1)
    e[0], e[-1] = c["rmin"], c["rmax"]
    return e


def prepare(case, seed):
    ctx = _context()
    p = cf.params(kind=case["kind"], edges=_edges(case), autocorr=case["auto"], periodic=case["periodic"],
                  box=case["box"] if case["periodic"] else 0.0, pimax=case["pimax"], npibins=case["npi"],
                  ravg=case["ravg"], weighted=case["weighted"])
    pts = [cf.points(*s) for s in _sets(case, seed)]
    return {"ctx": ctx, "params": p, "points": pts, "batch": case["ncat"] > 1, "auto": case["auto"]}


def run(state):
    if state["batch"]:
        return cf.cf_batch_count(state["ctx"], state["params"], state["points"])
    return cf.cf_count(state["ctx"], state["params"], state["points"][0], None if state["auto"] else state["points"][1])


# ---------------------------------------------------------------------------------------------
# the work of a pass, and its result in 64 bits
# ---------------------------------------------------------------------------------------------
def _volume(c):
    if c["kind"] == "theta":        # square degrees
        s = math.sin(math.radians(SPHERE[3])) - math.sin(math.radians(SPHERE[2]))
        return (SPHERE[1] - SPHERE[0]) * math.degrees(s)
    if c["kind"] == "mocks":
        s = math.sin(math.radians(CONE[3])) - math.sin(math.radians(CONE[2]))
        return math.radians(CONE[1] - CONE[0]) * s * (CONE[5] ** 3 - CONE[4] ** 3) / 3.0
    return c["box"] ** 3


def work(case):
    """bytes: every coordinate and weight once, every result once.  flops: the separation of each pair
    within the largest edge (eight operations; twenty for observed positions): uniform density plus,
    for an auto-correlation, the clusters' own pairs."""
    c = case
    size = (8 if c["f64"] else 4) * (4 if c["weighted"] else 3)
    slots = c["nbins"] * (c["npi"] if c["kind"] in ("rppi", "mocks") else 1)
    if c["kind"] == "theta":
        reach = math.pi * c["rmax"] ** 2
    elif c["kind"] == "r":
        reach = 4.0 / 3.0 * math.pi * c["rmax"] ** 3
    else:
        reach = 2.0 * math.pi * c["rmax"] ** 2 * c["pimax"]
    pairs = 0.0
    for n in _sizes(c):
        n2 = n if c["auto"] else c["n2"]
        pairs += (0.5 if c["auto"] else 1.0) * n * n2 * reach / _volume(c)
        if c["auto"] and c["members"] and c["kind"] != "theta":
            pairs += 0.5 * n * (c["members"] - 1)
    points = sum(_sizes(c)) + (0 if c["auto"] else c["n2"])
    out = 8 * slots * (2 + int(c["ravg"])) * c["ncat"]
    return {"bytes": float(points * size + out), "flops": pairs * (20.0 if c["kind"] == "mocks" else 8.0)}


def _min_image(d, L):
    d = torch.where(d > L / 2, d - L, d)
    return torch.where(d <= -L / 2, d + L, d)


def _columns(x, y, lo, side, ncol):
    """Points sorted by (x, y) column, and each column's start."""
    ix = torch.clamp(((x - lo[0]) / side[0]).floor().long(), 0, ncol[0] - 1)
    iy = torch.clamp(((y - lo[1]) / side[1]).floor().long(), 0, ncol[1] - 1)
    key = ix * ncol[1] + iy
    order = torch.argsort(key)
    start = torch.searchsorted(key[order], torch.arange(ncol[0] * ncol[1] + 1, device=x.device))
    return order, start.tolist()


def _exact_pairs(c, s1, s2):
    """npairs, sum of weights and of weighted separations per slot over ordered pairs, in float64."""
    kind, auto, nb, npi = c["kind"], s2 is None, c["nbins"], max(1, c["npi"])
    nslot = nb * (npi if kind in ("rppi", "mocks") else 1)
    e = torch.from_numpy(_edges(c)).to(DEV)
    if kind == "theta":
        e = 2.0 * torch.sin(e * (math.pi / 360.0))
    e2 = e * e
    p_edges = torch.arange(npi + 1, device=DEV, dtype=torch.float64) * (c["pimax"] / npi if c["pimax"] else 1.0)
    reach = float(e[-1])
    if kind == "mocks":
        reach = math.sqrt(c["rmax"] ** 2 + c["pimax"] ** 2)
    a = [t.double() for t in s1]
    b = a if auto else [t.double() for t in s2]
    L = c["box"] if c["periodic"] else 0.0
    lo, side, ncol = [], [], []
    for k in range(2):
        l0, l1 = (0.0, L) if L else (float(min(a[k].min(), b[k].min())), float(max(a[k].max(), b[k].max())))
        n = max(1, min(256, int((l1 - l0) / (reach * 1.0001)))) if l1 > l0 else 1
        lo.append(l0)
        ncol.append(n)
        side.append((l1 - l0) / n if l1 > l0 else 1.0)
    oa, sa = _columns(a[0], a[1], lo, side, ncol)
    ob, sb = _columns(b[0], b[1], lo, side, ncol)
    a, ida = [t[oa] for t in a], oa
    b, idb = [t[ob] for t in b], ob
    spread = 64         # copies of the histogram: fewer additions to one address
    cnt = torch.zeros(nslot * spread, dtype=torch.int64, device=DEV)
    ws = torch.zeros(nslot * spread, dtype=torch.float64, device=DEV)
    rs = torch.zeros_like(ws)
    weighted, ravg = c["weighted"], c["ravg"]

    def near(i, n):
        w = [i - 1, i, i + 1]
        return sorted({k % n for k in w}) if L else [k for k in w if 0 <= k < n]

    for cx in range(ncol[0]):
        for cy in range(ncol[1]):
            i0, i1 = sa[cx * ncol[1] + cy], sa[cx * ncol[1] + cy + 1]
            if i0 == i1:
                continue
            js = [(sb[kx * ncol[1] + ky], sb[kx * ncol[1] + ky + 1]) for kx in near(cx, ncol[0]) for ky in near(cy, ncol[1])]
            J = torch.cat([torch.arange(u, v, device=DEV) for u, v in js])
            if not J.numel():
                continue
            B = [t[J] for t in b]
            step = max(1, 40_000_000 // J.numel())
            for i in range(i0, i1, step):
                sl = slice(i, min(i1, i + step))
                A = [t[sl] for t in a]
                d = [A[k][:, None] - B[k][None, :] for k in range(3)]
                if L:
                    d = [_min_image(t, L) for t in d]
                xy2 = d[0] * d[0] + d[1] * d[1]
                r2 = xy2 + d[2] * d[2]
                if kind in ("r", "theta"):
                    hit = (r2 >= e2[0]) & (r2 < e2[-1])
                elif kind == "mocks":
                    hit = r2 < reach * reach * 1.000001
                else:
                    hit = (xy2 >= e2[0]) & (xy2 < e2[-1]) & (d[2].abs() < c["pimax"])
                if auto:
                    hit &= ida[sl][:, None] != idb[J][None, :]
                if kind == "mocks":
                    ii, jj = hit.nonzero(as_tuple=True)
                    v1, v2 = [A[k][ii] for k in range(3)], [B[k][jj] for k in range(3)]
                    s = [p - q for p, q in zip(v1, v2)]
                    m = [0.5 * (p + q) for p, q in zip(v1, v2)]
                    dot = lambda p, q: (p[0] * q[0] + p[1] * q[1]) + p[2] * q[2]  # noqa: E731
                    sl_, ll = dot(s, m), dot(m, m)
                    q2 = sl_ * sl_ / ll
                    v2_ = torch.clamp(dot(s, s) - q2, min=0.0)
                    ok = (q2 < p_edges[-1] ** 2) & (v2_ >= e2[0]) & (v2_ < e2[-1])
                    val, q2, ii, jj = v2_[ok], q2[ok], ii[ok], jj[ok]
                    slot = (torch.bucketize(val, e2, right=True) - 1) * npi + torch.bucketize(q2, p_edges ** 2, right=True) - 1
                else:
                    val = (r2 if kind in ("r", "theta") else xy2)[hit]
                    slot = torch.bucketize(val, e2, right=True) - 1
                    if kind == "rppi":
                        slot = slot * npi + torch.bucketize(d[2].abs()[hit], p_edges, right=True) - 1
                    if weighted:
                        ii, jj = hit.nonzero(as_tuple=True)
                slot = slot * spread + torch.arange(slot.numel(), device=DEV) % spread
                cnt += torch.bincount(slot, minlength=cnt.numel())
                if weighted or ravg:
                    w = A[3][ii] * B[3][jj] if weighted else torch.ones_like(val)
                    r = torch.sqrt(val)
                    if kind == "theta":
                        r = 2.0 * torch.asin(0.5 * r) * (180.0 / math.pi)
                    ws += torch.bincount(slot, weights=w, minlength=ws.numel())
                    rs += torch.bincount(slot, weights=w * r, minlength=rs.numel())
    fold = lambda t: t.view(nslot, spread).sum(1)  # noqa: E731
    return fold(cnt), fold(ws), fold(rs)


def _exact_one(c, s1, s2):
    cnt, ws, rs = (t.cpu().numpy() for t in _exact_pairs(c, s1, s2))
    shape = (c["nbins"], c["npi"]) if c["kind"] in ("rppi", "mocks") else (c["nbins"],)
    wsum = ws if c["weighted"] else cnt.astype(np.float64)
    out = {"npairs": cnt.astype(np.uint64).reshape(shape), "wsum": wsum.reshape(shape)}
    if c["ravg"]:
        out["ravg"] = np.where(wsum > 0, rs / np.where(wsum > 0, wsum, 1.0), 0.0).reshape(shape)
    if c["kind"] == "wp":
        wp = np.zeros(c["nbins"])
        if c["periodic"] and c["auto"]:
            n = float(c["n"])
            e = _edges(c)
            rr = n * (n - 1.0) / c["box"] ** 3 * math.pi * (e[1:] ** 2 - e[:-1] ** 2)
            wp = cnt.astype(np.float64) / rr - 2.0 * c["pimax"]
        out["wp"] = wp
    return out


def exact(case, seed):
    s = _sets(case, seed)
    if case["ncat"] > 1:
        return [_exact_one(case, t, None) for t in s]
    return _exact_one(case, s[0], None if case["auto"] else s[1])
