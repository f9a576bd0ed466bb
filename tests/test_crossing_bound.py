"""The distinct-layer vote's edge crossings and their error bound, checked on
the CPU.

k_vote_rows.cu votes a run of rows per d0 bin: along a column a hit's root
falls with rho, and edge d0 = d is crossed at the row coordinate
t = tc - kr w / (w^2 + c^2), w = d + s, in float32 with a bound eps.  The rows
up to floor(t - eps) have their root at or above the edge and the rows from
floor(t + eps) + 1 on below it, by the float64 definition; the rows between
are evaluated by the definition itself.  These tests restate the kernel's
float32 steps with numpy (each operation rounded once, fused ones formed in
float64 and rounded once, the reciprocal pushed to both ends of its error
bound) and check both statements on the geometries of every workload and of
the extreme-geometry GPU tests.  A bound a fortieth as large fails.
"""
import zlib

import numpy as np
import pytest

from test_aform_bound import F32, GEOMS, U, fma32, items

EPS32 = F32(U)


def dot2(a, p, plo, b, q, qlo):
    """a p + b q with the tables' remainders and the rounding errors carried."""
    u = (a * p).astype(F32)
    eu = fma32(a, p, -u)
    v = (b * q).astype(F32)
    ev = fma32(b, q, -v)
    h = (u + v).astype(F32)
    z = (h - u).astype(F32)
    lo = ((u - (h - z).astype(F32)).astype(F32) + (v - z).astype(F32)).astype(F32)
    low = fma32(a, plo, (b * qlo).astype(F32))
    return (h + (lo + ((eu + ev).astype(F32) + low).astype(F32)).astype(F32)).astype(F32)


def crossings(geom, x, y, k, t0, TR, rcp_err=0.0, scale=1.0, seed=0):
    """For each eligible item, the band's rows and one edge its curve can
    cross there: (lo, hi) rows and the definition's coordinates around them."""
    NR, ND, NP, rmax, dh = geom
    delta = 2.0 * dh / ND
    off = ND / 2 + 0.5
    drho = 2.0 * rmax / NR
    invd, off_f, delta_f = F32(1.0 / delta), F32(off), F32(delta)
    kr, drho_f = F32(NR / rmax), F32(drho)
    rho64 = (2 * np.arange(NR) + 1 - NR) * (rmax / NR)
    phi = (2 * np.arange(NP) + 1 - NP) * (np.pi / NP)
    sn64, cs64 = np.sin(phi), np.cos(phi)
    sn, cs = sn64.astype(F32), cs64.astype(F32)
    snl, csl = (sn64 - sn).astype(F32), (cs64 - cs).astype(F32)
    s = dot2(x, sn[k], snl[k], -y, cs[k], csl[k])
    c = dot2(x, cs[k], csl[k], y, sn[k], snl[k])
    R1 = np.abs(x) + np.abs(y)
    eR = F32(4e-7) * R1
    last = np.minimum(t0 + TR - 1, NR - 1)
    # rows where the first root is the only one (the kernel's rok)
    dext = F32((off + 0.5) * delta * 1.0001 + 0.01)
    with np.errstate(divide="ignore", invalid="ignore"):
        sp = (np.abs(s) + eR) * F32(1.000004) + F32(0.0102)
        cp = (c + eR) * F32(1.000004) + F32(0.0502)
        rok = np.maximum(1 / (dext + sp), 1 / np.sqrt(cp * cp + dext * dext))
        rok = np.minimum(rok, F32(0.985) / np.maximum(c, np.abs(s) + eR)) * F32(0.9997)
        half = (NR - 1) / 2.0
        ra = np.maximum(np.ceil(half - rok / drho), t0)
        rb = np.minimum(np.floor(half + rok / drho), last)
        ok = (ra <= rb) & (c > F32(12 * U) * R1) & (c >= F32(4e-4) * R1)
        ra, rb = np.where(ok, ra, 0).astype(int), np.where(ok, rb, 0).astype(int)
        rt = (np.maximum(np.abs(rho64[ra]), np.abs(rho64[rb])) * 1.0001).astype(F32)
        slope = F32(0.5) * drho_f * c * c * invd
        # walk_eps
        eS = F32(1.25) * EPS32 * np.abs(s) + F32(1e-13) * R1
        eC = F32(1.25) * EPS32 * c + F32(1e-13) * R1
        ic = F32(1.001) / c
        dmax = F32(off * delta + 0.01)
        eps = F32(4.0) * (kr * ic * ic * (EPS32 * (dmax + c) + eS + F32(1e-13) * R1) +
                          F32(NR) * (2 * eC * ic + 9 * EPS32))
        ok &= (slope <= 0.5) & (c * (2 * drho_f + rt) <= 0.97)
        ok &= np.where(slope <= 1 / 64, eps <= 8.0, (eps <= 0.25) & (c > F32(2.4e-7) * kr))
    sel = np.nonzero(ok)[0]
    x, y, k, s, c, ra, rb, eps = (a[sel] for a in (x, y, k, s, c, ra, rb, eps))
    eps = eps * F32(scale)
    X, Y = x.astype(np.float64), y.astype(np.float64)

    def u64(row):
        rho = rho64[row]
        sd = X * sn64[k] - Y * cs64[k]
        cd = X * cs64[k] + Y * sn64[k]
        q = -(1.0 + rho * sd + np.sqrt(1.0 - (rho * cd) ** 2))
        return ((rho * (X * X + Y * Y) + 2.0 * sd) / q) / delta + off

    # an edge between the coordinates of the window's ends (clipped to the axis)
    rng = np.random.default_rng(seed)
    hi_e = np.minimum(np.floor(u64(ra)), ND)
    lo_e = np.maximum(np.floor(u64(rb)) + 1, 0)
    e = np.floor(lo_e + rng.random(sel.size) * (hi_e - lo_e + 1))
    has = hi_e >= lo_e
    c2 = (c * c).astype(F32)
    w = np.maximum(fma32((e - off).astype(F32), delta_f, s), -c)
    rc = (1.0 / fma32(w, w, c2).astype(np.float64) * (1.0 + rcp_err)).astype(F32)
    t = fma32(-(kr * w).astype(F32), rc, F32(half)).astype(np.float64)
    lo, hi = np.floor(t - eps).astype(int), np.floor(t + eps).astype(int)
    above = has & (lo >= ra)           # row min(lo, rb) has its root at or above e
    below = has & (hi < rb)            # row max(hi + 1, ra) below
    bad = above & ~(u64(np.clip(lo, ra, rb)) >= e)
    bad |= below & ~(u64(np.clip(hi + 1, ra, rb)) < e)
    return int(has.sum()), int(bad.sum())


@pytest.mark.parametrize("TR", [32, 256])
@pytest.mark.parametrize("name", sorted(GEOMS))
def test_rows_on_both_sides_of_a_crossing(name, TR):
    geom, rr = GEOMS[name]
    x, y, k, t0, _, _ = items(geom, rr, 120000, seed=zlib.crc32(name.encode()) & 0xfff, TR=TR)
    n = 0
    for err in (-2 ** -23.0, 2 ** -23.0):
        n, bad = crossings(geom, x, y, k, t0, TR, rcp_err=err)
        assert bad == 0
    if name not in ("straight_far", "fine_bins_far_hits"):   # curves across many bins per row there
        assert n > 1000, f"too few crossings ({n})"


def test_bound_has_teeth():
    """A fortieth of the bound is exceeded on the 10k-hit geometry."""
    geom, rr = GEOMS["event100_256"]
    x, y, k, t0, _, _ = items(geom, rr, 1000000, seed=5, TR=256)
    n, bad = crossings(geom, x, y, k, t0, 256, rcp_err=2 ** -23.0, scale=1 / 40)
    assert n > 100000 and bad > 0


# ------------------------------------------------------------ cell by cell
def cell_edges(geom, radii, n, seed, scale=1.0, rcp_err=0.0):
    """Random hits of exact layers against random (row, edge)s of random
    columns near their roots: (checked, wrong sides)."""
    NR, ND, NP, rmax_, dh = geom
    delta = 2.0 * dh / ND
    off = ND / 2 + 0.5
    rng = np.random.default_rng(seed)
    rho64 = (2 * np.arange(NR) + 1 - NR) * (rmax_ / NR)
    phi = (2 * np.arange(NP) + 1 - NP) * (np.pi / NP)
    sn64, cs64 = np.sin(phi), np.cos(phi)
    sn, cs = sn64.astype(F32), cs64.astype(F32)
    snl, csl = (sn64 - sn).astype(F32), (cs64 - cs).astype(F32)
    dext = F32((off + 0.5) * delta * 1.0001 + 0.01)
    checked = wrong = 0
    for r in radii:
        ph = rng.uniform(-np.pi, np.pi, n)
        x, y = (r * np.cos(ph)).astype(F32), (r * np.sin(ph)).astype(F32)
        rr = np.sqrt(fma32(x, x, (y * y).astype(F32)).astype(np.float64)).astype(F32)
        rmin, rmax = rr.min(), rr.max()
        rv = min(1.95 / (dext + np.sqrt(max(1.95 * rmax * rmax - 0.95 * dext * dext, 0.0))),
                 0.95 / dext) * 0.9999
        half = (NR - 1) / 2.0
        drho = 2.0 * rmax_ / NR
        vA, vB = max(int(np.ceil(half - rv / drho)), 0), min(int(np.floor(half + rv / drho)), NR - 1)
        if vB <= vA:
            continue
        rt = F32(max(abs(rho64[vA]), abs(rho64[vB])))
        iu = F32(0.5) / (F32(1.0) - rt * dext)
        r2 = F32(0.5) * fma32(rmin, rmin, F32(rmax * rmax))
        eE = EPS32 * (iu * (8 * rt * (rmax * rmax + dext * dext) + 12 * dext) + 4 * rmax)
        eR2 = rt * iu * (F32(0.51) * (rmax - rmin) * (rmax + rmin) + 8 * EPS32 * rmax * rmax)
        hit = F32(1.25) * EPS32 * rmax + F32(2e-13) * rmax
        eps = np.float64(4.0 * (eE + eR2 + hit) * scale)   # (without the order's slack)
        k = rng.integers(0, NP, n)
        i = rng.integers(vA, vB + 1, n)
        s = dot2(x, sn[k], snl[k], -y, cs[k], csl[k])
        c = dot2(x, cs[k], csl[k], y, sn[k], snl[k])
        rho = rho64[i]
        X, Y = x.astype(np.float64), y.astype(np.float64)
        sd, cd = X * sn64[k] - Y * cs64[k], X * cs64[k] + Y * sn64[k]
        b = 1.0 + rho * sd
        D = 1.0 - (rho * cd) ** 2
        ok = (c > F32(12 * U) * (np.abs(x) + np.abs(y))) & (D > 0)
        with np.errstate(invalid="ignore", divide="ignore"):
            q = -(b + np.where(b >= 0, 1.0, -1.0) * np.sqrt(D))
            root = np.where(b >= 0, (rho * (X * X + Y * Y) + 2.0 * sd) / q, q / rho)
            u = root / delta + off
        ok &= (u > -3) & (u < ND + 3)
        j = np.clip(np.floor(np.where(ok, u, 0)) + rng.integers(0, 2, n), 0, ND)
        d = ((j - off).astype(F32) * F32(delta)).astype(F32)
        r32 = rho.astype(F32)
        num = fma32(fma32(r32, d, F32(2.0)), d, (r32 * r2).astype(F32))
        rc = (1.0 / fma32((F32(2.0) * r32).astype(F32), d, F32(2.0)).astype(np.float64) *
              (1.0 + rcp_err)).astype(F32)
        v = (num * rc).astype(F32).astype(np.float64)
        sig = -s.astype(np.float64)
        checked += int(ok.sum())
        wrong += int((ok & (sig > v + eps) & ~(u >= j)).sum())
        wrong += int((ok & (sig < v - eps) & ~(u < j)).sum())
    return checked, wrong


@pytest.mark.parametrize("name", ["single_64", "event100_256", "pileup_512"])
def test_side_of_an_edge_by_s(name):
    """A hit's -s beyond the bound of S(rho, d0 edge) puts its root on that
    side of the edge."""
    geom, _ = GEOMS[name]
    radii = [4.0 + l * 106.0 / 9.0 for l in range(10)]
    for err in (-2 ** -23.0, 2 ** -23.0):
        n, bad = cell_edges(geom, radii, 40000, seed=3, rcp_err=err)
        assert n > 20000 and bad == 0

