"""The cell-by-cell layer vote's bounds (k_vote_rows.cu), on the CPU, with hits
placed where they matter.

That path decides a hit's bin in a row by comparing -s (float32, s = x sin phi0
- y cos phi0) with S(rho, d0) at the bins' edges, and takes the hits of a layer
in the order of the hit index.  Two statements carry its exactness:

 - a hit whose -s lies more than eps beyond S at an edge has its root (of the
   float64 definition) on that side of the edge, eps being the bound on S's
   rounding, the layer's spread in r^2 and the float32 s;
 - in the index's order -s is never out of order by more than eta: the spread
   in r, atan2f's 3 ulp at a cell's boundary, the rounding of s.

Here hits are put within a few eps of an edge (the azimuth solved for, then
perturbed) and within a few ulp of the cells' boundaries, on layers of equal
radius and on layers with as large a spread as the kernel admits (eps up to a
twentieth of a bin).  The kernel's float32 steps are restated with numpy, the
reciprocal pushed to both ends of its error and atan2f by up to 3 ulp either
way.  An eighth of eps fails on layers of large spread (whose error is what the
bound allows for it), a 64th on layers of equal radius (sums of worst cases,
taken four times), and a third of eta on both.
"""
import numpy as np
import pytest

from test_aform_bound import F32, GEOMS, U, fma32
from test_crossing_bound import dot2

EPS32, SAFE = F32(U), F32(4.0)
AZ = 256
WORDS = {"single_64": 2, "event100_256": 8, "pileup_512": 4}   # rows of a tile, in words


def tables(geom):
    NR, ND, NP, rho_max, dh = geom
    phi = (2 * np.arange(NP) + 1 - NP) * (np.pi / NP)
    sn, cs = np.sin(phi), np.cos(phi)
    return phi, sn, cs, sn.astype(F32), cs.astype(F32), (sn - sn.astype(F32)).astype(F32), (
        cs - cs.astype(F32)).astype(F32)


def radius32(x, y):
    return np.sqrt(fma32(x, x, (y * y).astype(F32)).astype(np.float64)).astype(F32)


def layer_bounds(geom, rmin, rmax, i0, nrow):
    """The rows [vA, vB] (in the band) that a layer votes cell by cell, its eps
    without the order's slack and the slack eta, or None where the kernel goes
    hit by hit."""
    NR, ND, NP, rho_max, dh = geom
    delta, drho = 2.0 * dh / ND, 2.0 * rho_max / NR
    dext = F32((ND / 2 + 1.0) * delta * 1.0001 + 0.01)
    tc = 0.5 * (NR - 1) - i0
    rv = min(1.95 / (dext + np.sqrt(max(1.95 * rmax * rmax - 0.95 * dext * dext, 0.0))),
             0.95 / dext) * 0.9999
    vA, vB = max(int(np.ceil(tc - rv / drho)), 0), min(int(np.floor(tc + rv / drho)), nrow - 1)
    if vB - vA < 32:
        return None
    rho = ((2 * (i0 + np.array([vA, vB])) + 1 - NR) * (rho_max / NR)).astype(F32)
    rt = F32(np.abs(rho).max())
    iu = F32(0.5) / (F32(1.0) - rt * dext)
    eE = EPS32 * (iu * (F32(8.0) * rt * (rmax * rmax + dext * dext) + F32(12.0) * dext) + F32(4.0) * rmax)
    eR2 = rt * iu * (F32(0.51) * (rmax - rmin) * (rmax + rmin) + F32(8.0) * EPS32 * rmax * rmax)
    hit = F32(1.25) * EPS32 * rmax + F32(2e-13) * rmax
    eps, eta = SAFE * (eE + eR2 + hit), F32(1.01) * (rmax - rmin) + F32(2.3e-6) * rmax
    return (vA, vB, np.float64(eps), np.float64(eta)) if eps + eta <= 0.05 * delta else None


def largest_spread(geom, r, i0, nrow):
    """Half the relative spread of a layer's radii that the kernel still takes."""
    lo, hi = 0.0, 0.05
    for _ in range(40):
        mid = 0.5 * (lo + hi)
        ok = layer_bounds(geom, F32(r * (1 - mid)), F32(r * (1 + mid)), i0, nrow) is not None
        lo, hi = (mid, hi) if ok else (lo, mid)
    return lo


def edge_sides(name, spread, n, seed, scale=1.0, rcp_err=0.0):
    """Hits within five eps of a random (row, edge): (sides that the bound,
    scaled, decides; those that it decides wrongly; those within it)."""
    geom, _ = GEOMS[name]
    NR, ND, NP, rho_max, dh = geom
    delta, off = 2.0 * dh / ND, ND / 2 + 0.5
    phi, sn64, cs64, sn, cs, snl, csl = tables(geom)
    rng = np.random.default_rng(seed)
    decided = wrong = near = 0
    for l in range(10):
        r0 = 4.0 + l * 106.0 / 9.0
        nrow = min(32 * WORDS[name], NR)
        for i0 in range(0, NR, nrow):
            half = spread * largest_spread(geom, r0, i0, nrow) if spread else 0.0
            b = layer_bounds(geom, F32(r0 * (1 - half)), F32(r0 * (1 + half)), i0, nrow)
            if b is None:
                continue
            k, i = rng.integers(0, NP, n), i0 + rng.integers(b[0], b[1] + 1, n)
            j = rng.integers(0, ND + 1, n)
            r = r0 * (1.0 + half * rng.choice([-1.0, 1.0, 0.0], n))
            rho = (2 * i + 1 - NR) * (rho_max / NR)
            d = (j - off) * delta
            s = -(rho * (d * d + r * r) + 2 * d) / (2 * (1 + rho * d))
            s += rng.uniform(-5, 5, n) * b[2]
            ok = np.abs(s) < 0.999 * r
            s, r, rho, d, i, j, k = (a[ok] for a in (s, r, rho, d, i, j, k))
            az = phi[k] - np.arcsin(s / r)
            x, y = (r * np.cos(az)).astype(F32), (r * np.sin(az)).astype(F32)
            rr = radius32(x, y)
            rmin, rmax = rr.min(), rr.max()
            b = layer_bounds(geom, rmin, rmax, i0, nrow)
            if b is None:
                continue
            eps = b[2] * scale
            r2 = F32(0.5) * fma32(rmin, rmin, F32(rmax * rmax))
            s32 = dot2(x, sn[k], snl[k], -y, cs[k], csl[k])
            c32 = dot2(x, cs[k], csl[k], y, sn[k], snl[k])
            d32 = ((j - off).astype(F32) * F32(delta)).astype(F32)
            r32 = rho.astype(F32)
            num = fma32(fma32(r32, d32, F32(2.0)), d32, (r32 * r2).astype(F32))
            rc = (1.0 / fma32((F32(2.0) * r32).astype(F32), d32, F32(2.0)).astype(np.float64) *
                  (1.0 + rcp_err)).astype(F32)
            v, sig = (num * rc).astype(F32).astype(np.float64), -s32.astype(np.float64)
            # the float64 definition's root
            X, Y = x.astype(np.float64), y.astype(np.float64)
            sd, cd = X * sn64[k] - Y * cs64[k], X * cs64[k] + Y * sn64[k]
            bq, D = 1.0 + rho * sd, 1.0 - (rho * cd) ** 2
            q = -(bq + np.where(bq >= 0, 1.0, -1.0) * np.sqrt(D))
            u = np.where(bq >= 0, (rho * (X * X + Y * Y) + 2.0 * sd) / q, q / rho) / delta + off
            ok = c32 > F32(12 * U) * (np.abs(x) + np.abs(y))
            above, below = ok & (sig > v + eps), ok & (sig < v - eps)
            decided += int((above | below).sum())
            near += int((ok & ~above & ~below).sum())
            wrong += int((above & ~(u >= j)).sum() + (below & ~(u < j)).sum())
    return decided, wrong, near


@pytest.mark.parametrize("spread", [0.0, 0.5, 0.98])
@pytest.mark.parametrize("name", sorted(WORDS))
def test_a_hit_beyond_the_bound_is_on_that_side(name, spread):
    for err in (-2 ** -23.0, 2 ** -23.0):
        decided, wrong, near = edge_sides(name, spread, 20000, 11, rcp_err=err)
        assert wrong == 0
        assert decided > 50000 and near > 5000


@pytest.mark.parametrize("spread,part", [(0.0, 64), (0.98, 8)])
@pytest.mark.parametrize("name", sorted(WORDS))
def test_a_fraction_of_the_bound_fails(name, spread, part):
    assert edge_sides(name, spread, 40000, 11, scale=1 / part, rcp_err=2 ** -23.0)[1] > 0


def out_of_order(name, spread, n, seed):
    """The most by which -s is out of order in the index's order of a layer, over
    eta: hits within a few ulp of the cells' boundaries and in between."""
    geom, _ = GEOMS[name]
    NR, ND, NP, rho_max, dh = geom
    phi, sn64, cs64, sn, cs, snl, csl = tables(geom)
    rng = np.random.default_rng(seed)
    worst = 0.0
    for r0 in (4.0, 27.0, 62.0, 110.0):
        half = spread * largest_spread(geom, r0, 0, min(32 * WORDS[name], NR)) if spread else 0.0
        edge = rng.integers(0, AZ, n) * (2 * np.pi / AZ) - np.pi
        az = edge + np.where(rng.random(n) < 0.7, rng.normal(0, 6e-7, n), rng.uniform(0, 0.02, n))
        r = r0 * (1.0 + half * rng.choice([-1.0, 1.0], n))
        x, y = (r * np.cos(az)).astype(F32), (r * np.sin(az)).astype(F32)
        rr = radius32(x, y)
        rmin, rmax = rr.min(), rr.max()
        X, Y = x.astype(np.float64), y.astype(np.float64)
        a = np.arctan2(Y, X)
        a32 = a.astype(F32)   # atan2f: up to 3 ulp either way
        a32 = (a32 + rng.integers(-3, 4, n) * np.spacing(np.abs(a32))).astype(F32)
        cell = np.clip(np.floor(((a32 + F32(3.14159265)).astype(F32) *
                                 F32(AZ / F32(6.28318531))).astype(F32)).astype(int), 0, AZ - 1)
        eta = np.float64(F32(1.01) * (rmax - rmin) + F32(2.3e-6) * rmax)
        for k in rng.integers(0, NP, 12):
            # cells in azimuth order from half a turn before the column's; within a
            # cell the exact order
            first = int(np.floor((phi[k] - np.pi + np.pi) * AZ / (2 * np.pi)))
            turn = (cell - first) % AZ
            near = np.mod(a - phi[k] + np.pi, 2 * np.pi)
            at = np.lexsort((near, turn))
            kk = np.full(n, k)
            s = dot2(x, sn[kk], snl[kk], -y, cs[kk], csl[kk])
            c = dot2(x, cs[kk], csl[kk], y, sn[kk], snl[kk])
            sig = -s.astype(np.float64)[at][(c > F32(12 * U) * (np.abs(x) + np.abs(y)))[at]]
            worst = max(worst, float((np.maximum.accumulate(sig) - sig).max() / eta))
    return worst


@pytest.mark.parametrize("spread", [0.0, 0.5, 0.98])
@pytest.mark.parametrize("name", sorted(WORDS))
def test_the_index_is_in_order_within_the_slack(name, spread):
    worst = out_of_order(name, spread, 20000, 5)
    assert 1 / 3 < worst <= 1.0
