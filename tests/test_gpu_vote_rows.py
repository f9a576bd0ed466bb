"""The distinct-layer vote on row masks and the batch's bit-plane peaks, at
the edges of their tiles: rows that do not fill a word or a band, one row,
the fewest and the most d0 bins, every layer in use (counts of 16: the fifth
plane and the second round of layers), per-hit region sets, and curves of
every kind (walked, edge by edge, row by row, general).  Every comparison
with the oracle is exact.
"""
import numpy as np
import pytest

import oracle
from gpu_common import assert_same_tracks, cuda_ok, gpu_tracks_event, oracle_tracks, to_dev
from synth.events import Event

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]

CP = dict(pool=3, min_layers=4, n_layers=16, tol=0.05)

# n_rho, n_d0, n_phi0, rho_max, d0_half, layers in use, threshold
SHAPES = {
    "one_row": (1, 2, 8, 0.001, 4.0, 3, 1),
    "odd_rows": (33, 6, 16, 0.01, 3.0, 16, 3),
    "two_bands_short": (257, 34, 24, 0.0114, 12.0, 12, 4),
    "most_bins": (40, 512, 16, 0.0114, 25.0, 10, 3),
    "all_layers": (96, 64, 64, 0.0114, 10.0, 16, 9),
    "curling": (130, 62, 40, 0.08, 6.0, 11, 4),
    "columns_past_a_segment": (32, 30, 264, 0.0114, 10.0, 16, 7),
}


def scene(name, seed, n=900):
    nr, nd, nphi, rmax, dh, nl, thr = SHAPES[name]
    g = dict(n_rho=nr, n_d0=nd, n_phi0=nphi, rho_max=rmax, d0_half=dh, n_z0=16, n_cot=16,
             z0_max=20.0, cot_max=3.0, threshold=thr, count_bits=16)
    rng = np.random.Generator(np.random.Philox(400 + seed))
    lay = rng.integers(0, nl, n)
    r = (2.0 + 108.0 * lay / max(nl - 1, 1)) * rng.uniform(0.98, 1.02, n)
    ph = rng.uniform(-np.pi, np.pi, n)
    # a bundle of nearly straight tracks from the origin: cells that reach every layer
    b = rng.random(n) < 0.5
    ph[b] = (np.floor(rng.random(b.sum()) * 6) + 0.5) * 2 * np.pi / nphi + rng.normal(0, 2e-4, b.sum())
    f = np.float32
    return g, Event(x=(r * np.cos(ph)).astype(f), y=(r * np.sin(ph)).astype(f),
                    z=rng.uniform(-20, 20, n).astype(f), layer=lay.astype(np.int8),
                    track=np.full(n, -1, np.int32))


@pytest.mark.parametrize("bits", [16, 32])
@pytest.mark.parametrize("name", sorted(SHAPES))
def test_single_event(name, bits):
    g, ev = scene(name, 0)
    g["count_bits"] = bits
    cap = 1 << 15
    r = gpu_tracks_event(g, ev, cap, CP)
    o = oracle_tracks(g, ev, cap, CP)
    assert_same_tracks(r, o)
    if name in ("odd_rows", "columns_past_a_segment"):
        assert o["acc"].max() == 16


@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("name", sorted(SHAPES))
def test_batch(name, masked):
    """Two events of a batch (the second empty or short), twice, with and
    without per-hit region sets."""
    import torch
    from paper_1309_6275_gb300 import ht
    g, a = scene(name, 1)
    _, b = scene(name, 2, n=300)
    evs = [a, b]
    off = np.array([0, a.n_hits, a.n_hits + b.n_hits], np.int32)
    cat = lambda k, t: to_dev(np.concatenate([getattr(e, k) for e in evs]).astype(t))
    rng = np.random.Generator(np.random.Philox(9))
    masks = None
    if masked:   # sparse, dense and empty sets
        m = rng.integers(0, 1 << 63, off[-1], dtype=np.uint64)
        m &= rng.integers(0, 1 << 63, off[-1], dtype=np.uint64)
        m[rng.random(off[-1]) < 0.3] = ~np.uint64(0)
        m[rng.random(off[-1]) < 0.1] = 0
        masks = m
    cap = 1 << 15
    G = ht.Geometry(g)
    B = ht.Batch(G, max_events=3, max_hits=int(off[-1]) + 5, cap=cap)
    B.set_confirm(CP)
    hm = None if masks is None else to_dev(masks.view(np.int64))
    args = (cat("x", np.float32), cat("y", np.float32), cat("z", np.float32), cat("layer", np.uint8))
    for _ in range(2):
        B.run_tracks(*args, off, hit_masks=hm)
    torch.cuda.synchronize()
    for e, ev in enumerate(evs):
        r = B.event_results(off, e)
        o = oracle_tracks(g, ev, cap, CP, None if masks is None else masks[off[e]:off[e + 1]])
        assert r["votes"] == o["votes"]
        assert_same_tracks(dict(r, inl=o["inl"]), o, acc=False)
    B.close()
    G.close()


def test_hits_that_vote_nowhere():
    """NaN, infinite, huge and origin hits among ordinary ones change nothing
    but their own (absent or definition-given) votes."""
    g, ev = scene("all_layers", 3)
    bad = np.array([np.nan, np.inf, -np.inf, 1e30, 0.0], np.float32)
    for q, v in enumerate(bad):
        ev.x[7 * q] = v
    ev.y[28] = 0.0
    import torch
    from paper_1309_6275_gb300 import ht
    keep = np.isfinite(ev.x) & (np.abs(ev.x) < 1e29)
    acc_o, st = oracle.vote_layers(g, ev.x[keep], ev.y[keep], ev.layer[keep])
    G = ht.Geometry(g)
    acc = G.new_accumulator()
    stats = torch.zeros(2, dtype=torch.int64, device="cuda")
    ht.ht_vote_layers(G, to_dev(ev.x), to_dev(ev.y), to_dev(ev.layer.astype(np.uint8)), acc, stats)
    assert np.array_equal(acc.cpu().numpy().view(np.uint16), acc_o)
    assert int(stats[0]) == st["votes"]
    G.close()


# Dense events: layers voted cell by cell (24000 hits and more), with the layers
# and rows that leave that path: tight curls, spread radii, more hits of a cell
# than are put in order, hits that are not finite, a second round of layers.
DENSE = {   # n_rho, n_d0, n_phi0, rho_max, d0_half, layers
    "rings": (64, 64, 32, 0.0114, 20.0, 10),
    "pileup_like": (130, 66, 24, 0.0228, 30.0, 10),
    "curled": (96, 32, 16, 0.05, 8.0, 12),
    "few_bins": (40, 6, 16, 0.0114, 10.0, 8),
    "clustered": (64, 64, 32, 0.0114, 20.0, 10),
    "spread": (64, 64, 32, 0.0114, 20.0, 10),
    "doubled": (64, 64, 32, 0.0114, 20.0, 10),
    "not_finite": (64, 64, 32, 0.0114, 20.0, 10),
}


def dense(name, seed, n):
    nr, nd, nphi, rmax, dh, nl = DENSE[name]
    g = dict(n_rho=nr, n_d0=nd, n_phi0=nphi, rho_max=rmax, d0_half=dh, n_z0=16, n_cot=16,
             z0_max=20.0, cot_max=3.0, threshold=nl, count_bits=16)
    rng = np.random.Generator(np.random.Philox(900 + seed))
    lay = rng.integers(0, nl, n)
    r = 4.0 + 106.0 * lay / (nl - 1)
    ph = rng.uniform(-np.pi, np.pi, n)
    if name == "spread":
        r = r * np.where(lay % 2 == 0, rng.uniform(0.995, 1.005, n), 1.0)
    if name == "clustered":
        c = rng.random(n) < 0.3
        ph[c] = 0.4 + rng.uniform(0, 0.02, c.sum())
    if name == "doubled":
        ph[1::2], lay[1::2], r[1::2] = ph[0::2], lay[0::2], r[0::2]
    x, y = (r * np.cos(ph)).astype(np.float32), (r * np.sin(ph)).astype(np.float32)
    if name == "not_finite" and n > 500:
        x[5], y[77], x[300], x[400], y[400] = np.nan, np.inf, -np.inf, 0.0, 0.0
    return g, Event(x=x, y=y, z=rng.uniform(-20, 20, n).astype(np.float32),
                    layer=lay.astype(np.int8), track=np.full(n, -1, np.int32))


@pytest.mark.parametrize("name", sorted(DENSE))
def test_dense_batch(name):
    """A dense event, a small one and one at the line between the two ways,
    against the oracle: votes, peaks, confirmation, assignment, z vote."""
    import torch
    from paper_1309_6275_gb300 import ht
    evs = [dense(name, q, n)[1] for q, n in enumerate((25000, 1200, 24000))]
    g = dense(name, 0, 100)[0]
    off = np.concatenate([[0], np.cumsum([e.n_hits for e in evs])]).astype(np.int32)
    cat = lambda k, t: to_dev(np.concatenate([getattr(e, k) for e in evs]).astype(t))
    cap = 1 << 16
    G = ht.Geometry(g)
    B = ht.Batch(G, max_events=4, max_hits=int(off[-1]), cap=cap)
    B.set_confirm(CP)
    for _ in range(2):
        B.run_tracks(cat("x", np.float32), cat("y", np.float32), cat("z", np.float32),
                     cat("layer", np.uint8), off)
    torch.cuda.synchronize()
    for e, ev in enumerate(evs):
        r = B.event_results(off, e)
        ok = np.isfinite(ev.x) & np.isfinite(ev.y)   # (no such hit votes)
        acc, st = oracle.vote_layers(g, ev.x[ok], ev.y[ok], ev.layer[ok])
        pk, cnt = oracle.peaks(g, acc, cap)
        assert r["votes"] == st["votes"]
        assert r["count"] == cnt and np.array_equal(r["peaks"], pk)
        if ok.all() and cnt < 3000:
            assert_same_tracks(dict(r, inl=None), dict(oracle_tracks(g, ev, cap, CP), inl=None),
                               acc=False)
    B.close()
    G.close()
