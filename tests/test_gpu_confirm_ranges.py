"""The confirmation over the whole range of its parameters, against the
oracle: pools up to the largest int32 (every bin of the column)."""
import functools

import numpy as np
import pytest

import oracle
import synth
from gpu_common import cuda_ok, oracle_tracks, gpu_tracks_event, assert_same_tracks

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]

G64 = dict(n_rho=64, n_d0=64, n_phi0=64, rho_max=0.0114, d0_half=10.0, n_z0=16, n_cot=16,
           z0_max=20.0, cot_max=3.0, threshold=6, count_bits=16)


@functools.lru_cache(maxsize=4)
def scene(n, seed=0):
    return synth.make_event(synth.CONFIGS["stream2000_256"]["gen"], 700 + seed, target_hits=n)


@pytest.mark.parametrize("pool", [2**31 - 1, 2**31 - 2, 2**31 - 60, 64])
def test_a_pool_of_every_bin(pool):
    """The largest pools take the hits of every bin, as one of n_d0 does."""
    cp = dict(pool=pool, min_layers=6, n_layers=10, tol=0.02)
    ev = scene(1500)
    cap = 1 << 13
    r = gpu_tracks_event(G64, ev, cap, cp)
    o = oracle_tracks(G64, ev, cap, dict(cp, pool=64))
    assert (o["score"] > 0).sum() > 20
    assert_same_tracks(r, o)


@pytest.mark.parametrize("pool", [0, 2, 64])
@pytest.mark.parametrize("tol", [0.05, 1.0, 30.0, 1e6])
def test_tolerances_as_wide_as_the_pool(pool, tol):
    """Tolerances that reach most of a layer: the pool's windows instead of the
    circle's, and several passes of hits."""
    cp = dict(pool=pool, min_layers=4, n_layers=10, tol=tol)
    ev = scene(2600, 1)
    cap = 1 << 13
    r = gpu_tracks_event(G64, ev, cap, cp)
    o = oracle_tracks(G64, ev, cap, cp)
    assert (o["score"] > 0).sum() > (20 if pool else 5)
    assert_same_tracks(r, o)


def confirm_ms(cp, ev, g):
    """Time of ht_confirm alone (the least of five)."""
    import torch
    from gpu_common import to_dev
    from paper_1309_6275_gb300 import ht
    G = ht.Geometry(g)
    n, cap = ev.n_hits, 1 << 17
    x, y, lay = to_dev(ev.x), to_dev(ev.y), to_dev(ev.layer.astype(np.uint8))
    acc = G.new_accumulator()
    ht.ht_vote_layers(G, x, y, lay, acc)
    i32 = lambda *s: torch.zeros(s, dtype=torch.int32, device="cuda")
    peaks, cnt, score, inl, asg = i32(cap, 4), i32(1), i32(cap), i32(cap, 16), i32(n)
    ws = torch.empty(max(G.find_peaks_workspace_size(), ht.ht_confirm_workspace_size(G, n, cap)),
                     dtype=torch.uint8, device="cuda")
    ht.ht_find_peaks(G, acc, peaks, cap, cnt, ws)
    best = 1e9
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        ht.ht_confirm(G, cp, x, y, lay, peaks, cnt, cap, score, inl, asg, ws)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    G.close()
    return best


def test_a_wide_tolerance_costs_no_more_than_the_pool():
    """With a tolerance beyond the detector every pool hit is near the circle,
    so a candidate costs about its pool: on 10k hits a few times the narrow
    tolerance's time (which scans a fraction of it), where scanning the
    circle's window would cost the whole event per candidate and pass (over two
    hundred times)."""
    g = synth.track_geometry("event100_256")
    ev = synth.make_event(synth.CONFIGS["event100_256"]["gen"], 31, target_hits=10000)
    narrow = confirm_ms(dict(pool=4, min_layers=8, n_layers=10, tol=0.01), ev, g)
    wide = confirm_ms(dict(pool=4, min_layers=8, n_layers=10, tol=100.0), ev, g)
    assert wide < 20 * narrow, (narrow, wide)
