"""What a batch handle takes of the GPU's memory: counts for the plain path at
creation, bit planes when the track path is switched on and they need more
than the counts, and less scratch where there is no room for all of it."""
import numpy as np
import pytest

import oracle
from gpu_common import assert_same_tracks, batch_event, cuda_ok, oracle_tracks, to_dev
from synth.events import Event

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]

CP = dict(pool=4, min_layers=3, n_layers=10, tol=0.05)
MB = 1 << 20


def event(n, seed):
    rng = np.random.Generator(np.random.Philox(8100 + seed))
    lay = rng.integers(0, 10, n)
    r = 4.0 + 106.0 * lay / 9.0
    t = rng.integers(0, max(n // 9, 1), n)
    phi = rng.uniform(-np.pi, np.pi, n)[t]
    f = np.float32
    return Event(x=(r * np.cos(phi)).astype(f), y=(r * np.sin(phi)).astype(f),
                 z=rng.uniform(-20, 20, n).astype(f), layer=lay.astype(np.int8),
                 track=np.full(n, -1, np.int32))


def geometry(nr, nd, nphi, rho_max, threshold):
    return dict(n_rho=nr, n_d0=nd, n_phi0=nphi, rho_max=rho_max, d0_half=8.0, n_z0=16, n_cot=16,
                z0_max=20.0, cot_max=3.0, threshold=threshold, count_bits=16)


def free():
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("nr", [1, 8, 16])
def test_few_rows_take_the_counts_memory_until_the_track_path_is_asked_for(nr):
    """A word of a bit plane holds 32 rows however few there are: 24 bytes per
    (column, bin), against 2 per row for the counts."""
    from paper_1309_6275_gb300 import ht
    g = geometry(nr, 256, 2048, 0.001, 3)
    events, evs = 64, [event(600, 1), event(40, 2)]
    counts = nr * 256 * 2048 * 2 * events
    off = np.array([0, evs[0].n_hits, evs[0].n_hits + evs[1].n_hits], np.int32)
    G = ht.Geometry(g)
    ht.Batch(G, max_events=1, max_hits=1, cap=1).close()   # (a process's first handle loads the kernels)
    f0 = free()
    B = ht.Batch(G, max_events=events, max_hits=int(off[-1]), cap=1 << 12)
    took = f0 - free()
    # + the peaks' scratch (8 bytes and 32 of bits per segment of 256 columns)
    # and what is neither per cell nor per column
    assert took < counts + nr * 256 * 8 * 40 * events + 64 * MB
    cat = lambda k, t: to_dev(np.concatenate([getattr(e, k) for e in evs]).astype(t))
    x, y, z = (cat(k, np.float32) for k in "xyz")
    B.run(x, y, z, off)
    for e, ev in enumerate(evs):
        acc, st = oracle.vote(g, ev.x, ev.y)
        pk, cnt = oracle.peaks(g, acc, 1 << 12)
        r = batch_event(B, off, e)
        assert r["votes"] == st["votes"] and r["count"] == cnt and np.array_equal(r["peaks"], pk)
    f1 = free()
    B.set_confirm(CP)
    if nr < 12:
        assert f1 - free() > 24 * 256 * 2048 * events
    for _ in range(2):
        B.run_tracks(x, y, z, cat("layer", np.uint8), off)
        for e, ev in enumerate(evs):
            r = B.event_results(off, e)
            o = oracle_tracks(g, ev, 1 << 12, CP)
            assert r["votes"] == o["votes"]
            assert_same_tracks(dict(r, inl=o["inl"]), o, acc=False)
        B.run(x, y, z, off)   # the two paths take turns on the handle
    B.close()
    G.close()


def test_a_batch_that_has_no_room_for_the_peak_bits():
    """With 130 MB less free than the handle took at first it is made all the
    same, finding its peaks by a second comparison, and its track path with
    scratch for fewer events at a time."""
    import torch
    from paper_1309_6275_gb300 import ht
    g = geometry(2048, 512, 8, 0.0114, 4)     # 32 bytes of bits for 16 of counts
    evs = [event(500, 3 + e) for e in range(4)]
    off = np.concatenate([[0], np.cumsum([e.n_hits for e in evs])]).astype(np.int32)
    cat = lambda k, t: to_dev(np.concatenate([getattr(e, k) for e in evs]).astype(t))
    hits = [cat(k, np.float32) for k in "xyz"] + [cat("layer", np.uint8)]
    G = ht.Geometry(g)

    def run():
        B = ht.Batch(G, max_events=4, max_hits=int(off[-1]), cap=1 << 12)
        B.set_confirm(CP)
        took = before - free()
        out = []
        B.run(*hits[:3], off)
        out += [batch_event(B, off, e) for e in range(4)]
        B.run_tracks(*hits, off)
        out += [batch_event(B, off, e) for e in range(4)]
        B.close()
        return took, out

    before = free()
    took, full = run()
    before = free()
    rest = torch.empty(before - took + 130 * MB, dtype=torch.uint8, device="cuda")
    try:
        short = run()[1]
    finally:
        del rest
        torch.cuda.empty_cache()
    for a, b in zip(full, short):
        assert a["count"] == b["count"] > 0 and a["votes"] == b["votes"]
        for k in ("peaks", "assign", "zres"):
            assert np.array_equal(a[k], b[k])
    G.close()


@pytest.mark.parametrize("n_r,n_theta", [(32, 64), (500, 4096), (1024, 65536)])
def test_a_vertex_workspace_stays_below_the_accumulators(n_r, n_theta):
    """The peaks' scratch of several events at a time, at most 32 MB or one
    event's (40 bytes per 256 cells), whatever the accumulator's size."""
    from paper_1309_6275_gb300 import ht
    G = ht.Geometry(geometry(16, 32, 64, 0.0114, 3))
    V = ht.Vertex(G, dict(n_r=n_r, n_theta=n_theta, r_max=30.0, r_keep=1.0, threshold=3), 1, 16)
    one = n_r * -(-n_theta // 256) * 40
    assert V.ws.numel() <= max(32 * MB, 1.05 * one + 4096)
    V.close()
    G.close()
