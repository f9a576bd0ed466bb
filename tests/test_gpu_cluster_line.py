"""The plain batch vote around the hit counts up to which events vote in
clusters of tiles, plain, with per-hit region sets and under event masks,
against the oracle; and the vote under event masks timed against the plain
one."""
import numpy as np
import pytest

import oracle
from gpu_common import batch_event, cuda_ok, to_dev

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]


def cluster_hits(nd, kind):
    return {"plain": nd * max(nd, 128) * 3 // 32, "sets": 64 * nd,
            "masks": 24 * nd if nd > 128 else 0}[kind]


def scene(sizes, seed):
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    rng = np.random.Generator(np.random.Philox(7300 + seed))
    n = int(off[-1])
    r, ph = rng.uniform(3, 110, n), rng.uniform(-np.pi, np.pi, n)
    return (off, (r * np.cos(ph)).astype(np.float32), (r * np.sin(ph)).astype(np.float32),
            rng.uniform(-20, 20, n).astype(np.float32), rng)


@pytest.mark.parametrize("kind,nd", [("plain", 4), ("plain", 34), ("plain", 128), ("sets", 4),
                                     ("sets", 34), ("sets", 128), ("masks", 34), ("masks", 200)])
def test_events_on_both_sides_of_the_line(kind, nd):
    import torch
    from oracle import mlp
    from paper_1309_6275_gb300 import ht
    g = dict(n_rho=40, n_d0=nd, n_phi0=64, rho_max=0.0114, d0_half=20.0, n_z0=16, n_cot=16,
             z0_max=20.0, cot_max=3.0, threshold=6, count_bits=16)
    c = max(cluster_hits(nd, kind), 300)
    off, x, y, z, rng = scene([c - 1, c + 1, 0, c, 2 * c], nd)
    cap = 1 << 15
    u64 = lambda n: rng.integers(0, 1 << 63, n, dtype=np.uint64)
    masks = u64(len(x)) & u64(len(x))
    per_event = u64(5) | u64(5)
    i64 = lambda m: to_dev(m.view(np.int64))
    G = ht.Geometry(g)
    B = ht.Batch(G, max_events=5, max_hits=len(x), cap=cap)
    hits = [to_dev(a) for a in (x, y, z)]
    for _ in range(2):
        if kind == "sets":
            B.run_hit_masked(*hits, off, i64(masks))
        elif kind == "masks":
            B.run_masked(*hits, off, i64(per_event))
        else:
            B.run(*hits, off)
    torch.cuda.synchronize()
    for e in range(5):
        a, b = off[e], off[e + 1]
        r = batch_event(B, off, e)
        if kind == "masks":
            o = mlp.masked_event(g, x[a:b], y[a:b], z[a:b], int(per_event[e]), cap=cap)
            assert r["votes"] == o["votes"] and r["count"] == o["count"], e
            assert np.array_equal(r["peaks"], o["peaks"]), e
            continue
        acc, st = (oracle.vote_hitmask(g, x[a:b], y[a:b], masks[a:b]) if kind == "sets"
                   else oracle.vote(g, x[a:b], y[a:b]))
        pk, cnt = oracle.peaks(g, acc, cap)
        assert r["votes"] == st["votes"], e
        assert r["count"] == cnt and np.array_equal(r["peaks"], pk), e
    B.close()
    G.close()


def masked_over_plain():
    """The vote stage under masks of every region over the plain one."""
    import torch
    from paper_1309_6275_gb300 import ht
    g = dict(n_rho=256, n_d0=128, n_phi0=512, rho_max=0.0114, d0_half=20.0, n_z0=16, n_cot=16,
             z0_max=20.0, cot_max=3.0, threshold=60, count_bits=16)
    off, x, y, z, _ = scene([10000] * 4, 1)
    G = ht.Geometry(g)
    B = ht.Batch(G, max_events=4, max_hits=len(x), cap=1 << 18)
    x, y, z = to_dev(x), to_dev(y), to_dev(z)
    every = torch.full((4,), -1, dtype=torch.int64, device="cuda")
    best = [1e30, 1e30]
    for i in range(8):
        for q, f in enumerate((lambda: B.run(x, y, z, off), lambda: B.run_masked(x, y, z, off, every))):
            f()
            torch.cuda.synchronize()
            best[q] = min(best[q], B.stage_ms()[1])
    B.close()
    G.close()
    return best[1] / best[0]


def test_event_masks_cost_little_over_the_plain_vote():
    """Masks of every region restrict nothing: 0.99 of the plain vote (1.04 in
    clusters, with registers spilled)."""
    assert masked_over_plain() < 1.03
