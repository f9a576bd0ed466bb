"""The batched layer vote on both sides of the hit count from which an event's
dense layers go cell by cell, on test_gpu_vote_rows' dense scenes (tight
curls, spread radii, crowded cells, hits that are not finite), against the
oracle."""
import numpy as np
import pytest

import oracle
from gpu_common import cuda_ok, to_dev
from test_gpu_vote_rows import CP, DENSE, dense

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]

CELL_HITS = 28000


@pytest.mark.parametrize("name", sorted(DENSE))
def test_events_around_the_line(name):
    import torch
    from paper_1309_6275_gb300 import ht
    evs = [dense(name, 10 + q, n)[1] for q, n in enumerate((CELL_HITS - 2, 700, CELL_HITS,
                                                            CELL_HITS + 3000))]
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
    B.close()
    G.close()
