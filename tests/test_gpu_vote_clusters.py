"""The plain batch vote in clusters of tiles against the oracle: columns that
divide into clusters and columns that do not, both packed tile widths, rows
past the last full tile, an event with no hits, and an event above the packed
limit among small ones (its tiles take other launches).  Whole numbers:
equal."""
import numpy as np
import pytest

import oracle
from gpu_common import batch_event, cuda_ok, to_dev

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]

PACK_MAX = 32767   # hits of an event up to which every tile is packed


@pytest.mark.parametrize("big", [0, PACK_MAX, PACK_MAX + 1])
@pytest.mark.parametrize("nr,nd,nphi", [(32, 16, 32), (40, 18, 48), (70, 34, 40), (33, 256, 16),
                                        (33, 256, 24)])
def test_clusters_and_single_tiles_equal_the_oracle(nr, nd, nphi, big):
    import torch
    from paper_1309_6275_gb300 import ht
    g = dict(n_rho=nr, n_d0=nd, n_phi0=nphi, rho_max=0.0114, d0_half=20.0, n_z0=16, n_cot=16,
             z0_max=20.0, cot_max=3.0, threshold=6, count_bits=16)
    sizes = [300, big, 0, 1, 1000]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    n = int(off[-1])
    rng = np.random.Generator(np.random.Philox(1000 + nr + big))
    r, ph = rng.uniform(3, 110, n), rng.uniform(-np.pi, np.pi, n)
    x, y = (r * np.cos(ph)).astype(np.float32), (r * np.sin(ph)).astype(np.float32)
    z = rng.uniform(-20, 20, n).astype(np.float32)
    cap = 1 << 14
    G = ht.Geometry(g)
    B = ht.Batch(G, max_events=5, max_hits=n, cap=cap)
    for _ in range(2):   # plain launches, then the captured ones
        B.run(to_dev(x), to_dev(y), to_dev(z), off)
    torch.cuda.synchronize()
    for e in range(5):
        a, b = off[e], off[e + 1]
        acc, st = oracle.vote(g, x[a:b], y[a:b])
        pk, cnt = oracle.peaks(g, acc, cap)
        res = batch_event(B, off, e)
        assert res["votes"] == st["votes"], e
        assert res["count"] == cnt and np.array_equal(res["peaks"], pk), e
        if cnt <= cap:
            sub = np.arange(b - a)[::max(1, (b - a) // 300)].astype(np.int64)
            want = oracle.associate_dense(g, x[a:b], y[a:b], pk, hit_idx=sub)
            assert np.array_equal(res["assign"][sub], want), e
    B.close()
    G.close()
