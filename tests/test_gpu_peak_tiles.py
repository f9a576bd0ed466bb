"""The peak finder's tiles (16 d0 bins x 256 phi0 columns of a row) by how many
of their cells reach the threshold: none, few (compared one by one), the line
at 512 and many (the staged walk), on both counter widths and ragged sizes,
with the peak bits and without, against the oracle.  Whole numbers: equal."""
import numpy as np
import pytest

import oracle
from gpu_common import cuda_ok, to_dev

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]

THR = 5


def geometry(nr, nd, nphi, bits):
    return dict(n_rho=nr, n_d0=nd, n_phi0=nphi, rho_max=0.01, d0_half=2.0, n_z0=16, n_cot=16,
                z0_max=20.0, cot_max=3.0, threshold=THR, count_bits=bits)


def tiles(shape, hot, seed):
    """Counts below the threshold, and in every tile of 16 bins x 256 columns
    `hot` cells (at most all) of 5..8, so that neighbours tie often."""
    rng = np.random.Generator(np.random.Philox(seed))
    acc = rng.integers(0, THR, shape)
    nr, nd, nphi = shape
    for i in range(nr):
        for j in range(0, nd, 16):
            for k in range(0, nphi, 256):
                t = acc[i, j:j + 16, k:k + 256]
                at = rng.permutation(t.size)[:hot]
                v = t.ravel()
                v[at] = rng.integers(THR, THR + 4, at.size)
                acc[i, j:j + 16, k:k + 256] = v.reshape(t.shape)
    return acc


@pytest.mark.parametrize("bits", [16, 32])
@pytest.mark.parametrize("hot", [0, 1, 40, 511, 512, 513, 4096])
@pytest.mark.parametrize("shape", [(3, 32, 512), (5, 18, 264), (1, 2, 8)])
def test_tiles_by_cells_at_the_threshold(shape, hot, bits):
    import torch
    from paper_1309_6275_gb300 import ht
    g = geometry(*shape, bits)
    acc = tiles(shape, hot, 70 + hot)
    cap = 1 << 14
    pk_o, cnt_o = oracle.peaks(g, acc, cap=cap)
    G = ht.Geometry(g)
    a = to_dev(acc.astype(np.uint16).view(np.int16) if bits == 16 else acc.astype(np.int32))
    size = G.find_peaks_workspace_size()
    bits_bytes = (shape[0] * shape[1] * ((shape[2] + 255) // 256) * 32 + 255) // 256 * 256
    for ws in (size, size - bits_bytes, None):   # with the bits, without, no workspace
        pk = torch.full((cap, 4), -7, dtype=torch.int32, device="cuda")
        n = torch.zeros(1, dtype=torch.int32, device="cuda")
        if ws is None:
            ht.ht_find_peaks_noalloc(G, a, pk, cap, n)
        else:
            ht.ht_find_peaks(G, a, pk, cap, n, torch.empty(ws, dtype=torch.uint8, device="cuda"))
        torch.cuda.synchronize()
        k = min(cnt_o, cap)
        assert int(n.item()) == cnt_o, ws
        assert np.array_equal(pk[:k].cpu().numpy(), pk_o[:k]), ws
        assert (pk[k:] == -7).all(), ws
    G.close()


@pytest.mark.parametrize("full", [True, False])
def test_vertex_peaks_of_more_events_than_one_launch_takes(full):
    """33 events: two groups with the whole workspace, one event at a time
    with the smallest."""
    import torch
    from paper_1309_6275_gb300 import ht
    G = ht.Geometry(geometry(16, 16, 64, 16))
    vd = dict(n_r=20, n_theta=288, threshold=THR, r_max=10.0, r_keep=2.0)
    n_ev, cap = 33, 1 << 11
    V = ht.Vertex(G, vd, n_ev, cap)
    acc = np.concatenate([tiles((1, 20, 288), (0, 3, 600)[e % 3], 300 + e) for e in range(n_ev)])
    V.acc.copy_(to_dev(acc.astype(np.int32)))
    small = 2 * 512 + 256   # the counts and offsets of 40 segments, the scan's sums
    ws = V.ws if full else torch.empty(small, dtype=torch.uint8, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    r = ht.lib().ht_vertex_find(V.handle, V.acc.data_ptr(), n_ev, V.peaks.data_ptr(), cap,
                                V.counts.data_ptr(), V.first.data_ptr(), ws.data_ptr(), ws.numel(),
                                s)
    assert r == 0
    torch.cuda.synchronize()
    go = geometry(1, 20, 288, 32)
    for e in range(n_ev):
        pk_o, cnt_o = oracle.peaks(go, acc[e:e + 1], cap=cap)
        res = V.event_results(e)
        assert res["count"] == cnt_o
        assert np.array_equal(res["peaks"], pk_o)
    V.close()
    G.close()
