"""The refinement and the (z0, cot theta) vote at the edges of their lane
widths: candidates of 3 to 48 hits fitted by eight lanes (few candidates), by a
thread each (many) and by a warp (more than 32 hits), against the oracle; the
z vote with 1 to 40 hits per candidate and cot columns that do not fill a
warp, exactly."""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import cuda_ok, to_dev
from synth.events import helix_hits
from test_gpu_fit import compare, gpu_fit

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]


def tracks_of(sizes, seed):
    """Candidates with the given hit counts: smeared hits of one helix each on
    as many radii; (geometry, x, y, z, assign, peaks)."""
    g = synth.geometry_of("event100_256")
    rng = np.random.Generator(np.random.Philox(seed))
    phi0, _, _, rhos = oracle.tables(g)
    xs, ys, zs, a, pk = [], [], [], [], []
    for m, n in enumerate(sizes):
        i, j, k = (int(rng.integers(20, 236)), int(rng.integers(40, 88)), int(rng.integers(512)))
        delta = 2 * g["d0_half"] / g["n_d0"]
        d0 = (j - g["n_d0"] / 2) * delta + 0.2 * delta
        X, Y, Z, _, _ = helix_hits(float(rhos[i]), d0, float(phi0[k]), rng.normal(0, 3),
                                   rng.uniform(-2, 2), np.linspace(14.0, 84.0, n))
        assert len(X) == n
        xs.append(X + rng.normal(0, 20e-4, n)); ys.append(Y + rng.normal(0, 20e-4, n)); zs.append(Z)
        a.append(np.full(n, m)); pk.append((i, j, k, n))
    f = lambda v: np.concatenate(v).astype(np.float32)
    return g, f(xs), f(ys), f(zs), np.concatenate(a).astype(np.int32), np.array(pk, np.int32)


@pytest.mark.parametrize("copies", [1, 400])
@pytest.mark.parametrize("sel", [dict(), dict(road=1.0, cut=5.0)])
def test_fit_widths(copies, sel):
    """One copy: eight lanes or a warp per candidate; 400 events of the same
    candidates: a thread each.  Every copy is the oracle's fit."""
    import torch
    from paper_1309_6275_gb300 import ht
    sizes = [3, 4, 5, 8, 9, 10, 16, 17, 25, 31, 32, 33, 40, 48] * 2
    g, x, y, _, assign, pk = tracks_of(sizes, 5)
    G = ht.Geometry(g)
    cap = len(sizes) + 3
    off = np.arange(copies + 1) * len(x)
    peaks = np.zeros((copies, cap, 4), np.int32)
    peaks[:, :len(sizes)] = pk
    tr = gpu_fit(G, ht, to_dev(np.tile(x, copies)), to_dev(np.tile(y, copies)), off,
                 to_dev(np.tile(assign, copies)), to_dev(peaks.reshape(-1, 4)),
                 torch.full((copies,), len(sizes), dtype=torch.int32, device="cuda"), cap, **sel)
    for c in (0, copies // 2, copies - 1):
        n_fit, n_cmp = compare(g, x, y, assign, pk, tr[c * cap:c * cap + len(sizes)], **sel)
        assert n_fit == len([n for n in sizes if n >= 4]) and n_cmp >= n_fit - 4
    G.close()


@pytest.mark.parametrize("n_z0,n_cot", [(128, 128), (37, 20), (16, 45), (1, 1), (700, 33)])
def test_z_vote_widths(n_z0, n_cot):
    import torch
    from paper_1309_6275_gb300 import ht
    sizes = [1, 2, 3, 8, 10, 31, 32, 33, 40]
    g, x, y, z, assign, pk = tracks_of(sizes, 6)
    g.update(n_z0=n_z0, n_cot=n_cot)
    assign = np.concatenate([assign, [-1, len(sizes), len(sizes) + 1]]).astype(np.int32)
    x, y, z = (np.concatenate([v, v[:3]]) for v in (x, y, z))
    pk = np.concatenate([pk, pk[:1]])   # the last candidate: no hit but one below
    assign[-2] = -1
    G = ht.Geometry(g)
    n, cap = len(x), len(pk)
    out = torch.full((cap, 3), -9, dtype=torch.int32, device="cuda")
    ws = torch.empty(G.vote_z_workspace_size(n, cap), dtype=torch.uint8, device="cuda")
    ht.ht_vote_z(G, to_dev(x), to_dev(y), to_dev(z), to_dev(assign), to_dev(pk),
                 torch.tensor([cap], dtype=torch.int32, device="cuda"), cap, out, ws)
    keep = np.where(assign < cap, assign, -1)
    assert np.array_equal(out.cpu().numpy(), oracle.vote_z(g, x, y, z, keep, pk))
    G.close()
