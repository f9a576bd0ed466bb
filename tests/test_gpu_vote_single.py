"""The single-event distinct-layer vote where its tiles change: hit counts at
the edges of the warps' chunks, few rows (several hits per step) on few
and on many columns.  Cell for cell against the oracle.  The time bounds are
against the plain vote (ht_vote) of the same event, which evaluates every
(hit, row) of every column.
"""
import numpy as np
import pytest

import oracle
from gpu_common import assert_same_acc, cuda_ok, to_dev

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]


def geometry(nr, nd, nphi, bits=16):
    return dict(n_rho=nr, n_d0=nd, n_phi0=nphi, rho_max=0.0114, d0_half=10.0, n_z0=16, n_cot=16,
                z0_max=20.0, cot_max=3.0, threshold=4, count_bits=bits)


def hits(n, layers, seed):
    """Hits of tracks from near the origin on rings at 4 to 110 cm, in random order."""
    rng = np.random.Generator(np.random.Philox(4100 + seed))
    lay = rng.choice(np.asarray(layers), n)
    r = 4.0 + 106.0 * lay / 15.0
    t = rng.integers(0, max(n // 8, 1), n)
    phi, rho = rng.uniform(-np.pi, np.pi, n)[t], rng.uniform(-0.0114, 0.0114, n)[t]
    a = phi + np.arcsin(rho * r / 2) + rng.normal(0, 1e-3, n)
    return ((r * np.cos(a)).astype(np.float32), (r * np.sin(a)).astype(np.float32),
            lay.astype(np.uint8))


def check(g, x, y, lay):
    import torch
    from paper_1309_6275_gb300 import ht
    G = ht.Geometry(g)
    acc = G.new_accumulator()
    acc.fill_(-1)
    stats = torch.zeros(2, dtype=torch.int64, device="cuda")
    ht.ht_vote_layers(G, to_dev(x), to_dev(y), to_dev(lay), acc, stats)
    o, st = oracle.vote_layers(g, x, y, lay)
    a = acc.cpu().numpy()
    assert_same_acc(a.view(np.uint16) if a.dtype == np.int16 else a, o)
    assert int(stats[0]) == st["votes"]
    G.close()
    return o


@pytest.mark.parametrize("n", [0, 1, 2, 31, 33, 255, 256, 257, 319, 320, 321, 511, 513, 639, 640,
                               641, 1279, 1281])
def test_hits_at_the_edges_of_chunks(n):
    check(geometry(33, 34, 16), *hits(n, range(12), n))
    check(geometry(33, 34, 464), *hits(n, range(10), n))   # tiles of 256 threads


@pytest.mark.parametrize("nphi", [24, 480])
@pytest.mark.parametrize("nr", [1, 2, 3, 5, 8, 9, 16, 17, 31, 32, 48, 64])
def test_few_rows(nr, nphi):
    check(geometry(nr, 40, nphi, 16 if nr % 2 else 32), *hits(700, range(10), nr))


def least_us(f):
    """The least time of ten launches back to back, of five."""
    import torch
    best = 1e30
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(10):
            f()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 100.0)
    return best


def layer_over_plain(g, n, layers):
    """Time of ht_vote_layers over that of ht_vote, same event."""
    from paper_1309_6275_gb300 import ht
    x, y, lay = (to_dev(a) for a in hits(n, layers, 7))
    G = ht.Geometry(g)
    acc = G.new_accumulator()
    t = (least_us(lambda: ht.ht_vote_layers(G, x, y, lay, acc)) /
         least_us(lambda: ht.ht_vote(G, x, y, acc)))
    G.close()
    return t


def test_few_rows_cost_no_more_than_the_plain_vote():
    """8 rows, 20k hits: about 0.4 of the plain vote (a lane per row and hits
    that cannot vote among the others' lanes made it over 1.3)."""
    assert layer_over_plain(geometry(8, 64, 512), 20000, range(10)) < 1.3


@pytest.mark.parametrize("bits", [16, 32])
@pytest.mark.parametrize("layers", [range(11), range(10, 16), [15], [9, 10], range(16)],
                         ids=["11", "last6", "one", "both_sides", "16"])
def test_layers_of_the_second_round(layers, bits):
    """Layers past the ten that a tile holds at once: a second round of votes on
    the first one's counts, up to 16 in a cell."""
    o = check(geometry(70, 36, 16, bits), *hits(12000, layers, len(layers)))
    if len(layers) == 16:
        assert o.max() == 16


def test_sixteen_layers_write_the_counts_once():
    """300 hits, where writing the accumulator is most of the time: about 1.4
    of the plain vote (over 1.8 when the second round read it back and wrote
    it again)."""
    assert layer_over_plain(geometry(256, 128, 512), 300, range(16)) < 1.8


@pytest.mark.parametrize("nphi", [8, 16, 40])
@pytest.mark.parametrize("nr", [64, 65, 256, 300])
def test_few_columns(nr, nphi):
    """Fewer tiles than SMs at the widest bands: narrower ones."""
    check(geometry(nr, 40, nphi), *hits(700, range(10), nr))


def test_few_columns_use_the_sms():
    """8 columns of 256 rows, 20k hits: about a quarter of the plain vote (one
    tile per column on 8 SMs took about 0.7 of it)."""
    assert layer_over_plain(geometry(256, 128, 8), 20000, range(10)) < 0.45
