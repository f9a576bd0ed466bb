"""bench.py's operation count of the layer vote: runs of votes by the
definition's roots, against the oracle's votes and by hand; and the launches
of a track batch."""
import numpy as np

import bench
import oracle
import synth

G = dict(n_rho=64, n_d0=64, n_phi0=64, rho_max=0.0114, d0_half=10.0, n_z0=16, n_cot=16,
         z0_max=20.0, cot_max=3.0, threshold=4, count_bits=16)


def test_votes_are_the_oracles():
    ev = synth.make_event(synth.CONFIGS["single_64"]["gen"], 3)
    x, y = ev.x[:120], ev.y[:120]
    votes, runs = bench.count_runs(G, x, y)
    assert votes == oracle.vote(G, x, y)[1]["votes"]
    assert 0 < runs < votes


def test_runs_are_the_stretches_of_a_bin():
    """One hit, row by row from the oracle: a run begins where a row's bin is
    not the previous row's."""
    for g in (G, dict(G, n_rho=7)):
        for x, y in ((60.0, 1.0), (4.0, 0.3), (-80.0, 75.0)):
            x, y = np.array([x], np.float32), np.array([y], np.float32)
            acc, _ = oracle.vote(g, x, y)          # rows, bins, columns
            a = np.asarray(acc).reshape(g["n_rho"], g["n_d0"], g["n_phi0"]) > 0
            begins = a[0].sum() + (a[1:] & ~a[:-1]).sum()
            votes, runs = bench.count_runs(g, x, y)
            assert votes == a.sum() and runs == begins
    votes, runs = bench.count_runs(dict(G, n_rho=1), np.array([50.0], np.float32),
                                   np.array([9.0], np.float32))
    assert votes == runs > 0                       # one row: every vote is a run


def test_a_sample_stands_for_the_events():
    evs = [synth.make_event(synth.CONFIGS["stream2000_256"]["gen"], s, target_hits=n)
           for s, n in ((1, 400), (2, 1600))]
    g = dict(G, n_phi0=128)
    x, y = (np.concatenate([getattr(e, q) for e in evs]) for q in "xy")
    votes, runs = bench.count_runs(g, x[::5], y[::5])
    got = bench.runs_per_vote(g, evs)
    assert abs(got / (runs / votes) - 1.0) < 0.1
    assert got == bench.runs_per_vote(g, evs)      # (seeded)


def test_track_launches():
    """The index, the vote, the peaks, the confirmation and the z vote; with the
    proposal the network, and one vote instead of the sort and two."""
    assert bench.track_launches() == 6 + 3 + 5 + 3 + 6
    assert bench.track_launches(learned=True) == bench.track_launches() - 1
