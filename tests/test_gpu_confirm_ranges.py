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
