"""Performance cases of the track finder: the calls a program makes, over the
sizes it makes them with.

A case is one pass of a program's loop through the public binding
(paper_1309_6275_gb300.ht, .learned, .displaced): device or pinned host hits
in, candidates, assignments, scores and fitted values out.  Sizes, parameters
and event mixes are the workloads of synth/configs.py (64^3 cells and ~275
hits, 256 x 128 x 512 cells and 2k-60k hits, 512 x 256 x 1024 cells and 50k
hits, displaced jets).

Every result of the transform is a whole number that the definition fixes
(vote counts, candidate cells, hit indices), so it has no nearer value than
itself; `exact` covers the computed numbers: the refinement's fits and the
training step's probabilities, gradients and updated state.
"""
import math

import numpy as np
import torch

import synth
from paper_1309_6275_gb300 import displaced, ht, learned

# candidate slots per event, by accumulator geometry (the densest events of
# the ranges below give about half of it)
CAP = {"single_64": 1 << 14, "event100_256": 1 << 18, "stream2000_256": 1 << 18,
       "pileup_512": 1 << 19, "jets4_256": 1 << 16}


def _case(name, kind, workload, events, lo, hi, **more):
    return dict(name=name, kind=kind, workload=workload, events=events, hits_lo=lo, hits_hi=hi,
                **more)


def listed():
    return [
        # one sparse event, every call of the path: a trigger's latency
        _case("plain_event_64", "plain_event", "single_64", 1, 0, 0, phi0=64),
        # the same event on the track path (layer vote, confirmation)
        _case("tracks_event_64", "tracks_event", "single_64", 1, 0, 0, phi0=64),
        # the swept-interval vote's use: a sparse event on four times the columns
        _case("swept_event_256", "swept_event", "single_64", 1, 0, 0, phi0=256),
        # the first example of the README: one ~10k-hit event, call by call
        _case("plain_event_10k", "plain_event", "event100_256", 1, 10000, 10000),
        # batches of ~10k-hit events on the track path
        _case("tracks_batch_10k", "tracks_batch", "event100_256", 25, 10000, 10000),
        # the stream the benchmark times: 2k-60k hits, a threshold per event
        _case("tracks_batch_stream", "tracks_batch", "stream2000_256", 25, 2000, 60000),
        # pile-up: few events, large accumulators
        _case("tracks_batch_pileup", "tracks_batch", "pileup_512", 2, 50000, 50000),
        # the stream with the learned per-hit proposal restricting the vote
        _case("tracks_batch_learned", "learned_batch", "stream2000_256", 25, 2000, 60000),
        # the stream end to end through host buffers
        _case("tracks_host_stream", "tracks_host", "stream2000_256", 25, 2000, 60000),
        # plain batch plus the second transform: displaced jets of ~400 hits
        _case("jets_batch", "jets_batch", "jets4_256", 25, 0, 0),
        # refinement of ~10k-hit events' tracks
        _case("refit_batch", "refit", "event100_256", 25, 10000, 10000),
        # one minibatch of the proposal's training (eight ~10k-hit events)
        _case("train_step", "train", "event100_256", 8, 10000, 10000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plain_event", "plain_event", "tracks_event", "tracks_event",
                       "swept_event", "plain_batch", "tracks_batch", "tracks_batch",
                       "tracks_batch", "learned_batch", "tracks_host", "jets_batch", "refit",
                       "train"])
    if kind in ("plain_event", "tracks_event"):
        if rng.random() < 0.5:
            return _case("", kind, "single_64", 1, 0, 0, phi0=32 * rng.randint(2, 8))
        n = _log(rng, 1500, 40000)
        return _case("", kind, "event100_256", 1, n, n)
    if kind == "swept_event":
        return _case("", kind, "single_64", 1, 0, 0, phi0=32 * rng.randint(2, 8))
    if kind in ("jets_batch",):
        return _case("", kind, "jets4_256", _log(rng, 1, 25), 0, 0)
    if kind in ("refit", "train"):
        n = _log(rng, 2000, 12000)
        return _case("", kind, "event100_256", rng.randint(1, 8 if kind == "train" else 25), n, n)
    if kind == "tracks_batch" and rng.random() < 0.25:
        n = _log(rng, 5000, 50000)
        return _case("", kind, "pileup_512", rng.randint(1, 2), n, n)
    lo = _log(rng, 2000, 20000)
    return _case("", kind, "stream2000_256", _log(rng, 1, 12), lo, _log(rng, lo, 60000))


# ------------------------------------------------------------------ inputs
def _hit_targets(case, rng):
    """The events' hit counts, log-uniform on the case's range: the middles of
    as many equal parts of it as there are events, in random order, so that
    the batches of a case hold the same number of hits."""
    if case["hits_hi"] <= 0:
        return [None] * case["events"]
    a, b = math.log(case["hits_lo"]), math.log(case["hits_hi"])
    n = case["events"]
    return [int(round(math.exp(a + (b - a) * (v + 0.5) / n))) for v in rng.permutation(n)]


def _cut(ev, n):
    """The event's first n hits (they are in random order; the generator ends
    with the track that passes the target)."""
    for k in ("x", "y", "z", "layer", "track"):
        setattr(ev, k, getattr(ev, k)[:n])
    ev.n_track_hits = np.bincount(ev.track[ev.track >= 0], minlength=len(ev.rho))
    return ev


def _events(case, seed):
    gen = synth.CONFIGS[case["workload"]]["gen"]
    rng = np.random.Generator(np.random.Philox(seed))
    seeds = [int(s) for s in rng.integers(0, 1 << 31, case["events"])]
    if gen.get("kind") == "jets":
        return [synth.make_jet_event(gen, s) for s in seeds]
    return [_cut(synth.make_event(gen, s, target_hits=t), t)
            for s, t in zip(seeds, _hit_targets(case, rng))]


def _max_hits(case, n):
    """Hits a handle is made for: those of a batch of fixed size, else the most
    that the mix can give (10 layers, tracks and noise)."""
    if case["hits_hi"] > 0:
        return n
    gen = synth.CONFIGS[case["workload"]]["gen"]
    tracks = gen["n_jets"] * gen["tracks_per_jet"] if gen.get("kind") == "jets" else gen["n_tracks"]
    return case["events"] * int(math.ceil(10 * tracks * (1.0 + gen["noise_frac"])))


def _hits(evs):
    off = np.zeros(len(evs) + 1, np.int32)
    off[1:] = np.cumsum([e.n_hits for e in evs])
    x, y, z = (np.concatenate([getattr(e, k) for e in evs]) for k in "xyz")
    return off, x, y, z, np.concatenate([e.layer for e in evs]).astype(np.uint8)


def _dev(*arrays):
    return tuple(torch.from_numpy(a).cuda() for a in arrays)


def _geometry(case, tracks):
    w = case["workload"]
    g = synth.track_geometry(w) if tracks else synth.geometry_of(w)
    if "phi0" in case:
        g["n_phi0"] = case["phi0"]
    return g


# -------------------------------------------------------- tracks to refine
def _truth_candidates(case, seed):
    """The candidates a perfect track path would confirm: per event, each
    track with at least 7 hits and its cell off the axes' edges, in cell
    order, and each hit's candidate."""
    g = synth.geometry_of(case["workload"])
    out = []
    for ev in _events(case, seed):
        i = np.floor((ev.rho + g["rho_max"]) / (2.0 * g["rho_max"] / g["n_rho"]))
        j = np.floor(ev.d0 * g["n_d0"] / (2.0 * g["d0_half"]) + g["n_d0"] / 2 + 0.5)
        k = np.floor((ev.phi0 + math.pi) * g["n_phi0"] / (2.0 * math.pi)) % g["n_phi0"]
        ok = (ev.n_track_hits >= 7) & (i >= 0) & (i < g["n_rho"]) & (j >= 0) & (j < g["n_d0"])
        t = np.flatnonzero(ok)
        t = t[np.lexsort((k[t], j[t], i[t]))]
        rank = np.full(len(ev.rho) + 1, -1)   # the last entry: noise hits (track -1)
        rank[t] = np.arange(len(t))
        pk = np.stack([i[t], j[t], k[t], ev.n_track_hits[t]], 1).astype(np.int32)
        out.append((ev, pk, rank[ev.track].astype(np.int32)))
    return g, out


# the road holds every hit of a track whose cell is the candidate (half a
# cell is up to 1.2 cm at 110 cm)
FIT = dict(min_hits=4, iters=5, sigma=20e-4, road=1.5, cut=5.0, iters2=3)


def _fit_views(out):
    """An ht_track record's fields: six float64, chi2, then whole numbers."""
    return dict(p=out.view(torch.float64).view(-1, 8)[:, :6],
                chi2=out.view(torch.float32).view(-1, 16)[:, 12],
                whole=out.view(torch.int32).view(-1, 16)[:, 13:])


# --------------------------------------------------------- training inputs
LR, B1, B2, EPS, STEP0 = 2e-3, 0.9, 0.999, 1e-8, 1000


def _train_inputs(case, seed):
    """A minibatch and the state of a training run under way: the shipped
    weights, moments of the size its gradients have."""
    evs = _events(case, seed)
    g = synth.geometry_of(case["workload"])
    _, x, y, z, lay = _hits(evs)
    lab = np.concatenate([learned.labels_of(g, e) for e in evs]).astype(np.int32)
    params = learned.load_weights(learned.default_weights_path())[0]
    rng = np.random.Generator(np.random.Philox(seed + 1))
    m = (1e-3 * rng.standard_normal(params.size)).astype(np.float32)
    v = (1e-6 * (0.5 + rng.random(params.size))).astype(np.float32)
    return x, y, z, lay, lab, params, m, v


# ----------------------------------------------------------------- prepare
def prepare(case, seed):
    kind, w = case["kind"], case["workload"]
    cap = CAP[w]
    st = dict(kind=kind)
    if kind == "train":
        x, y, z, lay, lab, params, m, v = _train_inputs(case, seed)
        t = learned.Trainer(max_hits=len(x), lr=LR, beta1=B1, beta2=B2, eps=EPS)
        t.load_state(dict(params=params, m=m, v=v, step=STEP0))
        st.update(trainer=t, hits=_dev(x, y, z, lay, lab))
        return st
    if kind == "refit":
        g, evs = _truth_candidates(case, seed)
        off, x, y, _, _ = _hits([e for e, _, _ in evs])
        cap = case["hits_hi"] // 8
        peaks = np.zeros((len(evs), cap, 4), np.int32)
        for e, (_, pk, _) in enumerate(evs):
            peaks[e, :len(pk)] = pk
        n = torch.tensor([len(pk) for _, pk, _ in evs], dtype=torch.int32).cuda()
        st.update(G=ht.Geometry(g), cap=cap, counts=n,
                  hits=_dev(x, y, off, np.concatenate([a for _, _, a in evs])),
                  peaks=torch.from_numpy(peaks.reshape(-1, 4)).cuda(),
                  out=torch.zeros(len(evs) * cap * 64, dtype=torch.uint8, device="cuda"),
                  ws=torch.empty(ht.ht_fit_workspace_size(len(evs), cap, len(x)),
                                 dtype=torch.uint8, device="cuda"))
        return st
    evs = _events(case, seed)
    off, x, y, z, lay = _hits(evs)
    n = _max_hits(case, int(off[-1]))
    tracks = kind in ("tracks_event", "tracks_batch", "tracks_host", "learned_batch")
    if kind == "jets_batch":
        vd = synth.CONFIGS[w]["vertex"]
        p = displaced.DisplacedJetPipeline(synth.geometry_of(w), vd, len(evs), n, cap=cap)
        p.V.peaks.zero_()
        st.update(pipe=p, batch=p.B, hits=_dev(x, y, z), off=off)
    elif kind in ("plain_event", "swept_event", "tracks_event"):
        G = ht.Geometry(_geometry(case, tracks))
        p = ht.EventPipeline(G, n, cap)
        p.peaks.zero_()
        p.zres.zero_()
        p.assign.zero_()
        st.update(G=G, pipe=p, hits=_dev(x, y, z))
        if tracks:
            st.update(conf=synth.track_of(w), layer=_dev(lay)[0],
                      score=torch.zeros(cap, dtype=torch.int32, device="cuda"),
                      inliers=torch.zeros((cap, 16), dtype=torch.int32, device="cuda"),
                      ws=torch.empty(max(p.workspace.numel(), ht.ht_confirm_workspace_size(G, n, cap)),
                                     dtype=torch.uint8, device="cuda"))
    else:
        G = ht.Geometry(_geometry(case, tracks))
        b = ht.Batch(G, max_events=len(evs), max_hits=n, cap=cap)
        st.update(G=G, batch=b, off=off)
        if tracks:
            b.set_confirm(synth.learned_of(w)["track"] if kind == "learned_batch"
                          else synth.track_of(w))
        if kind == "tracks_host":
            st.update(hits=tuple(torch.from_numpy(a).pin_memory() for a in (x, y, z, lay)),
                      tracks=torch.zeros((len(evs) * 16384, 8), dtype=torch.int32).pin_memory(),
                      ntracks=torch.zeros(len(evs), dtype=torch.int32),
                      assign=torch.zeros(n, dtype=torch.int32).pin_memory())
        else:
            st.update(hits=_dev(x, y, z, lay) if tracks else _dev(x, y, z))
        if kind == "learned_batch":
            st.update(params=learned.bf16_params(learned.load_weights(learned.default_weights_path())[0]),
                      topk=synth.learned_of(w)["topk"],
                      masks=torch.zeros(n, dtype=torch.int64, device="cuda"))
    if "batch" in st:
        b = st["batch"]
        b.peaks.zero_()      # slots past an event's count are not written
        b.zres.zero_()
        b.assign.zero_()
    return st


# --------------------------------------------------------------------- run
def _votes(stats):
    # the counters' even entries: votes cast (the odd ones count evaluations
    # that were repeated in a wider type, which says how, not what)
    return stats[0::2]


def _batch_outputs(b, **more):
    return dict(peaks=b.peaks, counts=b.counts, assign=b.assign, zres=b.zres,
                votes=_votes(b.stats), **more)


def run(st):
    kind = st["kind"]
    if kind in ("plain_event", "swept_event"):
        p = st["pipe"]
        p.run(*st["hits"], swept=kind == "swept_event")
        return dict(acc=p.acc, peaks=p.peaks, count=p.count, assign=p.assign, zres=p.zres,
                    votes=_votes(p.stats))
    if kind == "tracks_event":
        G, p, ws = st["G"], st["pipe"], st["ws"]
        x, y, z = st["hits"]
        assign = p.assign[:x.numel()]
        ht.ht_vote_layers(G, x, y, st["layer"], p.acc, p.stats)
        ht.ht_find_peaks(G, p.acc, p.peaks, p.cap, p.count, ws)
        ht.ht_confirm(G, st["conf"], x, y, st["layer"], p.peaks, p.count, p.cap, st["score"],
                      st["inliers"], assign, ws)
        ht.ht_vote_z(G, x, y, z, assign, p.peaks, p.count, p.cap, p.zres, ws)
        return dict(acc=p.acc, peaks=p.peaks, count=p.count, assign=p.assign, zres=p.zres,
                    votes=_votes(p.stats), score=st["score"], inliers=st["inliers"])
    if kind == "plain_batch":
        b = st["batch"]
        b.run(*st["hits"], st["off"])
        return _batch_outputs(b)
    if kind == "tracks_batch":
        b = st["batch"]
        b.run_tracks(*st["hits"], st["off"])
        return _batch_outputs(b, score=b.score)
    if kind == "learned_batch":
        b = st["batch"]
        b.run_tracks(*st["hits"], st["off"], params_bf16=st["params"], hit_masks=st["masks"],
                     topk=st["topk"])
        return _batch_outputs(b, score=b.score, masks=st["masks"])
    if kind == "tracks_host":
        if not st["batch"].run_tracks_host(*st["hits"], st["off"], st["tracks"], st["ntracks"],
                                           st["assign"]):
            raise RuntimeError("more tracks than slots")
        return dict(tracks=st["tracks"], ntracks=st["ntracks"], assign=st["assign"])
    if kind == "jets_batch":
        p = st["pipe"]
        p.run(*st["hits"], st["off"])
        v = p.V
        return _batch_outputs(p.B, vacc=v.acc, vpeaks=v.peaks, vcounts=v.counts, vfirst=v.first,
                              vvotes=_votes(v.stats))
    if kind == "refit":
        x, y, off, assign = st["hits"]
        ht.ht_fit_tracks(st["G"], x, y, off, assign, st["peaks"], st["counts"], st["cap"],
                         st["out"], st["ws"], **FIT)
        return _fit_views(st["out"])
    t = st["trainer"]
    t.step(*st["hits"])
    return dict(prob=t.prob, grad=t.grad, params=t.P, m=t.M, v=t.V)


# -------------------------------------------------------------------- work
def work(case):
    """Inputs read once and outputs written once (candidate lists, whose
    length the hits decide, are left out), and the operations: for each hit
    its azimuth terms in every column (3 products and sums for s and c each)
    and one comparison per accumulator cell; the fit's sums; the training
    step's matrix products."""
    w = case["workload"]
    gen = synth.CONFIGS[w]["gen"]
    g = _geometry(case, False)
    per = (math.sqrt(case["hits_lo"] * case["hits_hi"]) if case["hits_lo"] == case["hits_hi"]
           else (case["hits_hi"] - case["hits_lo"]) /
           math.log(case["hits_hi"] / case["hits_lo"])) if case["hits_hi"] > 0 else \
        (275 if gen.get("kind") != "jets" else 400)
    n = per * case["events"]
    kind = case["kind"]
    if kind == "train":
        return {"bytes": n * (17 + 256) + 4 * 25664 * 7.0, "flops": n * 25344 * 2 * 3.0}
    if kind == "refit":
        return {"bytes": n * 12 + n / 11 * (16 + 64), "flops": n * 40 * 11.0}
    cells = g["n_rho"] * g["n_d0"] * g["n_phi0"]
    b = n * (12 + 4)
    if kind not in ("plain_event", "swept_event", "plain_batch", "jets_batch"):
        b += n                                         # layers
    if kind in ("plain_event", "swept_event", "tracks_event"):
        b += cells * g["count_bits"] / 8               # the accumulator is an output
    if kind == "learned_batch":
        b += n * 8                                     # region sets
    flops = n * g["n_phi0"] * 6.0 + cells * case["events"]
    if kind == "learned_batch":
        flops += n * 25344 * 2.0
    return {"bytes": float(b), "flops": float(flops)}


# ------------------------------------------------------------------- exact
def _residuals(p, x, y):
    rho, d0, phi0 = (p[:, q, None] for q in range(3))
    sn, cs = np.sin(phi0), np.cos(phi0)
    s, c, r2 = x * sn - y * cs, x * cs + y * sn, x * x + y * y
    F = rho * d0 * d0 + 2.0 * (1.0 + rho * s) * d0 + rho * r2 + 2.0 * s
    J = np.stack([0.5 * (d0 * d0 + 2.0 * s * d0 + r2), rho * d0 + 1.0 + rho * s,
                  (1.0 + rho * d0) * c], -1)
    return 0.5 * F, J


def _normal(p, x, y, keep):
    r, J = _residuals(p, x, y)
    r, J = r * keep, J * keep[..., None]
    return r, np.einsum("mha,mhb->mab", J, J), np.einsum("mha,mh->ma", J, r)


def _exact_refit(case, seed):
    """Gauss-Newton of every candidate at once, hits padded per candidate."""
    g, evs = _truth_candidates(case, seed)
    cap = case["hits_hi"] // 8
    p_all = np.zeros((len(evs), cap, 6))
    chi_all = np.zeros((len(evs), cap), np.float64)
    whole = np.zeros((len(evs), cap, 3), np.int32)
    for e, (ev, pk, asg) in enumerate(evs):
        m = len(pk)
        order = np.flatnonzero(asg >= 0)
        order = order[np.argsort(asg[order], kind="stable")]
        cnt = np.bincount(asg[order], minlength=m)
        first = np.cumsum(cnt) - cnt
        col = np.arange(len(order)) - first[asg[order]]
        x, y = np.zeros((m, cnt.max())), np.zeros((m, cnt.max()))
        have = np.zeros((m, cnt.max()), bool)
        x[asg[order], col], y[asg[order], col] = ev.x[order], ev.y[order]
        have[asg[order], col] = True
        p = np.stack([(2.0 * pk[:, 0] + 1 - g["n_rho"]) * g["rho_max"] / g["n_rho"],
                      (pk[:, 1] - 0.5 * g["n_d0"]) * (2.0 * g["d0_half"] / g["n_d0"]),
                      (2.0 * pk[:, 2] + 1 - g["n_phi0"]) * math.pi / g["n_phi0"]], 1)
        keep = have & (np.abs(_residuals(p, x, y)[0]) <= FIT["road"])
        if (keep.sum(1) < FIT["min_hits"]).any():
            return None
        for it in range(FIT["iters"] + FIT["iters2"]):
            if it == FIT["iters"]:
                keep = have & (np.abs(_residuals(p, x, y)[0]) <= FIT["cut"] * FIT["sigma"])
                if (keep.sum(1) < FIT["min_hits"]).any():
                    return None
            _, A, gr = _normal(p, x, y, keep)
            p = p - np.linalg.solve(A, gr[..., None])[..., 0]
        r, A, _ = _normal(p, x, y, keep)
        cov = np.linalg.inv(A) * FIT["sigma"] ** 2
        p_all[e, :m, :3] = p
        p_all[e, :m, 3:] = np.sqrt(np.einsum("maa->ma", cov))
        chi_all[e, :m] = (r * r).sum(1) / FIT["sigma"] ** 2
        whole[e, :m, 0], whole[e, :m, 1] = keep.sum(1), 1
    return dict(p=p_all.reshape(-1, 6), chi2=chi_all.reshape(-1), whole=whole.reshape(-1, 3))


def _bf16(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).to(torch.bfloat16).to(
        torch.float64).numpy()


def _exact_train(case, seed):
    """The network in float64 with parameters, features and hidden layers
    rounded to BF16; mean cross entropy; one Adam step."""
    x, y, z, lay, lab, params, m, v = _train_inputs(case, seed)
    q, sizes, at = _bf16(params), [(6, 128), (128, 128), (128, 64)], 0
    W = []
    for i, o in sizes:
        W.append((q[at:at + i * o].reshape(i, o), q[at + i * o:at + i * o + o]))
        at += i * o + o
    f32 = np.float32
    zs = f32(110.0) * f32(math.sinh(2.5))
    f = _bf16(np.stack([x / f32(110), y / f32(110), z / zs, np.sqrt(x * x + y * y) / f32(110),
                        np.arctan2(y, x) / f32(math.pi), lay.astype(f32) / f32(9)], 1))
    h1 = _bf16(np.maximum(f @ W[0][0] + W[0][1], 0.0))
    h2 = _bf16(np.maximum(h1 @ W[1][0] + W[1][1], 0.0))
    a = h2 @ W[2][0] + W[2][1]
    a = np.exp(a - a.max(1, keepdims=True))
    prob = a / a.sum(1, keepdims=True)
    use = lab >= 0
    d3 = prob * use[:, None]
    d3[np.flatnonzero(use), lab[use]] -= 1.0
    d3 /= max(int(use.sum()), 1)
    d2 = (d3 @ W[2][0].T) * (h2 > 0)
    d1 = (d2 @ W[1][0].T) * (h1 > 0)
    grad = np.concatenate([t.reshape(-1) for t in (f.T @ d1, d1.sum(0), h1.T @ d2, d2.sum(0),
                                                   h2.T @ d3, d3.sum(0))])
    m = B1 * m.astype(np.float64) + (1 - B1) * grad
    v = B2 * v.astype(np.float64) + (1 - B2) * grad * grad
    t = STEP0 + 1
    P = params.astype(np.float64) - LR * (m / (1 - B1 ** t)) / (np.sqrt(v / (1 - B2 ** t)) + EPS)
    return dict(prob=prob, grad=grad, params=P, m=m, v=v)


def exact(case, seed):
    if case["kind"] == "refit":
        return _exact_refit(case, seed)
    if case["kind"] == "train":
        return _exact_train(case, seed)
    return None
