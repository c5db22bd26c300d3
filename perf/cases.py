"""Timed cases of the decoder: what a user has it do, through its public Python entry points.

A case is one call (or one request loop) on syndromes sampled on the GPU from the seed:

  batch   decode_batch: offline decoding of a batch of shots, of one graph or of several distances mixed;
          with one shot it is a real-time caller that waits for a single window
  diag    decode_batch_ex with the per-shot diagnostics (the parallel event count study)
  stream  SlidingWindow.decode: long histories decoded window by window with carried defects
  serve   Stream: a burst of windows in host memory, submitted and polled until all are back

Graphs are the rotated surface code's under phenomenological noise (one probability, or one per edge drawn from
[p, p_hi]) or circuit-level noise, at the distances and rates of the benchmark, the studies and the tests.
Outputs are whole numbers: the observables, the matching weights and the status of every shot.
"""

import functools
import math

import numpy as np
import torch

import paper_2609_12262_gb300 as qec
from paper_2609_12262_gb300.window import SlidingWindow
from synth import rotated_surface_code, rotated_surface_code_circuit

PHENOM, UNIFORM, PHYSICAL = "phenomenological", "uniform", "physical"


def _case(kind, d, shots, p, *, d_hi=0, d_step=2, rounds=0, noise=PHENOM, p_hi=0.0, commit=0, name=None):
    """d .. d_hi: the distances mixed in one call (d_hi = 0: d alone); rounds = 0: d noisy rounds; shots: per call,
    over all distances; commit: layers committed per window (windows are twice as long)."""
    c = {"kind": kind, "d": d, "d_hi": d_hi or d, "d_step": d_step, "rounds": rounds, "shots": shots, "p": p,
         "p_hi": p_hi, "noise": noise, "commit": commit}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a real-time caller with one window in hand, an own weight per edge as a calibrated device has it: a small
        # code (launches and latency count) ...
        _case("batch", 11, 1, 0.002, p_hi=0.006, name="one_d11"),
        # ... the largest window of the serving mix ...
        _case("batch", 25, 1, 0.002, p_hi=0.004, name="one_d25"),
        # ... and the largest window of the scaling study
        _case("batch", 51, 1, 0.003, name="one_d51"),
        # the smallest benchmark configuration: many tiny shots in one call
        _case("batch", 5, 10000, 0.005, name="batch_d5"),
        # the non-uniform benchmark configuration: an own probability, hence weight, per edge
        _case("batch", 11, 100000, 0.002, p_hi=0.006, name="batch_d11_weights"),
        # the headline batch: a million shots, d = 7 .. 21 mixed
        _case("batch", 7, 1000000, 0.003, d_hi=21, name="batch_mixed"),
        # batches of large windows (the per-round scaling study): one warp per window, and block-wide teams
        _case("batch", 31, 3000, 0.003, name="batch_d31"),
        _case("batch", 51, 1200, 0.003, name="batch_d51"),
        # the event-count study on the graph of the full syndrome-extraction circuit
        _case("diag", 13, 1024, 0.001, noise=UNIFORM, name="diag_circuit_d13"),
        # stored histories decoded in sliding windows (the stream study)
        _case("stream", 11, 20000, 0.003, rounds=110, commit=11, name="stream_d11"),
        # the live histories of a few logical qubits, window after window
        _case("stream", 21, 16, 0.003, rounds=210, commit=21, name="stream_live_d21"),
        # a burst of requests of the serving mix (d = 9, 13, .. 25)
        _case("serve", 9, 2000, 0.003, d_hi=25, d_step=4, name="serve_mix"),
    ]


def _events(d, p):
    """Detection events of a shot of d rounds, about."""
    return 2.94 * p * d ** 3


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(("batch", "batch", "batch", "batch", "diag", "stream", "serve"))
    p = round(_log(rng, 0.001, 0.005), 5)
    if kind == "serve":
        return _case(kind, rng.choice((5, 7, 9)), rng.randint(200, 4000), p, d_hi=rng.choice((15, 21, 25)),
                     d_step=rng.choice((2, 4)))
    if kind == "stream":
        d = rng.choice((5, 7, 9, 11, 13, 15))
        live = rng.random() < 0.3
        return _case(kind, d, rng.randint(8, 64) if live else int(_log(rng, 20, 2000)), p,
                     rounds=rng.randint(4 * d, 10 * d), commit=rng.randint(d // 2 + 1, d + 2))
    if kind == "diag":
        noise = rng.choice((PHENOM, UNIFORM, PHYSICAL))
        p = round(_log(rng, 2e-4, 1e-3), 6)
        return _case(kind, rng.choice((5, 7, 9, 11, 13)), rng.randint(100, 1024), p, noise=noise)
    form = rng.choice(("one", "one", "same", "same", "mixed", "weights"))
    if form == "one":
        p = max(p, 0.002)
        return _case(kind, rng.randrange(11, 53, 2), rng.choice((1, 1, 2, 7)), round(p / 2, 5), p_hi=round(3 * p / 2, 5))
    if form == "mixed":
        lo = rng.randrange(5, 15, 2)
        return _case(kind, lo, int(_log(rng, 500, 200000)), p, d_hi=lo + 2 * rng.randint(1, 5))
    d = int(_log(rng, 5, 52)) // 2 * 2 + 1
    most = 2e8 / (20 + _events(d, p)) ** 1.8   # below the headline batch's time
    shots = int(_log(rng, 20, min(300000.0, most)))
    if form == "weights":
        return _case(kind, d, shots, round(p / 2, 5), p_hi=round(3 * p / 2, 5))
    return _case(kind, d, shots, p)


@functools.lru_cache(maxsize=16)
def _phys(d, rounds, p, p_hi, noise):
    if noise != PHENOM:
        return rotated_surface_code_circuit(d, rounds or None, p, noise)
    if p_hi:
        return rotated_surface_code(d, rounds or None, p_range=(p, p_hi), p_seed=1)
    return rotated_surface_code(d, rounds or None, p)


def _physical_graphs(case):
    return [_phys(d, case["rounds"], case["p"], case["p_hi"], case["noise"])
            for d in range(case["d"], case["d_hi"] + 1, case["d_step"])]


def _syndromes(pg, shots, gen):
    """Syndrome rows of `shots` independent shots, int32 [shots, words] on the GPU: every physical edge flips with
    its own probability (geometric gaps at the largest probability, thinned to each edge's), and a detector is set
    when an odd number of its edges flipped."""
    dev = gen.device
    m, top = len(pg.u), float(np.max(pg.p))
    cells = shots * m
    n = int(cells * top + 12 * math.sqrt(cells * top + 1) + 32)
    u = 1.0 - torch.rand(n, generator=gen, device=dev, dtype=torch.float64)
    at = torch.cumsum(torch.floor(torch.log(u) / math.log1p(-top)).to(torch.int64) + 1, 0) - 1
    if float(np.min(pg.p)) < top:
        keep = torch.from_numpy(np.asarray(pg.p, np.float64) / top).to(dev)
        at = at[at < cells]
        at = at[torch.rand(at.numel(), generator=gen, device=dev, dtype=torch.float64) < keep[at % m]]
    else:
        at = at[at < cells]
    shot, edge = torch.div(at, m, rounding_mode="floor"), at % m
    a = torch.from_numpy(pg.u.astype(np.int64)).to(dev)[edge]
    b = torch.from_numpy(pg.v.astype(np.int64)).to(dev)[edge]
    base = shot * (pg.words * 32)
    bits = torch.cat([base + a, (base + b)[b >= 0]])
    bits, count = torch.unique(bits, return_counts=True)
    bits = bits[count % 2 == 1]
    rows = torch.zeros(shots * pg.words, dtype=torch.int64, device=dev)
    rows.index_add_(0, bits >> 5, torch.ones_like(bits) << (bits & 31))
    rows = torch.where(rows >= 1 << 31, rows - (1 << 32), rows).to(torch.int32)
    return rows.view(shots, pg.words)


def _mixed(pgs, shots, gen):
    """Shots of several graphs in one shuffled batch: (graph of shot int32, row offset int64, rows int32)."""
    dev = gen.device
    gid = torch.arange(shots, device=dev) * len(pgs) // shots
    gid = gid[torch.randperm(shots, generator=gen, device=dev)]
    words = torch.tensor([g.words for g in pgs], device=dev)[gid]
    off = torch.cumsum(words, 0) - words
    syn = torch.zeros(int(words.sum()), dtype=torch.int32, device=dev)
    for i, pg in enumerate(pgs):
        mine = off[gid == i]
        if mine.numel():
            rows = _syndromes(pg, mine.numel(), gen)
            syn[mine[:, None] + torch.arange(pg.words, device=dev)] = rows
    return gid.to(torch.int32), off, syn


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    pgs = _physical_graphs(case)
    state = {"kind": case["kind"], "shots": case["shots"], "graphs": [qec.Graph.from_phys(g) for g in pgs],
             "gid": None, "off": None}
    if len(pgs) > 1:
        state["gid"], state["off"], state["syn"] = _mixed(pgs, case["shots"], gen)
    else:
        state["syn"] = _syndromes(pgs[0], case["shots"], gen).view(-1)
    if case["kind"] == "stream":
        state["window"] = SlidingWindow(state["graphs"][0], pgs[0].nz, 2 * case["commit"], case["commit"])
    if case["kind"] == "serve":   # requests arrive in host memory
        state["gid"] = state["gid"].cpu().numpy()
        state["off"] = state["off"].cpu().numpy()
        state["syn"] = state["syn"].cpu().numpy().view(np.uint32)
        state["ids"] = np.arange(case["shots"], dtype=np.uint64)
        state["stream"] = qec.Stream(device_budget_bytes=6 << 30, max_inflight=16384)
    return state


def _serve(state):
    stream, n = state["stream"], state["shots"]
    obs, weight, status = np.zeros(n, np.uint64), np.zeros(n, np.int64), np.full(n, -1, np.int32)
    sent = back = 0
    while back < n:
        if sent < n:
            sent += stream.submit_many(state["graphs"], state["gid"][sent:], state["off"][sent:], state["syn"],
                                       state["ids"][sent:])
        r = stream.poll()
        if len(r):
            k = r["request_id"].astype(np.int64)
            obs[k], weight[k], status[k] = r["obs"], r["weight"], r["status"]
            back += len(r)
    return obs.view(np.int64), weight, status


def run(state):
    kind = state["kind"]
    if kind == "serve":
        return _serve(state)
    if kind == "stream":
        return state["window"].decode(state["syn"], state["shots"])
    if kind == "diag":
        return qec.decode_batch_ex(state["graphs"], state["syn"], state["gid"], state["off"],
                                   num_shots=state["shots"])
    return qec.decode_batch(state["graphs"], state["syn"], state["gid"], state["off"], num_shots=state["shots"])


def work(case):
    """Each syndrome row and each graph (two endpoints, weight and observable per edge) read once, each output
    written once.  Decoding is integer work on per-shot state that is no input or output: no flops are counted."""
    pgs = _physical_graphs(case)
    rows = sum(4 * g.words for g in pgs) / len(pgs) * case["shots"]
    if case["kind"] == "stream":
        out = 12
    else:
        out = 20 + (32 if case["kind"] == "diag" else 0)
    if len(pgs) > 1:
        out += 12   # graph index and row offset of every shot, read
    return {"bytes": rows + out * case["shots"] + sum(20 * len(g.u) for g in pgs), "flops": 0}


def _exact_weight(dist, edge_of, events):
    """Smallest total weight that matches `events` in pairs or with the boundary, over all subsets."""
    k = len(events)
    best = [math.inf] * (1 << k)
    best[0] = 0
    for s in range(1, 1 << k):
        i = s.bit_length() - 1
        rest = s ^ (1 << i)
        b = best[rest] + edge_of[events[i]]
        for j in range(i):
            if rest >> j & 1:
                b = min(b, best[rest ^ (1 << j)] + dist[events[i], events[j]])
        best[s] = b
    return best[-1]


def exact(case, seed):
    """The matching weights of small shots by exhaustive pairing on all-pairs shortest distances.  The observables
    of equally light matchings differ, so they have no value of their own; every status is 0."""
    if case["kind"] != "batch" or case["d_hi"] > 5 or case["shots"] > 20000 or max(case["p"], case["p_hi"]) > 0.006:
        return None
    pg = _physical_graphs(case)[0]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    rows = _syndromes(pg, case["shots"], gen).cpu().numpy().view(np.uint8)
    bits = np.unpackbits(rows, axis=1, bitorder="little")
    n = pg.num_detectors
    dist = np.full((n, n), np.inf)
    np.fill_diagonal(dist, 0)
    side = np.full(n, np.inf)
    for u, v, w in zip(pg.u, pg.v, pg.w):
        if v < 0:
            side[u] = min(side[u], w)
        else:
            dist[u, v] = dist[v, u] = min(dist[u, v], w)
    for k in range(n):   # paths do not pass through the boundary
        dist = np.minimum(dist, dist[:, k:k + 1] + dist[k:k + 1, :])
    side = np.min(dist + side[None, :], axis=1)
    events = [np.nonzero(b)[0] for b in bits]
    if max(map(len, events)) > 16:
        return None
    weight = np.array([_exact_weight(dist, side, e) for e in events], np.float64)
    return None, weight.astype(np.int64), np.zeros(case["shots"], np.int32)
