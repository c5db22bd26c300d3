"""Islands that meet after one of them was joined with something else: shots of a close pair and a lone event on
either side of it, where that happens often, in hierarchical against global mode (which knows no islands).  Both
give the same matching, so weights and observables are equal.  Needs a GB300."""

import numpy as np
import pytest

from synth import rotated_surface_code
from tests.test_gpu_diag import qd, run  # noqa: F401

pytestmark = pytest.mark.gpu


def pairs_with_lone_events(pg, shots, seed):
    rng = np.random.default_rng(seed)
    inner = pg.v >= 0
    near = [[] for _ in range(pg.num_detectors)]
    for a, b in zip(pg.u[inner], pg.v[inner]):
        near[a].append(b)
        near[b].append(a)
    degree = np.array([len(x) for x in near])
    table = np.zeros((pg.num_detectors, degree.max()), np.int64)
    for i, x in enumerate(near):
        table[i, :len(x)] = x

    def walk(x, steps):
        for k in range(steps.max()):
            y = table[x, rng.integers(0, degree[x])]
            x = np.where(k < steps, y, x)
        return x

    a = rng.integers(0, pg.num_detectors, shots)
    b = walk(a, np.ones(shots, int))
    events = [a, b, walk(a, np.full(shots, 3)), walk(b, rng.integers(3, 6, shots))]
    rows = np.zeros((shots, pg.words), np.uint32)
    for e in events:   # an event met twice is none
        rows[np.arange(shots), e >> 5] ^= np.uint32(1) << (e & 31).astype(np.uint32)
    return rows


@pytest.mark.parametrize("team,shots", [(1, 100000), (4, 20000), (16, 20000)])
def test_joined_islands_equal_global_mode(qd, team, shots):  # noqa: F811
    pg = rotated_surface_code(13, 13, p_range=(0.001, 0.02), p_seed=1)
    g = qd.Graph.from_phys(pg)
    syn = pairs_with_lone_events(pg, shots, 100 + team)
    qd.set_tuning(team_warps=team)
    try:
        hier, glob = run(qd, [g], syn, "hier"), run(qd, [g], syn, "global")
        for x, y in zip(hier[:3], glob[:3]):
            assert np.array_equal(x, y), np.nonzero(x != y)[0][:5]
    finally:
        qd.set_tuning(team_warps=-1)


def chain(rng, n):
    """A path between two boundaries, with a boundary edge at some detectors in between."""
    u, v = list(range(n - 1)) + [0, n - 1], list(range(1, n)) + [-1, -1]
    side = rng.choice(n, size=int(rng.integers(0, 4)), replace=False).tolist()
    return n, u + side, v + [-1] * len(side)


def tree(rng, n):
    u = list(range(1, n))
    v = [int(rng.integers(max(0, i - 5), i)) for i in u]
    side = rng.choice(n, size=int(rng.integers(1, 5)), replace=False).tolist()
    return n, u + side, v + [-1] * len(side)


def grid(rng, n):
    a = int(rng.integers(3, 7))
    b = n // a
    at = np.arange(a * b).reshape(a, b)
    u = np.concatenate([at[:-1].ravel(), at[:, :-1].ravel(), at[:, 0], at[:, -1]]).tolist()
    v = np.concatenate([at[1:].ravel(), at[:, 1:].ravel(), np.full(2 * a, -1)]).tolist()
    return a * b, u, v


@pytest.mark.parametrize("team", [1, 4, 16])
@pytest.mark.parametrize("kind", [chain, tree, grid], ids=["chain", "tree", "grid"])
def test_sparse_shots_of_small_graphs_equal_the_oracle(qd, kind, team):  # noqa: F811
    """Without diagnostics, where clusters of more events have closed forms too."""
    import torch
    from oracle import OracleGraph
    from synth import pack_defects
    rng = np.random.default_rng(team)
    qd.set_tuning(team_warps=team)
    try:
        for wmax in (1, 5, 30, 100) * 2:
            n, u, v = kind(rng, int(rng.integers(30, 60)))
            w = rng.integers(max(1, wmax // 3), wmax + 1, len(u))
            o = [0 if b >= 0 else 1 << (i % 2) for i, b in enumerate(v)]
            near = [[] for _ in range(n)]
            for a, b in zip(u, v):
                if b >= 0:
                    near[a].append(b)
                    near[b].append(a)
            rows = []
            for _ in range(1000):
                x, events = int(rng.integers(0, n)), set()
                for _ in range(int(rng.integers(2, 8))):
                    events ^= {x}
                    for _ in range(int(rng.integers(1, 6))):
                        x = int(rng.choice(near[x]))
                rows.append(pack_defects(np.array(sorted(events), int), n))
            rows = np.stack(rows)
            g, og = qd.Graph(n, u, v, w, o, num_observables=2), OracleGraph(n, u, v, w, o)
            obs, weight, status = qd.decode_batch([g], torch.from_numpy(rows.view(np.int32).reshape(-1)).cuda())
            torch.cuda.synchronize()
            rw, ro, rs = og.decode_bitmaps(rows, "hier")
            got = status.cpu().numpy(), weight.cpu().numpy(), qd.to_uint64(obs)
            for x, y in zip(got, (rs, rw, ro)):
                assert np.array_equal(x, y), (wmax, np.nonzero(x != y)[0][:5])
    finally:
        qd.set_tuning(team_warps=-1)
