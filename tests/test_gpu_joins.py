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
