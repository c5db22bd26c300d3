"""The decoder's ball table and islands at the edges of their range, against the
oracle: events far apart (regions that grow past the table's radius, so that the
shot goes over to explored balls), islands past one and two events per lane, level-1 radii below, at and beyond what a list
holds, circuit-level weights, and both execution modes, for every team size.
Results are whole numbers and must be equal.  Needs a GB300."""

import numpy as np
import pytest

from oracle import OracleGraph
from synth import pack_defects, rotated_surface_code, rotated_surface_code_circuit, sample_shots, unpack_defects
from tests.test_gpu_diag import COL, FIELDS, qd, run  # noqa: F401

pytestmark = pytest.mark.gpu


def far_apart(pg, shots, seed):
    """Rows of 1 to 8 events at random places."""
    rng = np.random.default_rng(seed)
    return np.stack([pack_defects(rng.choice(pg.num_detectors, size=1 + i % 8, replace=False), pg.num_detectors)
                     for i in range(shots)])



CASES = [
    # (graph, level-1 override in edges (d1, b1), shots sampled or far apart)
    ("d5_far", rotated_surface_code(5, 5, 0.003), None, "far"),
    ("d13_far", rotated_surface_code(13, 13, 0.003), None, "far"),
    ("d11_weights_far", rotated_surface_code(11, 11, p_range=(0.001, 0.02), p_seed=4), None, "far"),
    ("d13_p01", rotated_surface_code(13, 13, 0.01), None, "sampled"),
    ("circuit_d9", rotated_surface_code_circuit(9, 9, 0.002), None, "sampled"),
    ("circuit_d7_far", rotated_surface_code_circuit(7, 7, 0.001), None, "far"),
    # islands of more events than a warp has lanes, of more than two per lane,
    # and batches whose other shots leave them to the overflow pass
    ("circuit_d13_dense", rotated_surface_code_circuit(13, 13, 0.0025), None, "sampled"),
    ("d15_dense", rotated_surface_code(15, 15, 0.012), None, "sampled"),
    # 3 and 6 edges: more vertices within b_1 than a first level-1 ball was
    # ever enumerated for; 9 edges: more than a list of the table holds
    ("b1_3_edges", rotated_surface_code(13, 13, 0.001), (1, 3), "sampled"),
    ("b1_6_edges", rotated_surface_code(15, 15, 0.001), (2, 6), "sampled"),
    ("b1_9_edges", rotated_surface_code(17, 17, 0.001), (3, 9), "sampled"),
]


@pytest.mark.parametrize("team", [1, 4, 16])
@pytest.mark.parametrize("name,pg,level1,kind", CASES, ids=[c[0] for c in CASES])
def test_ball_table_edges(qd, team, name, pg, level1, kind):  # noqa: F811
    kw = {}
    if level1:
        w = 2 * int(pg.w.max())
        kw = {"d1": level1[0] * w + 1, "b1": level1[1] * w + 1 + level1[0]}
    shots = 24
    syn = far_apart(pg, shots, 5) if kind == "far" else sample_shots(pg, shots, 6)[0]
    g, og = qd.Graph.from_phys(pg, **kw), OracleGraph.from_phys(pg, **kw)
    qd.set_tuning(team_warps=team)
    try:
        for mode in ("hier", "global"):
            Wt, O, S, D = run(qd, [g], syn, mode)
            for i in range(shots):
                r = og.diag(unpack_defects(syn[i], pg.num_detectors), mode)
                got = (int(Wt[i]), int(O[i]), int(S[i]))
                assert got == (r["weight"], r["obs"], r["status"]), (name, mode, i)
                if r["clusters_above_l1"] <= 1:
                    assert tuple(int(D[i, COL[f]]) for f in FIELDS) == tuple(int(r[f]) for f in FIELDS), (name, mode, i)
    finally:
        qd.set_tuning(team_warps=-1)


# windows of a sliding decode at rates where events at the open end stand alone,
# with boundaries within (d = 13) and beyond (d = 21) the table's reach
WINDOWS = [("d13", 13, 26, 13, dict(p=0.003)), ("d15", 15, 30, 15, dict(p=0.003)), ("d15_short", 15, 18, 9, dict(p=0.001)),
           ("d21", 21, 42, 21, dict(p=0.001)), ("d17_weights", 17, 34, 17, dict(p_range=(0.001, 0.004), p_seed=3))]


@pytest.mark.parametrize("team", [1, 16])
@pytest.mark.parametrize("name,d,W,C,kw", WINDOWS, ids=[c[0] for c in WINDOWS])
def test_window_tables(qd, team, name, d, W, C, kw):  # noqa: F811
    import torch
    from oracle.window import sliding_window_decode
    from paper_2609_12262_gb300.window import SlidingWindow
    pg = rotated_surface_code(d, W + C, **kw)
    shots = 10
    syn = sample_shots(pg, shots, 9)[0]
    qd.set_tuning(team_warps=team)
    try:
        dec = SlidingWindow(qd.Graph.from_phys(pg), pg.nz, W, C)
        obs, st = dec.decode(torch.from_numpy(syn.view(np.int32).reshape(-1)).cuda(), shots)
        torch.cuda.synchronize()
        ro, rs = sliding_window_decode(pg, syn, W, C)
        assert np.array_equal(st.cpu().numpy(), rs) and np.array_equal(qd.to_uint64(obs), ro)
    finally:
        qd.set_tuning(team_warps=-1)
