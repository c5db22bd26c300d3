"""The kernels on the host emulation of tests/emulation.py (no GPU), against the oracle.

The lanes of a warp run in any order between two warp wide operations there: results that need a wait that is not
written down differ, fault or never end.  Results are whole numbers and must be equal."""

import pytest

from tests import emulation

DECODE = """
import numpy as np, torch
from oracle import OracleGraph
from synth import *
from tests import emulation
q = emulation.load(order=%(order)d)
def check(pg, shots, mode, team, split=1, seed=5, **kw):
    g, og = q.Graph.from_phys(pg, **kw), OracleGraph.from_phys(pg, **kw)
    syn, _ = sample_shots(pg, shots, seed)
    q.set_tuning(team_warps=team, team_split_events=split)
    o, w, s, _ = q.decode_batch_ex([g], torch.from_numpy(syn.view(np.int32).reshape(-1)), mode=mode, diag=False,
                                   stream=emulation.STREAM)
    rw, ro, rs = og.decode_bitmaps(syn, mode)
    assert np.array_equal(s.numpy(), rs) and np.array_equal(w.numpy(), rw) and np.array_equal(q.to_uint64(o), ro)
"""


@pytest.mark.parametrize("order", [0, 1, 2], ids=["ascending", "descending", "random"])
def test_islands_with_blossoms_in_any_lane_order(order):
    emulation.run(DECODE % {"order": order} + """
check(rotated_surface_code(11, 11, 0.01), 60, "hier", 1)
check(rotated_surface_code(9, 9, p_range=(0.001, 0.02), p_seed=1), 60, "hier", 4)
""", timeout=300)


@pytest.mark.parametrize("order", [0, 1, 2], ids=["ascending", "descending", "random"])
def test_general_path_of_one_warp_in_any_lane_order(order):
    emulation.run(DECODE % {"order": order} + """
check(rotated_surface_code(7, 7, 0.01), 40, "global", 1)
check(rotated_surface_code(9, 9, p_range=(0.001, 0.02), p_seed=1), 20, "global", 1)
check(rotated_surface_code(7, 7, 0.01), 20, "global", 16, split=20)   # the first warp of a block
""", timeout=300)


def test_walks_over_an_island_end_on_a_broken_tree():
    # two nodes that are each other's tree parent (or blossom), which no event leaves behind: the walk gives up
    emulation.program("""
#include <cstdio>
using namespace qec;
static Isl<1> I;
static void clear() {
    memset(&I, 0, sizeof I);
    memset(I.tpar, -1, sizeof I.tpar);
    memset(I.bpar, -1, sizeof I.bpar);
}
int main() {
    clear();
    I.tpar[0] = 1; I.tpar[1] = 2; I.tpar[2] = 1;
    isl_flip(I, 0);
    if (!I.err) return 1;
    clear();
    I.bpar[3] = 40; I.bpar[40] = 41; I.bpar[41] = 40; I.bpar[5] = 41;
    isl_child_of(I, 50, 3);
    isl_dist(I, 3, 5);
    clear();
    I.tpar[0] = 1; I.tpar[1] = 0; I.tpar[6] = 7; I.tpar[7] = 6;
    static int ok[32];
    emu::launch(1, 32, [&] { ok[threadIdx.x] = isl_blossom(I, 32, 0, 0, 6, 6, 8, 0, threadIdx.x); });
    for (int l = 0; l < 32; l++) if (ok[l]) return 2;
    // and the ordinary case still works: 0 -> inner 1 -> root 2
    clear();
    I.tpar[0] = 1; I.tpar[1] = 2; I.tps[1] = 1; I.tpo[1] = 2; I.tps[0] = 0; I.tpo[0] = 1;
    isl_flip(I, 0);
    return I.err || I.mate[1] != 2 || I.mate[2] != 1;
}
""")


# (user weights of the edges between boundary, the named events and boundary; weight and observable of the matching):
# an island that stands met nothing while its neighbour was small, and is met once that one has been joined and grown
JOINS = [([[100, 100], [100, 100, 10], [100], [100, 100, 100, 20], [100, 100, 50]], 530, 0),
         ([[50, 50], [50, 50, 5], [50], [50, 50, 50, 10], [50, 50, 25]], 265, 0),
         ([[40, 40, 40, 45], [50, 50, 50], [50], [40, 40, 40, 35], [40, 40, 30]], 305, 0)]

JOIN_CODE = """
def decode(g, events, mode, diag):
    row = pack_defects(np.asarray(events), g.num_detectors)
    o, w, s, _ = q.decode_batch_ex([g], torch.from_numpy(row.view(np.int32)), mode=mode, diag=diag, num_shots=1,
                                   stream=emulation.STREAM)
    return int(w[0]), int(q.to_uint64(o)[0]), int(s[0])
pg = rotated_surface_code(13, 13, p_range=(0.001, 0.02), p_seed=1)
surface = q.Graph.from_phys(pg)
for team in (1, 4, 16):
    q.set_tuning(team_warps=team)
    for diag in (False, True):
        for segments, weight, obs in %r:
            u, v, w, o, named, at, n = [], [], [], [], [], -1, sum(map(len, segments)) - 1
            for segment in segments:
                for x in segment:
                    u.append(max(at, 0)), v.append(-1 if at < 0 or at == n - 1 else at + 1)
                    if at < 0: o.append(1)
                    else: o.append(0)
                    w.append(x)
                    at += 1
                named.append(at)
            g = q.Graph(n, u, v, w, o)
            for mode in ("hier", "global"):
                got = decode(g, named[:-1], mode, diag)
                assert got == (weight, obs, 0), (team, diag, mode, segments, got)
        for events, weight in (([409, 552, 559, 625], 587), ([551, 731, 736, 754], 502), ([55, 115, 139, 157], 541)):
            assert decode(surface, events, "hier", diag) == (weight, 0, 0), (team, diag, events)
"""


def test_an_island_that_stands_is_met_by_a_joined_one():
    emulation.run(DECODE % {"order": 0} + JOIN_CODE % (JOINS,))


def test_batches_outside_the_fast_path_stay_with_their_warps():
    # one block takes what a warp leaves to the second pass, with some hundred barriers per shot; a batch whose every
    # shot is outside the fast path's limits (by its mode or band) keeps its warps
    emulation.run(DECODE % {"order": 0} + """
def barriers(*a, **kw):
    before = q.lib().emu_barriers()
    check(*a, **kw)
    return q.lib().emu_barriers() - before
pg, shots = rotated_surface_code(7, 7, 0.01), 60
few = barriers(pg, shots, "hier", 1)
assert few < 10 * shots, few
assert barriers(pg, shots, "global", 1) < 10 * shots
q.set_tuning(band_factor=2)
assert barriers(pg, shots, "hier", 1) < 10 * shots
""")


def test_the_route_of_a_joined_shot_does_not_depend_on_the_order_of_lanes_or_warps():
    # b reached its boundary, is joined with x and ends smaller; a is joined with the pair c, d at the same time and
    # would stop where b's first radius was
    emulation.run(DECODE % {"order": 0} + """
u, v, w, o, place = [], [], [], [], {}
def detector(name=None):
    if name not in place or name is None:
        place[name if name else len(place)] = len(place)
    return place[name] if name else len(place) - 1
for a, b, length in (("a", "d", 150), ("d", "c", 50), ("c", None, 35), ("a", None, 200), ("a", "b", 230),
                     ("b", None, 100), ("b", "x", 150), ("x", None, 80)):
    at, end = detector(a), detector(b) if b else -1
    while length > 0:
        nxt = end if length <= 50 else detector()
        u.append(at), v.append(nxt), w.append(min(length, 50)), o.append(0)
        at, length = nxt, length - 50
g = q.Graph(len(place), u, v, w, o)
row = torch.from_numpy(pack_defects(sorted(place[k] for k in "abcdx"), len(place)).view(np.int32))
for team in (1, 4, 16):
    q.set_tuning(team_warps=team)
    barriers = set()
    for order in range(5):
        q.lib().emu_order(order, 7)
        before = q.lib().emu_barriers()
        _, weight, status = q.decode_batch([g], row, num_shots=1, stream=emulation.STREAM)
        barriers.add(q.lib().emu_barriers() - before)
        assert (int(weight[0]), int(status[0])) == (335, 0), (team, order, weight, status)
    assert len(barriers) == 1 and max(barriers) < 60, (team, barriers)
""")


def test_replacing_a_commit_region_waits_for_the_device():
    emulation.run(DECODE % {"order": 0} + """
g = q.Graph.from_phys(rotated_surface_code(5, 5, 0.003))
region = np.full(g.words, 0xffff, np.uint32)
g.set_commit_region(region)
for new in (region * 3, None):
    before = q.lib().emu_syncs()
    g.set_commit_region(new)
    assert q.lib().emu_syncs() == before + 1
""")


def test_a_commit_region_that_could_not_be_made_is_none():
    emulation.run(DECODE % {"order": 0} + """
g = q.Graph.from_phys(rotated_surface_code(5, 5, 0.003))
region = np.full(g.words, 0xffff, np.uint32)
rows = torch.ones(g.words, dtype=torch.int32)
def decode():
    obs, carry, status = torch.zeros(1, dtype=torch.int64), torch.empty_like(rows), torch.zeros(1, dtype=torch.int32)
    q.decode_window_batch([g], rows, obs, carry, status, num_shots=1, stream=emulation.STREAM)
    assert int(status[0]) == 0
for n in (1, 2):
    q.lib().emu_fail_alloc(n)
    for call in (lambda: g.set_commit_region(region), decode):
        try:
            call()
        except q.QecError:
            continue
        raise AssertionError(n)
g.set_commit_region(region)
decode()
""")


def test_distances_along_chains_of_heavy_edges():
    # equal to a heap's on random graphs, from one start and from several, and quick where distances are long
    emulation.program("""
#include <chrono>
#include <random>
static void graph(int n, const std::vector<std::array<int, 3>> &edges, std::vector<int> &row, std::vector<Slot> &slots) {
    row.assign((size_t)n + 1, 0);
    for (auto &e : edges) { row[(size_t)e[0] + 1]++; row[(size_t)e[1] + 1]++; }
    for (int x = 0; x < n; x++) row[(size_t)x + 1] += row[(size_t)x];
    slots.resize(2 * edges.size() + 1);
    std::vector<int> at(row);
    for (auto &e : edges) {
        slots[(size_t)at[(size_t)e[0]]++] = Slot{e[1], e[2]};
        slots[(size_t)at[(size_t)e[1]]++] = Slot{e[0], e[2]};
    }
}
int main() {
    std::mt19937 rng(1);
    std::vector<int> row;
    std::vector<Slot> slots;
    for (int trial = 0; trial < 300; trial++) {
        const int n = 2 + (int)(rng() % 200), w = 1 + (int)(rng() % (trial % 3 ? 100 : 65535));
        std::vector<std::array<int, 3>> edges;
        for (int i = 0; i < n * (int)(1 + rng() % 3); i++) {
            const int a = (int)(rng() % (unsigned)n), b = (int)(rng() % (unsigned)n);
            if (a != b) edges.push_back({a, b, 1 + (int)(rng() % (unsigned)w)});
        }
        graph(n, edges, row, slots);
        Distances ring(row, slots, w), heap(row, slots, 1 << 16);
        std::vector<long long> a((size_t)n, LLONG_MAX), b;
        std::vector<int> starts;
        for (int x = 0; x < n; x++)
            if (rng() % 8 == 0 || x == 0) { a[(size_t)x] = (long long)(rng() % 100000u); starts.push_back(x); }
        b = a;
        ring.run(a, starts);
        heap.run(b, starts);
        if (a != b) return 1;
    }
    const int n = 16000, w = 65534;
    std::vector<std::array<int, 3>> edges;
    for (int i = 0; i + 1 < n; i++) edges.push_back({i, i + 1, w});
    graph(n, edges, row, slots);
    Distances D(row, slots, w);
    std::vector<long long> dist((size_t)n);
    const auto t = std::chrono::steady_clock::now();
    D.from(0, dist);
    if (dist[(size_t)n - 1] != (long long)w * (n - 1)) return 2;
    return std::chrono::duration<double>(std::chrono::steady_clock::now() - t).count() < 0.5 ? 0 : 3;
}
""".replace("#include <chrono>", "#include <array>\n#include <chrono>"), source="capi.cpp")


def test_the_event_budget_of_closed_forms():
    # six level-1 clusters of three events that all reach the boundary: each budget gives the status that the run over
    # everything gives, which counts 5 steps per cluster and one at the end
    emulation.run(DECODE % {"order": 0} + """
u, v, w, o = [], [], [], []
for c in range(6):
    for x, y, weight in ((0, 1, 50), (1, 2, 50), (0, 2, 50), (0, None, 10), (1, None, 11), (2, None, 12)):
        u.append(3 * c + x), v.append(-1 if y is None else 3 * c + y), w.append(weight), o.append(0)
g = q.Graph(18, u, v, w, o)
row = torch.from_numpy(pack_defects(list(range(18)), 18).view(np.int32))
q.set_tuning(team_warps=1)
for budget in range(1, 70):
    q.set_tuning(max_events=budget)
    for diag in (False, True):
        _, weight, status, _ = q.decode_batch_ex([g], row, num_shots=1, diag=diag, stream=emulation.STREAM)
        assert int(status[0]) == (q.SHOT_OK if budget >= 31 else q.SHOT_BUDGET_EXCEEDED), (budget, diag)
""")


def test_equal_windows_share_one_graph():
    # eight windows: all but the last, which has another commit region, are equal where the
    # edges have one weight, and all differ where each edge has its own
    emulation.run(DECODE % {"order": 0} + """
from oracle.window import sliding_window_decode
from paper_2609_12262_gb300.window import SlidingWindow
for kw, graphs in (({"p": 0.01}, 2), ({"p_range": (0.005, 0.02), "p_seed": 2}, 8)):
    pg = rotated_surface_code(5, 44, **kw)
    syn, _ = sample_shots(pg, 8, 3)
    dec = SlidingWindow(q.Graph.from_phys(pg), pg.nz, 10, 5)
    assert len(dec.windows) == 8 and len({id(x[3]) for x in dec.windows}) == graphs
    obs, status = dec.decode(torch.from_numpy(syn.view(np.int32).reshape(-1)), 8, stream=emulation.STREAM)
    ro, rs = sliding_window_decode(pg, syn, 10, 5)
    assert np.array_equal(status.numpy(), rs) and np.array_equal(q.to_uint64(obs), ro)
""")


def test_a_radius_below_zero_ends_the_island():
    # two regions past the reach meet unnoticed, and an inner region between them shrinks below zero: the shot goes to
    # the run over everything at once, without steps on a state that no shot can be in (its times overflow)
    lib = emulation.build(out=emulation.OUT + "/checked",
                          flags=("-fsanitize=signed-integer-overflow", "-fno-sanitize-recover=all"))
    emulation.run((DECODE % {"order": 0}).replace("load(", "load(%r, " % lib) + """
pg = rotated_surface_code(11, 11, p_range=(0.001, 0.004), p_seed=3)
row = pack_defects([38, 162, 232, 237, 238, 412, 417], pg.num_detectors)[None, :]
g, og = q.Graph.from_phys(pg), OracleGraph.from_phys(pg)
for team in (1, 4, 16):
    q.set_tuning(team_warps=team)
    o, w, s = q.decode_batch([g], torch.from_numpy(row.view(np.int32)), num_shots=1, stream=emulation.STREAM)
    rw, ro, rs = og.decode_bitmaps(row, "hier")
    assert (int(w[0]), int(q.to_uint64(o)[0]), int(s[0])) == (rw[0], ro[0], rs[0])
""")


def test_events_joined_earlier_follow_their_component():
    # the pair that joined an event in one round is gone in the next: its label alone ties it to what it was joined with
    emulation.run(DECODE % {"order": 0} + """
for seed, events, weight in ((6, [195, 202, 531, 627, 634, 803, 904, 923, 1007, 1085], 893),
                             (9, [91, 210, 252, 295, 361, 379, 546, 649], 957),
                             (28, [555, 675, 712, 718, 723, 876, 927, 1011, 1031, 1052], 1052)):
    pg = rotated_surface_code(13, 13, p_range=(0.001, 0.02), p_seed=seed)
    g, row = q.Graph.from_phys(pg), torch.from_numpy(pack_defects(events, pg.num_detectors).view(np.int32))
    for team in (1, 4, 16):
        q.set_tuning(team_warps=team)
        for order in range(5):
            q.lib().emu_order(order, 3)
            _, w, status = q.decode_batch([g], row, num_shots=1, stream=emulation.STREAM)
            assert (int(w[0]), int(status[0])) == (weight, 0), (seed, team, order, int(w[0]))
""")


def test_level1_clusters_that_grow_into_each_other():
    # a cluster of three reaches its boundary later than b_1 / 2 and covers part of the next cluster's region
    emulation.run(DECODE % {"order": 0} + """
for pg, events in ((rotated_surface_code(9, 9, p_range=(0.0005, 0.1), p_seed=5), [77, 229, 232, 237]),
                   (rotated_surface_code(17, 17, p_range=(0.001, 0.05), p_seed=2), [1343, 1590, 1599, 1606]),
                   (rotated_surface_code(17, 17, p_range=(0.001, 0.05), p_seed=5), [928, 1337, 1344, 1353])):
    g, og, row = q.Graph.from_phys(pg), OracleGraph.from_phys(pg), pack_defects(events, pg.num_detectors)
    for team in (1, 4, 16):
        q.set_tuning(team_warps=team)
        for diag in (False, True):
            o, w, s, _ = q.decode_batch_ex([g], torch.from_numpy(row.view(np.int32)), num_shots=1, diag=diag,
                                           stream=emulation.STREAM)
            r = og.decode(events, "hier")
            assert r.touch_violations and (int(w[0]), int(q.to_uint64(o)[0]), int(s[0])) == (r.weight, r.obs, r.status)
""")


def test_two_wide_regions_that_know_each_other_too_late():
    # both are past the reach's cap where they meet, and one records the other only after that
    emulation.run(DECODE % {"order": 0} + """
for seed, events in ((3, [38, 98, 102, 114, 338, 502, 513, 573]), (4, [227, 299, 332, 432, 443, 503]),
                     (5, [23, 99, 154, 159, 202, 287, 332, 337]), (7, [136, 251, 311, 328, 334, 372, 388, 512])):
    pg = rotated_surface_code(11, 11, p_range=(0.002, 0.006), p_seed=seed)
    g, row = q.Graph.from_phys(pg), pack_defects(events, pg.num_detectors)[None, :]
    rw, ro, rs = OracleGraph.from_phys(pg).decode_bitmaps(row, "hier")
    for team in (1, 4, 16):
        q.set_tuning(team_warps=team)
        o, w, s = q.decode_batch([g], torch.from_numpy(row.view(np.int32)), num_shots=1, stream=emulation.STREAM)
        assert (int(w[0]), int(q.to_uint64(o)[0]), int(s[0])) == (rw[0], ro[0], rs[0]), (seed, team)
""")
