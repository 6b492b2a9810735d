"""GPU parity at the sizes where one kernel form gives way to another: tile
and list edges, remainders, and the smallest and largest of a form's range.
Every output is compared with the CPU oracle, whole numbers exactly."""
import numpy as np
import pytest
import torch

from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_06751_gb300 import build as B
    B.build()
    from paper_2606_06751_gb300 import stagefrontier
    return stagefrontier


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def host(t):
    return t.cpu().numpy()


# one tile of entries and one more, cluster sizes 1 to 8, lists that overflow
# (every entry positive) and sparse ones, ties across CTAs, k of 1 and 32
@pytest.mark.parametrize("nW,S,R,k", [(3, 1, 2048, 5), (2, 1, 2049, 32), (2, 2, 2049, 32), (1, 3, 5461, 7),
                                      (2, 8, 2049, 32), (1, 8, 8192, 32), (1, 5, 16385, 1)])
@pytest.mark.parametrize("positive", [1.0, 0.05, 0.0])
def test_topk_lists(sf, nW, S, R, k, positive):
    rng = np.random.default_rng(S * R + k)
    X = rng.integers(0, 4, size=(nW, S)).astype(np.int64)
    E = rng.integers(1, 50, size=(nW, S, R)).astype(np.int64) << 40
    E[rng.random(E.shape) >= positive] = 0
    o = O.topk(X, E, k)
    t = sf.sf_topk_suspects(dev(X), dev(E), k)
    assert np.array_equal(host(t.stage), o.stage) and np.array_equal(host(t.stage_value), o.stage_value)
    assert np.array_equal(host(t.pair), o.pair) and np.array_equal(host(t.pair_value), o.pair_value)


# windows shorter and longer than the gate kernel's 256 segments, up to 32
# stages, leaders that change within and across segments and unsure steps
@pytest.mark.parametrize("T,S,W", [(30, 2, 7), (600, 5, 255), (1025, 31, 512), (3000, 32, 3000), (700, 1, 256)])
def test_gates_switches(sf, T, S, W):
    rng = np.random.default_rng(T + S)
    d = rng.integers(1, 1000, size=(T, 2, S)).astype(np.int64)
    runs = np.repeat(rng.integers(0, S, size=T), rng.integers(1, 6, size=T))[:T]
    lead = rng.random(T) < 0.8
    d[np.nonzero(lead)[0], :, runs[lead]] += 50000
    o = O.label_windows(d, W)
    m = sf.sf_window_median(dev(d), W)
    ev = sf.sf_direct_gain(dev(d), W, m)
    g = sf.sf_label_gates(T, 2, S, W, ev)
    assert np.array_equal(host(g.n_confident), o.n_confident) and np.array_equal(host(g.n_switch), o.n_switch)
    for got, want in ((g.labels, o.labels), (g.route_mask, o.route_mask), (g.amb_mask, o.amb_mask)):
        assert np.array_equal(host(got).astype(np.uint32), want)
    assert np.array_equal(host(g.share), o.share) and np.array_equal(host(g.gain), o.gain)


# a warp per step and a CTA or a cluster of CTAs per step
@pytest.mark.parametrize("T,R,S", [(700, 512, 3), (700, 513, 8), (5, 64, 6), (1, 65, 16), (2, 2047, 5), (1, 8192, 8),
                                   (16, 8191, 4), (300, 4096, 2), (1, 65536, 3), (2500, 40, 20)])
def test_ties_splits(sf, T, R, S):
    d_np = np.random.default_rng(T + R).integers(0, 4, size=(T, R, S)).astype(np.int64)
    assert np.array_equal(host(sf.sf_frontier_ties(dev(d_np))), O.frontier(d_np).ties)


def durations(T, R, S, kind, seed):
    """ms work; `long`: steps around 2^32 ns, where 32-bit row sums end; `far`:
    one rank 2^31 ns and more from the others in some steps."""
    rng = np.random.default_rng(seed)
    d = np.rint(rng.uniform(1e6, 5e7, size=S) * np.exp(0.1 * rng.standard_normal((T, R, S)))).astype(np.int64)
    if kind == "long":
        total = d.sum(axis=2)
        edge = (1 << 32) - 1 + rng.integers(-2, 3, size=(T, R))
        pick = rng.random((T, R)) < 0.3
        d[..., S - 1] += np.where(pick, edge - total, 0)
    if kind == "far":
        t = np.nonzero(rng.random(T) < 0.3)[0]
        d[t, rng.integers(R, size=t.size), rng.integers(S, size=t.size)] += rng.integers(1 << 31, 1 << 34, size=t.size)
    if kind == "tail":
        d = np.rint(d * np.where(rng.random((T, R, 1)) < 0.01, 30.0, 1.0)).astype(np.int64)
    return d


# windows whose columns single lanes hold (where they are enough) and longer ones:
# rows of each form and one more, a short last window, odd column counts, columns
# whose values differ in their high words
@pytest.mark.parametrize("T,R,S,W", [(70, 3, 5, 16), (33, 7, 3, 32), (100, 5, 7, 33), (128, 31, 1, 64), (200, 9, 9, 65),
                                     (305, 11, 8, 100), (210, 33, 4, 104), (300, 13, 3, 105), (257, 16, 2, 128),
                                     (260, 16, 2, 129), (305, 200, 20, 100), (1000, 40, 2, 250), (1001, 6, 4, 500),
                                     (2000, 5, 2, 1000), (700, 3, 3, 300)])
@pytest.mark.parametrize("kind", ["ms", "far", "tail", "few", "words"])
def test_median_lanes(sf, T, R, S, W, kind):
    d_np = durations(T, R, S, kind, T + W)
    if kind == "words":  # most values share a high word, a few lie above and below, in row 0 of some columns too
        rng = np.random.default_rng(T)
        d_np += 1 << 32
        d_np[rng.random(d_np.shape) < 0.02] += 1 << 33
        d_np[rng.random(d_np.shape) < 0.02] -= 1 << 32
        d_np[0, ::3] += 1 << 33
    if kind == "few":
        d_np = np.random.default_rng(T).integers(0, 3, size=(T, R, S)).astype(np.int64) - 1
    assert np.array_equal(host(sf.sf_window_median(dev(d_np), W)), O.window_median(d_np, W))


# windows enough for a lane per column on 152 SMs: rows of each form and one more, columns
# for one tile of lanes and two, odd counts, a short last window; and one column, row or
# window to the other side of the lines
@pytest.mark.parametrize("T,R,S,W", [(9800, 4, 8, 16), (9740, 3, 20, 16), (9720, 16, 2, 32), (10100, 16, 4, 33), (19500, 31, 2, 64),
                                     (20001, 13, 5, 65), (31000, 5, 12, 100), (31650, 20, 4, 104), (32000, 19, 3, 105),
                                     (38930, 33, 3, 128), (77900, 8, 11, 128), (9760, 11, 3, 16), (9800, 1, 7, 16), (31000, 12, 2, 50),
                                     (31000, 10, 2, 50), (62000, 4, 4, 100), (60700, 5, 4, 100), (4615, 72, 8, 100), (21324, 8, 16, 100)])
@pytest.mark.parametrize("kind", ["ms", "words", "far"])
def test_median_lanes_many_windows(sf, T, R, S, W, kind):
    test_median_lanes(sf, T, R, S, W, kind)


# steps held on chip: keys per lane, per warp, the CTA form's columns in registers
# and in shared memory, the first ranks past each, columns in which every key falls
# into a few bins, and medians on both sides of the bracket
@pytest.mark.parametrize("T,R,S", [(40, 1, 4), (1, 1, 1), (40, 2, 2), (30, 32, 17), (30, 33, 17), (30, 64, 9), (30, 65, 16),
                                   (30, 128, 8), (30, 129, 8), (20, 256, 3), (20, 257, 4), (9, 1024, 2),
                                   (9, 4099, 1), (7, 1001, 13), (7, 2893, 8), (7, 2945, 8), (5, 700, 32),
                                   (40, 16, 8), (41, 17, 16), (30, 104, 10), (30, 105, 5), (33, 128, 32), (7, 2048, 9),
                                   (5, 2049, 1), (5, 2050, 2), (6, 2051, 3), (5, 4097, 5), (4, 8192, 8), (3, 9001, 16),
                                   (2, 16385, 12), (2, 32768, 8), (2, 4500, 32), (1, 65536, 8), (300, 3000, 4)])
@pytest.mark.parametrize("kind", ["ms", "long", "far", "tail", "halves"])
def test_rank_on_chip(sf, T, R, S, kind):
    d_np = durations(T, R, S, kind, T + R + S)
    if kind == "halves":  # ranks split into two far groups, lane by lane: empty and misleading brackets
        d_np[:, np.arange(R) % 32 < (R + S) % 32, 0] *= 9
    o = O.rank_lag(d_np)
    st = sf.new_status("cuda")
    g = sf.sf_rank_lag(dev(d_np), status=st)
    sp = sf.sf_raw_spread(dev(d_np), 4, t0=3, status=st)
    Lw, Gw = sf.sf_rank_lag_windows(dev(d_np), 4, t0=3, status=st)
    oL, oG = O.rank_lag_windows(d_np, 4, 3)
    assert int(st.item()) == 0
    assert np.array_equal(host(g.L), o.L) and np.array_equal(host(g.dL), o.dL) and np.array_equal(host(g.G), o.G)
    assert np.array_equal(host(sp), O.raw_spread(d_np, 4, 3))
    assert np.array_equal(host(Lw), oL) and np.array_equal(host(Gw), oG)


# the forms that take many steps (lanes, warps), and the lines between the others: stages
# and steps on both sides of each
@pytest.mark.parametrize("T,R,S", [(1600, 1, 4), (1519, 40, 3), (1520, 40, 3), (1600, 16, 8), (1601, 17, 16), (1700, 32, 17),
                                   (1600, 33, 17), (1600, 64, 9), (1600, 65, 16), (1600, 65, 8), (1600, 104, 10),
                                   (1530, 105, 32), (1600, 128, 8), (1600, 128, 9), (1600, 100, 5),
                                   (607, 300, 2), (608, 300, 2), (303, 1025, 3), (304, 1025, 3), (310, 2048, 4),
                                   (700, 1500, 1), (75, 1250, 9), (75, 1251, 9), (76, 2048, 9), (7, 2048, 7), (20, 1100, 6),
                                   (151, 2500, 6), (152, 2500, 6), (152, 2501, 6), (153, 2050, 11), (10, 2500, 4),
                                   (310, 2501, 4), (151, 6001, 3), (152, 6001, 3), (9, 6000, 3), (152, 2250, 9),
                                   (152, 2251, 9), (759, 16, 10), (760, 16, 10), (1064, 13, 8), (506, 9, 17), (507, 16, 17),
                                   (835, 64, 20), (836, 64, 20), (761, 96, 32)])
@pytest.mark.parametrize("kind", ["ms", "long", "far", "tail", "halves"])
def test_rank_forms(sf, T, R, S, kind):
    test_rank_on_chip(sf, T, R, S, kind)


# steps that are not whole 128-byte rows: every stage count, small steps (whole
# steps per tile) and steps of one or more tiles with one, two and four warp
# groups, a tensor and medians that end inside a row, tensors below one row;
# then whole-row steps around the limits between those forms
TILED = [(300, 31, 1, 70), (4000, 3, 2, 500), (200, 61, 3, 33), (50, 127, 4, 20), (90, 201, 5, 40), (33, 97, 6, 11),
         (500, 31, 7, 64), (40, 101, 8, 9), (77, 63, 9, 30), (31, 85, 10, 16), (64, 55, 11, 20), (25, 99, 12, 7),
         (80, 41, 13, 33), (22, 73, 14, 10), (45, 67, 15, 13), (3, 5, 1, 2), (1, 1, 1, 1), (2000, 1, 5, 300),
         (9, 9001, 1, 4), (7, 5001, 2, 3), (11, 1001, 3, 4), (9, 2001, 4, 4), (13, 1000, 5, 6), (8, 700, 6, 3),
         (10, 601, 7, 4), (9, 1001, 8, 4), (7, 2003, 9, 3), (6, 1701, 10, 4), (8, 333, 11, 3), (9, 501, 12, 5),
         (6, 2001, 13, 2), (7, 403, 14, 3), (5, 1555, 15, 2), (4, 32767, 3, 2),
         (40, 128, 8, 15), (40, 130, 8, 15), (30, 64, 16, 12), (12, 512, 8, 5), (12, 514, 8, 5), (9, 2048, 8, 4),
         (9, 96, 14, 4), (20, 192, 10, 6), (7, 1024, 16, 3)]


@pytest.mark.parametrize("T,R,S,W", TILED)
@pytest.mark.parametrize("kind", ["ms", "long"])
def test_tiled_passes(sf, T, R, S, W, kind):
    d_np = durations(T, R, S, kind, T + R + S)
    d, st = dev(d_np), sf.new_status("cuda")
    f, o = sf.sf_frontier(d, status=st), O.frontier(d_np)
    assert np.array_equal(host(f.a), o.a) and np.array_equal(host(f.lead), o.lead)
    assert np.array_equal(host(f.makespan), o.makespan)
    win, ow = sf.sf_window_aggregate(d, W, t0=1, status=st), O.windows(d_np, W, 1)
    assert np.array_equal(host(win.X), ow.X) and np.array_equal(host(win.E), ow.E)
    assert np.array_equal(host(win.C), ow.C) and np.array_equal(host(win.step_lead), ow.step_lead)
    b, ob = sf.sf_window_baselines(d, W, status=st), O.baselines(d_np, W)
    assert np.array_equal(host(b.M), ob.M) and np.array_equal(host(b.SLOW), ob.SLOW)
    assert np.array_equal(host(b.RANK0), ob.RANK0)
    assert np.array_equal(host(b.SUM.view(torch.int64))[..., 0], ob.SUM.astype(np.int64))
    m_np = O.window_median(d_np, W)
    ev, ow = sf.sf_direct_gain(d, W, dev(m_np), lead_credit=True, status=st), O.windows(d_np, W)
    assert np.array_equal(host(ev.X), ow.X) and np.array_equal(host(ev.Y), O.direct_gain(d_np, W, m_np))
    assert np.array_equal(host(ev.E), ow.E) and np.array_equal(host(ev.C), ow.C)
    wall = d_np.sum(axis=2) + 1000
    lab = sf.sf_label_windows(d, W, wall=dev(wall), other_stage=S - 1, status=st)
    ol = O.label_windows(d_np, W, wall=wall, other_stage=S - 1)
    assert np.array_equal(host(lab.labels).astype(np.uint32), ol.labels) and np.array_equal(host(lab.Y), ol.Y)
    assert int(st.item()) == 0


# few ranks: a lane per (step, stage), every scan depth, one to 32 groups in blocks
# and in any order, a group without ranks, the last rank count and one more, steps
# past 32 bits, a partial last tile and window
@pytest.mark.parametrize("T,R,S,G", [(20000, 7, 1, 2), (10001, 9, 2, 3), (5000, 40, 4, 1), (4001, 33, 7, 5),
                                     (2600, 65, 8, 32), (2001, 50, 13, 4), (1300, 192, 16, 3), (1300, 193, 16, 3),
                                     (700, 20, 24, 6), (650, 12, 32, 2)])
@pytest.mark.parametrize("kind", ["blocks", "mixed", "long"])
def test_group_lanes(sf, T, R, S, G, kind):
    d_np = durations(T, R, S, "long" if kind == "long" else "ms", T + R)
    rng = np.random.default_rng(T)
    group = np.sort(rng.integers(0, max(1, G - 1), size=R)) if kind == "blocks" else rng.integers(0, G, size=R)
    group = group.astype(np.int32)
    o = O.group_windows(d_np, group, G, 100, 3)
    st = sf.new_status("cuda")
    g = sf.sf_group_aggregate(dev(d_np), dev(group), G, 100, t0=3, status=st)
    assert int(st.item()) == 0
    assert np.array_equal(host(g.X), np.transpose(o.X, (1, 0, 2))) and np.array_equal(host(g.D), o.D.T)


# the same where the lanes have many tiles each: windows that end within a tile, the
# largest rank and group counts, stages in the lanes' every layout
@pytest.mark.parametrize("T,R,S,G", [(100001, 20, 1, 3), (60000, 192, 3, 2), (30000, 40, 4, 1), (40000, 65, 8, 32),
                                     (6000, 31, 10, 7), (12000, 50, 13, 4), (9000, 20, 24, 6)])
@pytest.mark.parametrize("kind", ["blocks", "mixed", "long"])
def test_group_lanes_many_steps(sf, T, R, S, G, kind):
    test_group_lanes(sf, T, R, S, G, kind)


# small steps: windows of a tile's 16 steps and one less and more, a short last
# window, a tile of ranks and one more, the largest small step and the next
@pytest.mark.parametrize("T,R,S,N", [(100, 16, 8, 16), (95, 31, 7, 15), (100, 47, 8, 17), (1000, 48, 8, 100),
                                     (77, 49, 8, 40), (333, 383, 1, 50), (200, 385, 1, 64), (64, 12, 32, 33),
                                     (40, 3, 3, 40), (19, 1, 1, 16), (30, 5, 4, 1 << 40)])
def test_gathered_tiles(sf, T, R, S, N):
    d = np.random.default_rng(T + R).integers(0, 1 << 62, size=(T, R, S), dtype=np.int64)
    g = np.concatenate([d[t:t + N].transpose(1, 0, 2).reshape(-1) for t in range(0, T, N)])
    out = torch.empty((T, R, S), dtype=torch.int64, device="cuda")
    sf.sf_gathered_to_steps(dev(g), T, R, S, N, dst=out)
    assert np.array_equal(host(out), d)


# the same with tiles for every SM: one tile short of that, the largest steps that go by
# tiles and the next ones, ranks in one tile and in equal and unequal shares of two
@pytest.mark.parametrize("T,R,S,N", [(2432, 5, 4, 16), (2416, 5, 4, 16), (3648, 16, 8, 16), (3632, 16, 8, 16), (2600, 31, 7, 17),
                                     (5000, 64, 4, 100), (5000, 65, 4, 100), (4000, 40, 8, 33), (4000, 42, 8, 33),
                                     (3700, 96, 1, 50), (9600, 97, 1, 50), (12200, 128, 1, 500), (2600, 127, 3, 40), (2600, 128, 3, 40),
                                     (2600, 129, 3, 40), (3100, 10, 32, 40), (5000, 53, 6, 500), (2500, 3, 3, 1 << 40)])
def test_gathered_tiles_everywhere(sf, T, R, S, N):
    test_gathered_tiles(sf, T, R, S, N)


# few steps of many ranks: odd stage counts, T at the SM count, at the most that are
# resident at once and past it, whole clusters and single CTAs per step, shares of
# 8192 ranks and more (four rows in flight), the fewest ranks and one less
@pytest.mark.parametrize("T,R,S", [(3, 1025, 3), (100, 5001, 5), (305, 1100, 7), (2, 9000, 9), (40, 1500, 11),
                                   (151, 1024, 8), (152, 1023, 8), (153, 1025, 8), (456, 1100, 8), (457, 1100, 8),
                                   (762, 1030, 4), (160, 2100, 10), (60, 16500, 12), (151, 2000, 14), (152, 2000, 14),
                                   (200, 1030, 13), (900, 1024, 2)])
@pytest.mark.parametrize("kind", ["ms", "long"])
def test_split_steps(sf, T, R, S, kind):
    d_np = durations(T, R, S, kind, T + R + S)
    d, st = dev(d_np), sf.new_status("cuda")
    f, o = sf.sf_frontier(d, status=st), O.frontier(d_np)
    assert np.array_equal(host(f.a), o.a) and np.array_equal(host(f.lead), o.lead)
    assert np.array_equal(host(f.makespan), o.makespan)
    win, ow = sf.sf_window_aggregate(d, 50, t0=7, status=st), O.windows(d_np, 50, 7)
    assert np.array_equal(host(win.X), ow.X) and np.array_equal(host(win.E), ow.E)
    assert np.array_equal(host(win.C), ow.C) and np.array_equal(host(win.step_lead), ow.step_lead)
    assert int(st.item()) == 0


# four and two rows in flight per thread, by stages, ranks and steps
@pytest.mark.parametrize("T,R,S", [(8, 1500, 2), (54, 1030, 4), (200, 1100, 8), (100, 8192, 8), (140, 1100, 10), (75, 2100, 12),
                                   (45, 1501, 12), (16, 1300, 16), (4, 33000, 6), (200, 1024, 7), (130, 1050, 14)])
@pytest.mark.parametrize("kind", ["ms", "long"])
def test_split_rows(sf, T, R, S, kind):
    test_split_steps(sf, T, R, S, kind)


# every stage count of its own kernel and those without, in steps of one and two
# rows of 256 ranks, more groups than the lanes take
@pytest.mark.parametrize("T,R,S", [(500, r, s) for s in (2, 3, 5, 7, 9, 11, 12, 13) for r in (256, 257, 513)])
def test_group_stages(sf, T, R, S):
    d_np = durations(T, R, S, "ms", R + S)
    group = np.sort(np.random.default_rng(S).integers(0, 33, size=R)).astype(np.int32)
    o = O.group_windows(d_np, group, 33, 90, 3)
    st = sf.new_status("cuda")
    g = sf.sf_group_aggregate(dev(d_np), dev(group), 33, 90, t0=3, status=st)
    assert int(st.item()) == 0
    assert np.array_equal(host(g.X), np.transpose(o.X, (1, 0, 2))) and np.array_equal(host(g.D), o.D.T)


# few steps: a step's ranks over a cluster of two, four and eight CTAs, in shares that
# end inside a group, groups in blocks and mixed
@pytest.mark.parametrize("T,R,S,G", [(1, 8191, 8, 64), (90, 8200, 6, 61), (150, 4097, 10, 33), (300, 2048, 4, 300),
                                     (20, 17000, 18, 130), (200, 2049, 16, 9), (7, 30001, 3, 3)])
@pytest.mark.parametrize("kind", ["blocks", "mixed", "long"])
def test_few_steps_groups(sf, T, R, S, G, kind):
    d_np = durations(T, R, S, "long" if kind == "long" else "ms", T + R)
    group = np.random.default_rng(T).integers(0, G, size=R)
    group = (group if kind == "mixed" else np.sort(group)).astype(np.int32)
    o = O.group_windows(d_np, group, G, 40, 3)
    st = sf.new_status("cuda")
    g = sf.sf_group_aggregate(dev(d_np), dev(group), G, 40, t0=3, status=st)
    assert int(st.item()) == 0
    assert np.array_equal(host(g.X), np.transpose(o.X, (1, 0, 2))) and np.array_equal(host(g.D), o.D.T)


# few steps of many ranks, moved in pieces: whole and ragged ones, odd and even stage
# counts, the fewest units that are split and one rank less, a short last window
@pytest.mark.parametrize("T,R,S,N", [(1, 8191, 8, 1), (90, 8200, 6, 40), (7, 30001, 3, 2), (400, 2048, 8, 150),
                                     (400, 2047, 8, 150), (20, 2731, 3, 7), (20, 2730, 3, 7)])
def test_gathered_pieces(sf, T, R, S, N):
    d = np.random.default_rng(T + R).integers(0, 1 << 62, size=(T, R, S), dtype=np.int64)
    g = np.concatenate([d[t:t + N].transpose(1, 0, 2).reshape(-1) for t in range(0, T, N)])
    out = torch.empty((T, R, S), dtype=torch.int64, device="cuda")
    sf.sf_gathered_to_steps(dev(g), T, R, S, N, dst=out)
    assert np.array_equal(host(out), d)


# columns in shared memory whose median lies in the last bins below 2^32, by their
# values and relative to rank 0: one to eight warps per column
@pytest.mark.parametrize("T,R,S", [(6, 4000, 3), (160, 2500, 6), (4, 9000, 2), (160, 2050, 11), (3, 11001, 1),
                                   (200, 3000, 4)])
@pytest.mark.parametrize("relative", [False, True])
@pytest.mark.parametrize("late", [1 << 23, 64])
def test_rank_bracket_at_word_end(sf, T, R, S, relative, late):
    rng = np.random.default_rng(T + R + S)
    d_np = rng.integers(0, 8, size=(T, R, S))
    top = (1 << 31 if relative else 1 << 32) - 8 * S - 1
    waits = rng.random((T, R)) < 0.25
    d_np[..., 0] = np.where(waits, rng.integers(top // 2, top * 3 // 4, size=(T, R)), top - rng.integers(late, size=(T, R)))
    if relative:
        d_np[:, 0, 0] = 0
        d_np[..., 0] += 1 << 33
    o = O.rank_lag(d_np)
    st = sf.new_status("cuda")
    g = sf.sf_rank_lag(dev(d_np), status=st)
    sp = sf.sf_raw_spread(dev(d_np), 4, t0=3, status=st)
    assert int(st.item()) == 0
    assert np.array_equal(host(g.L), o.L) and np.array_equal(host(g.dL), o.dL) and np.array_equal(host(g.G), o.G)
    assert np.array_equal(host(sp), O.raw_spread(d_np, 4, 3))


# medians that stay in shared memory, in one slot and in two: CTA ranges of 25 steps that
# start and end at every place of windows of 24 (on a window's last step, one step into the
# next), whole-row steps and ragged ones, without and with the quality sums
@pytest.mark.parametrize("R,S", [(512, 10), (1001, 5), (300, 10), (700, 12)])
def test_resident_medians_at_range_edges(sf, R, S):
    T, W = 25 * torch.cuda.get_device_properties(0).multi_processor_count, 24
    d_np = durations(T, R, S, "ms", R)
    d, m_np = dev(d_np), O.window_median(d_np, W)
    m, st = dev(m_np), sf.new_status("cuda")
    X, Y = O.windows(d_np, W).X, O.direct_gain(d_np, W, m_np)
    wall = dev(d_np.sum(axis=2) + 1000)
    for _ in range(8):
        ev = sf.sf_direct_gain(d, W, m, status=st)
        assert np.array_equal(host(ev.X), X) and np.array_equal(host(ev.Y), Y)
        ev = sf.sf_direct_gain(d, W, m, wall=wall, status=st)
        assert np.array_equal(host(ev.X), X) and np.array_equal(host(ev.Y), Y)
    assert int(st.item()) == 0


def evidence(d, W, wall=None, other=-1):
    """What sf_direct_gain reports beside the oracle's sums: the leader byte with its
    confidence at eta_Q = 1/20, and the quality sums (residual, overlap, wall)."""
    P = d.cumsum(axis=2)
    F = P.max(axis=1)
    a = np.diff(F, axis=1, prepend=0)
    best = a.argmax(axis=1)
    rest = a.copy()
    rest[np.arange(len(a)), best] = 0
    sure = (F[:, -1] > 0) & ((a.max(axis=1) - rest.max(axis=1)) * 20 >= F[:, -1])
    o = d[:, :, other] if other >= 0 else np.zeros(d.shape[:2], np.int64)
    if wall is None:
        sums = (o, np.zeros_like(o), P[:, :, -1])
    else:
        e = wall - (P[:, :, -1] - o)
        sums = (np.maximum(e, 0), np.maximum(-e, 0), wall)
    q = [[sum(map(int, x[t:t + W].sum(axis=1))) for x in sums] for t in range(0, len(d), W)]
    return (best | np.where(sure, 128, 0)).astype(np.uint8), q


def check_evidence(sf, d_np, W, options, place=dev):
    """Every form of the pass in `options` (wall, other_stage); place: medians to the device."""
    d, st = dev(d_np), sf.new_status("cuda")
    m_np, ow = O.window_median(d_np, W), O.windows(d_np, W)
    m, Y = place(m_np), O.direct_gain(d_np, W, m_np)
    for wall, other in options:
        ev = sf.sf_direct_gain(d, W, m, wall=None if wall is None else dev(wall), other_stage=other, lead_credit=True,
                               status=st)
        assert int(st.item()) == 0
        assert np.array_equal(host(ev.X), ow.X) and np.array_equal(host(ev.Y), Y) and np.array_equal(host(ev.D), ow.D)
        assert np.array_equal(host(ev.E), ow.E) and np.array_equal(host(ev.C), ow.C)
        lead, q = evidence(d_np, W, wall, other)
        assert np.array_equal(host(ev.step_lead), lead)
        if wall is not None or other >= 0:
            got = host(ev.quality.view(torch.int64)).astype(object) & ((1 << 64) - 1)
            assert [[int(w[2 * i]) | int(w[2 * i + 1]) << 64 for i in range(3)] for w in got] == q


def check_passes(sf, d_np, W):
    d, st = dev(d_np), sf.new_status("cuda")
    b, ob = sf.sf_window_baselines(d, W, status=st), O.baselines(d_np, W)
    s2 = host(b.SUM.view(torch.int64)).astype(object) & ((1 << 64) - 1)
    assert (s2[..., 0] + (s2[..., 1] << 64) == ob.SUM).all()
    assert np.array_equal(host(b.M), ob.M) and np.array_equal(host(b.SLOW), ob.SLOW)
    assert np.array_equal(host(b.RANK0), ob.RANK0)
    f, o = sf.sf_frontier(d, status=st), O.frontier(d_np)
    assert np.array_equal(host(f.a), o.a) and np.array_equal(host(f.lead), o.lead)
    assert np.array_equal(host(f.makespan), o.makespan) and int(st.item()) == 0
    g, ow = sf.sf_window_aggregate(d, W, status=st), O.windows(d_np, W)
    assert np.array_equal(host(g.X), ow.X) and np.array_equal(host(g.D), ow.D)
    assert np.array_equal(host(g.E), ow.E) and np.array_equal(host(g.C), ow.C) and int(st.item()) == 0


# either side of the lines between a warp, a CTA and a cluster of CTAs per step on 152 SMs
@pytest.mark.parametrize("T,R,S", [(607, 33, 3), (608, 128, 9), (700, 129, 20), (759, 340, 14), (760, 340, 20),
                                   (760, 341, 20), (760, 512, 9), (1823, 512, 8), (1824, 512, 7), (305, 600, 14),
                                   (456, 601, 9), (457, 600, 16), (20, 1151, 8), (20, 1152, 8), (75, 2500, 16), (9, 33, 32)])
def test_ties_forms(sf, T, R, S):
    d_np = np.random.default_rng(T + R).integers(0, 4, size=(T, R, S)).astype(np.int64)
    d_np[::3] += 1 << 31
    assert np.array_equal(host(sf.sf_frontier_ties(dev(d_np))), O.frontier(d_np).ties)


# few steps that are not whole 128-byte rows: a CTA per step up to 20 KB and 304 or 456
# steps, tiles above; fewer steps than a CTA has warp groups for, medians beside the tiles
@pytest.mark.parametrize("T,R,S,W", [(456, 640, 4, 100), (457, 640, 4, 100), (304, 319, 8, 304), (305, 319, 8, 100),
                                     (10, 2560, 1, 4), (10, 2561, 1, 4), (200, 171, 12, 50), (304, 285, 9, 100),
                                     (100, 1024, 8, 30), (153, 1024, 8, 153), (303, 700, 6, 7), (455, 641, 5, 100),
                                     (607, 600, 8, 100), (608, 600, 8, 100)])
@pytest.mark.parametrize("kind", ["ms", "long"])
def test_few_steps(sf, T, R, S, W, kind):
    d_np = durations(T, R, S, kind, T + R)
    check_evidence(sf, d_np, W, [(None, -1), (d_np.sum(axis=2) + 1000, S - 1)])
    check_passes(sf, d_np, W)


# steps enough for a lane per (step, stage): every scan depth, one to 16 steps a tile, a
# partial last tile and window, steps past 32 bits, sums past 64
LANES = [(20000, 3, 1, 999), (9001, 60, 2, 500), (6000, 7, 6, 250), (4000, 33, 13, 300), (3000, 100, 16, 3000),
         (2600, 64, 11, 2600), (1300, 12, 24, 100), (700, 9, 32, 64), (650, 130, 17, 50),
         # the most ranks that a pass takes by lanes, and the fewest steps
         (6000, 48, 6, 333), (9800, 48, 8, 700), (2600, 48, 11, 2600), (4000, 32, 13, 300), (4000, 16, 14, 250),
         (4900, 48, 16, 500), (1530, 96, 17, 50), (4600, 97, 17, 500), (2500, 130, 24, 100),
         (20000, 128, 1, 500), (20000, 192, 1, 999), (19500, 193, 1, 500), (9800, 96, 2, 333), (9800, 128, 2, 500),
         (6100, 128, 3, 100), (6500, 64, 4, 999), (5000, 100, 4, 500), (4900, 101, 4, 700),
         (39000, 128, 2, 1000), (48700, 49, 3, 999), (45700, 17, 10, 5000),
         (620, 40, 17, 100), (620, 41, 17, 100), (1000, 128, 24, 500), (1400, 200, 32, 1000)]


@pytest.mark.parametrize("T,R,S,W", LANES)
@pytest.mark.parametrize("kind", ["ms", "long", "huge"])
def test_step_lanes(sf, T, R, S, W, kind):
    d_np = durations(T, R, S, "long" if kind == "long" else "ms", T + R)
    if kind == "huge":
        d_np = np.minimum(d_np * (1 << 17), (1 << 46) // S)
    rng = np.random.default_rng(T)
    wall = d_np.sum(axis=2) + rng.integers(-100000, 100000, size=(T, R))
    check_evidence(sf, d_np, W, [(None, -1), (wall, -1), (wall, S - 1), (None, S // 2)])
    check_passes(sf, d_np, W)


# medians that are only 8-byte aligned: steps of many and of few ranks, few steps and many
@pytest.mark.parametrize("T,R,S,W", [(5000, 31, 7, 500), (5000, 130, 4, 500), (300, 40, 6, 50), (12, 1500, 10, 4)])
@pytest.mark.parametrize("kind", ["ms", "long"])
def test_unaligned_medians(sf, T, R, S, W, kind):
    def place(m_np):
        buf = torch.empty(m_np.size + 1, dtype=torch.int64, device="cuda")
        buf[1:] = torch.from_numpy(m_np).cuda().view(-1)
        m = buf[1:].view(m_np.shape)
        assert m.data_ptr() % 16 == 8
        return m
    d_np = durations(T, R, S, kind, T + R)
    check_evidence(sf, d_np, W, [(None, -1), (d_np.sum(axis=2) + 1000, 0)], place)


# durations and totals out of range are flagged by every form: lanes, warps, tiles and CTAs
@pytest.mark.parametrize("T,R,S", [(6000, 7, 6), (700, 9, 32), (2000, 60, 16), (40, 16, 8), (30, 100, 8), (30, 100, 9),
                                   (9, 300, 5), (4, 3000, 4), (3, 8192, 8), (2, 5000, 13), (100, 128, 8), (300, 200, 3),
                                   (10001, 9, 2)])
def test_status_bits_of_every_form(sf, T, R, S):
    group = dev(np.zeros(R, np.int32))
    calls = dict(frontier=lambda d, st: sf.sf_frontier(d, status=st),
                 ties=lambda d, st: sf.sf_frontier_ties(d, a=torch.zeros((T, S), dtype=torch.int64, device="cuda"), status=st),
                 windows=lambda d, st: sf.sf_window_aggregate(d, 50, status=st),
                 baselines=lambda d, st: sf.sf_window_baselines(d, 50, status=st),
                 gain=lambda d, st: sf.sf_direct_gain(d, 50, torch.ones((-(-T // 50), R, S), dtype=torch.int64, device="cuda"), status=st),
                 lag=lambda d, st: sf.sf_rank_lag(d, status=st), spread=lambda d, st: sf.sf_raw_spread(d, 50, status=st),
                 groups=lambda d, st: sf.sf_group_aggregate(d, group, 1, 50, status=st))
    at = (T * 2 // 3, R * 3 // 4, S // 2)
    for values, bit in (({at: -5}, sf.SF_ST_NEGATIVE), ({at: 1 << 47}, sf.SF_ST_RANGE),
                        ({at[:2] + (0,): 1 << 46, at[:2] + (S - 1,): 1 << 46}, sf.SF_ST_RANGE),
                        ({at: (1 << 47) - 1 - S}, 0)):
        d_np = np.ones((T, R, S), np.int64)
        for i, v in values.items():
            d_np[i] = v
        d = dev(d_np)
        for name, call in calls.items():
            if name == "spread" and len(values) == 2:
                continue  # durations only
            st = sf.new_status("cuda")
            call(d, st)
            assert int(st.item()) & 3 & (bit or 3) == bit, (name, values)
    wall = np.ones((T, R), np.int64)
    m = torch.ones((-(-T // 50), R, S), dtype=torch.int64, device="cuda")
    for v, bit in ((-1, sf.SF_ST_NEGATIVE), (1 << 47, sf.SF_ST_RANGE)):
        wall[at[:2]] = v
        st = sf.new_status("cuda")
        sf.sf_direct_gain(dev(np.ones((T, R, S), np.int64)), 50, m, wall=dev(wall), status=st)
        assert int(st.item()) & bit
