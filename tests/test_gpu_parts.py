"""The peel by parts (coarse ranges of bitruss numbers, then each range by a block
or a cluster of its own) at the sizes where it can go wrong: against the CPU
oracle on small graphs, against closed forms on bicliques, and against the
grid-wide peel (kept in use by a limit that addresses it) on larger ones.
Supports, bitruss numbers and the peel's statistics are whole numbers and have
to be equal."""
import numpy as np
import pytest

import oracle
from paper_2001_06111_gb300 import bitruss as bt
from paper_2001_06111_gb300 import build, synth
from tests import pins

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def h():
    build.build()
    handle = bt.bt_create(0)
    yield handle
    handle.close()


def grid_peel(h, *args, **kw):
    bt.bt_set_limits(h, join_cap=1 << 30)  # far above any cap: the grid-wide kernel, its defaults
    try:
        return bt.bt_decompose(h, *args, **kw)
    finally:
        bt.bt_set_limits(h)


# one part up to 1,024 edges, ranges above
@pytest.mark.parametrize("m", [1, 2, 33, 1023, 1024, 1025, 3001])
def test_small_graphs_against_the_oracle(h, m):
    nU, nL = max(2, m // 8), max(2, m // 12)
    g = synth.random_tiny(m, nU, nL, m) if m < 100 else synth.chunglu(nU, nL, m, 2.3, 2.4, seed=m)
    s0, p0 = oracle.bitruss(g.edges, g.nU, g.nL)
    sup, phi, _ = bt.bt_decompose(h, g.edges, g.nU, g.nL)
    np.testing.assert_array_equal(sup, s0)
    np.testing.assert_array_equal(phi.astype(np.uint64), p0)


# every edge of K_{a,b} has support and bitruss number (a-1)(b-1).  All edges leave
# in one batch: batches above the 512 kept in shared memory and the 1,024 threads,
# more touched blooms than a block lists (C(a,2) of them), parts around the
# 43,008 edges whose supports fit a block (above: a cluster)
@pytest.mark.parametrize("a,b", [(16, 32), (16, 33), (31, 33), (32, 33), (91, 92), (128, 336), (128, 337), (211, 210)])
def test_bicliques(h, a, b):
    e = pins.biclique(a, b)
    sup, phi, st = bt.bt_decompose(h, e, a, b)
    want = (a - 1) * (b - 1)
    assert (sup == want).all() and (phi == want).all()
    assert (st["rounds"], st["levels"], st["phi_max"]) == (1, 1, want)


# dense planted blocks: parts heavy enough for clusters, blooms of many pairs,
# groups of one, two and more pairs in a bloom
@pytest.mark.parametrize("m,nplant,lo,hi,flags", [(20001, 6, 10, 40, 0), (150001, 3, 100, 200, 0),
                                                  (150001, 3, 100, 200, bt.BT_TIE_LOWER_FIRST),
                                                  (300007, 2, 250, 300, 0), (400003, 0, 0, 0, 0)])
def test_same_as_the_grid_peel(h, m, nplant, lo, hi, flags):
    g = synth.chunglu(m // 12, m // 30, m, 2.1, 2.4, seed=m, nplant=nplant, plant_lo=lo, plant_hi=hi, plant_p=0.9)
    ref = grid_peel(h, g.edges, g.nU, g.nL, flags=flags)
    for _ in range(2):
        out = bt.bt_decompose(h, g.edges, g.nU, g.nL, flags=flags)
        np.testing.assert_array_equal(out[0], ref[0])
        np.testing.assert_array_equal(out[1], ref[1])
        assert out[2] == ref[2]


def union(*gs):
    """Graphs side by side, edges in one shuffled list: (edges, nU, nL)."""
    oU = oL = 0
    es = []
    for e, a, b in gs:
        es.append(np.asarray(e, np.int64) + [oU, oL])
        oU, oL = oU + a, oL + b
    e = np.concatenate(es)
    return np.random.default_rng(len(e)).permutation(e).astype(np.int32), oU, oL


def uniform(nU, nL, m):
    k = np.random.default_rng(m).choice(nU * nL, m, replace=False)
    return np.stack([k // nL, k % nL], 1), nU, nL


def blocks(c, a, b):
    return union(*[(pins.biclique(a, b), a, b)] * c)


def skewed(m):
    g = synth.chunglu(m // 8, m // 12, m, 2.2, 2.4, seed=m)
    return g.edges, g.nU, g.nL


# which way a graph is peeled: by the grid where nearly all links are on edges within a
# factor of 8 in support, or where one range would take longer than that; edges in
# no butterfly beside the ranges; a cluster for a part of few with many links
ROUTES = {
    "narrow-block": lambda: (pins.biclique(70, 70)[:-50], 70, 70),
    "narrow-random": lambda: uniform(300, 400, 9000),
    "narrow-low": lambda: uniform(900, 900, 12000),
    "low-supports": lambda: union(uniform(3000, 3000, 60000), blocks(1, 12, 12)),
    "low-supports-and-more": lambda: union(uniform(3000, 3000, 60000), blocks(12, 40, 40)),
    "factor-8": lambda: union(blocks(3, 21, 21), blocks(1, 57, 57)),
    "factor-8-and-more": lambda: union(blocks(3, 21, 21), blocks(1, 60, 60)),
    "one-range": lambda: union(blocks(1, 200, 200), blocks(5, 100, 100)),
    "few-parts": lambda: union(blocks(1, 200, 200), blocks(20, 60, 60), blocks(1000, 20, 20)),
    "no-butterflies": lambda: (np.stack([np.arange(5000)] * 2, 1).astype(np.int32), 5000, 5000),
    "almost-none": lambda: union((np.stack([np.arange(5000)] * 2, 1), 5000, 5000), blocks(1, 2, 2)),
    "zeros-and-narrow": lambda: union(uniform(60000, 60000, 60000), blocks(4, 30, 30)),
    "zeros-and-skewed": lambda: union(uniform(60000, 60000, 60000), skewed(20000)),
    "skewed": lambda: skewed(20000),
    "skewed-and-block": lambda: union(skewed(60000), blocks(1, 100, 120)),
    "skewed-and-narrow": lambda: union(skewed(3000), blocks(1, 100, 120)),
}


@pytest.mark.parametrize("name", sorted(ROUTES))
def test_routes_same_as_the_grid_peel(h, name):
    e, nU, nL = ROUTES[name]()
    ref = grid_peel(h, e, nU, nL)
    out = bt.bt_decompose(h, e, nU, nL)
    np.testing.assert_array_equal(out[0], ref[0])
    np.testing.assert_array_equal(out[1], ref[1])
    assert out[2] == ref[2]


# a graph not for parts is given up after the coarse peel's first look (its two kernels of
# preparation and itself), not after a split; one without butterflies needs nothing more
@pytest.mark.parametrize("name,more", [("narrow-block", 3), ("narrow-random", 3), ("narrow-low", 3), ("factor-8", 3), ("low-supports", 3),
                                       ("zeros-and-narrow", 3), ("almost-none", 3), ("no-butterflies", 0)])
def test_given_up_early(h, name, more):
    e, nU, nL = ROUTES[name]()
    grid_peel(h, e, nU, nL)
    launches = bt.bt_profile_read(h)["launches"]
    bt.bt_decompose(h, e, nU, nL)
    assert bt.bt_profile_read(h)["launches"] == launches + more


@pytest.mark.parametrize("flags", [0, bt.BT_PC_RECOUNT])
@pytest.mark.parametrize("name", ["narrow-random", "one-range", "few-parts", "zeros-and-narrow", "zeros-and-skewed"])
def test_routes_of_progressive_passes(h, name, flags):
    e, nU, nL = ROUTES[name]()
    bt.bt_set_limits(h, join_cap=1 << 30)
    ref = bt.bt_decompose_progressive(h, e, nU, nL, tau=0.3, flags=flags)
    bt.bt_set_limits(h)
    out = bt.bt_decompose_progressive(h, e, nU, nL, tau=0.3, flags=flags)
    np.testing.assert_array_equal(out[0], ref[0])
    np.testing.assert_array_equal(out[1], ref[1])
    assert out[2] == ref[2]


@pytest.mark.parametrize("n,hi", [(3, 300), (5, 600), (40, 20000)])
def test_batches_same_as_the_grid_peel(h, n, hi):
    gs = [synth.batch_graph(900 + i, hi=hi) for i in range(n)]
    gs = [(g.edges, g.nU, g.nL) for g in gs] + [(np.empty((0, 2), np.int32), 3, 2), (pins.biclique(40, 50), 40, 50)]
    bt.bt_set_limits(h, join_cap=1 << 30)
    ref, st0 = bt.bt_decompose_batch(h, gs, count_threads=512, peel_item=32)
    bt.bt_set_limits(h)
    out, st1 = bt.bt_decompose_batch(h, gs, count_threads=512, peel_item=32)
    assert st0 == st1
    for (s0, p0), (s1, p1) in zip(ref, out):
        np.testing.assert_array_equal(s0, s1)
        np.testing.assert_array_equal(p0, p1)


# K_{n,n} without one edge: the 2n - 2 edges at its ends leave first, then the rest
# at the same level, so all pairs are groups of more than two in one part; 1,640
# a side make 2.2e9 pairs, more than 2^31 of them in such groups
@pytest.mark.parametrize("n", [61, 300, 1640])
def test_pair_places_of_all_32_bits(n):
    e = pins.biclique(n, n)
    e = e[(e[:, 0] > 0) | (e[:, 1] > 0)]
    with bt.bt_create(0) as own:  # (its memory goes back with it: 150 GB for 1,640)
        sup, phi, st = bt.bt_decompose(own, e, n, n)
    at_end = (e[:, 0] == 0) | (e[:, 1] == 0)
    assert (sup == np.where(at_end, (n - 1) * (n - 2), n * (n - 2))).all()
    assert (phi == (n - 1) * (n - 2)).all()
    assert (st["rounds"], st["levels"], st["phi_max"]) == (2, 1, (n - 1) * (n - 2))


# every item size a batch may ask for, on blocks of many links an edge and one level:
# all edges leave in one jump, so one round queues every link (K_{60,60} is the
# smallest of these whose 32-entry items number more than its 64-entry items
# leave room for)
@pytest.mark.parametrize("item", [32, 64, 128])
@pytest.mark.parametrize("sides", [[(60, 60)], [(100, 100)], [(128, 336)], [(200, 200)],
                                   [(60, 60), (33, 40), (128, 200), (200, 200)]])
def test_bicliques_by_item_size(h, sides, item):
    out, st = bt.bt_decompose_batch(h, [(pins.biclique(a, b), a, b) for a, b in sides], count_threads=512,
                                    peel_item=item)
    assert (st["rounds"], st["levels"]) == (len({(a - 1) * (b - 1) for a, b in sides}),) * 2
    for (a, b), (sup, phi) in zip(sides, out):
        assert (sup == (a - 1) * (b - 1)).all() and (phi == (a - 1) * (b - 1)).all()


# passes of the progressive compression: assigned edges among the pairs, a first part
# below the recorded levels (the default reading) or none (Alg. 7's)
@pytest.mark.parametrize("flags", [0, bt.BT_PC_RECOUNT])
@pytest.mark.parametrize("m,tau,nplant", [(1500, 0.5, 0), (12000, 0.1, 0), (40001, 0.3, 4), (90001, 1.0, 3)])
def test_progressive_same_as_the_grid_peel(h, m, tau, nplant, flags):
    g = synth.chunglu(m // 8, m // 14, m, 2.1, 2.4, seed=m, nplant=nplant, plant_lo=20, plant_hi=60, plant_p=0.9)
    bt.bt_set_limits(h, join_cap=1 << 30)
    ref = bt.bt_decompose_progressive(h, g.edges, g.nU, g.nL, tau=tau, flags=flags)
    bt.bt_set_limits(h)
    out = bt.bt_decompose_progressive(h, g.edges, g.nU, g.nL, tau=tau, flags=flags)
    np.testing.assert_array_equal(out[0], ref[0])
    np.testing.assert_array_equal(out[1], ref[1])
    assert out[2] == ref[2]
