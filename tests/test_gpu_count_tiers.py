"""The counting kernels at the edges of their tiers: start vertices counted by a
warp (up to 256 wedges over up to 32 middle vertices) and by a block, chunks of
1,024 middle vertices, and counters inside and below the 90,112 ranks (16 bits)
or 45,056 (32 bits) kept in shared memory."""
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


def check(h, e, nU, nL):
    np.testing.assert_array_equal(bt.bt_count_support(h, e, nU, nL), oracle.support(e, nU, nL))
    st = bt.bt_build_index(h, e, nU, nL)
    assert 4 * st["n_butterflies"] == int(oracle.support(e, nU, nL).sum())


# K_{a,b}: support (a-1)(b-1); wedges and middle vertices around 256 and 32 and around 1,024
@pytest.mark.parametrize("a,b", [(2, 2), (8, 32), (8, 33), (9, 31), (16, 16), (17, 16), (32, 32), (33, 32), (2, 1023),
                                 (2, 1024), (2, 1025), (3, 2049)])
def test_bicliques(h, a, b):
    sup = bt.bt_count_support(h, pins.biclique(a, b), a, b)
    assert (sup == (a - 1) * (b - 1)).all()
    st = bt.bt_build_index(h, pins.biclique(a, b), a, b)
    assert st["n_butterflies"] == a * (a - 1) * b * (b - 1) // 4


# tiles of exactly 1,024 middle vertices, whose last windows of wedges are not full,
# with assigned edges among them (a pass of the progressive compression at every
# level): all edges of K_{a,b} and b more upper vertices of one edge each
@pytest.mark.parametrize("a,b", [(2, 1024), (3, 1024), (2, 2047), (3, 2048)])
def test_full_tiles_with_assigned_edges(h, a, b):
    e = np.concatenate([pins.biclique(a, b), np.stack([a + np.arange(b), np.arange(b)], 1)]).astype(np.int32)
    want = np.where(e[:, 0] < a, (a - 1) * (b - 1), 0)
    for tau in (0.5, 1.0):
        sup, phi, _ = bt.bt_decompose_progressive(h, e, a + b, b, tau=tau)
        np.testing.assert_array_equal(sup.astype(np.int64), want)
        np.testing.assert_array_equal(phi.astype(np.int64), want)


# a hub pair over all lower vertices beside many vertices of low degree: end vertices
# far below the hub, in and out of the counters in shared memory
@pytest.mark.parametrize("nU,nL", [(90110, 700), (90112, 700), (140000, 3000)])
def test_counters_below_the_window(h, nU, nL):
    rng = np.random.default_rng(nU)
    hubs = np.stack(np.meshgrid([0, 1], np.arange(nL), indexing="ij"), -1).reshape(-1, 2)
    u = np.repeat(np.arange(2, nU), 2)
    v = rng.integers(0, nL // 2, u.size // 2)
    rest = np.stack([u, np.stack([v, v + 1 + rng.integers(0, nL // 2 - 1, v.size)], 1).reshape(-1)], 1)
    e = np.concatenate([hubs, rest]).astype(np.int32)
    check(h, e, nU, nL)


# 2^16 and more middle vertices: 32-bit counters.  Four upper vertices have edges,
# so the supports follow from their common neighbours (paths of three edges from u
# to v, less those over (u, v)).
@pytest.mark.parametrize("nL", [65535, 65536, 70001])
def test_start_vertex_of_many_middles(h, nL):
    lower = np.arange(nL)
    e = np.concatenate([np.stack([np.full(nL, i), lower], 1) for i in range(3)]
                       + [np.stack([np.full(50, 3), lower[:50]], 1)]).astype(np.int32)
    adj = np.zeros((4, nL), dtype=np.int64)
    adj[e[:, 0], e[:, 1]] = 1
    paths = (adj @ adj.T) @ adj
    want = paths[e[:, 0], e[:, 1]] - adj.sum(1)[e[:, 0]] - adj.sum(0)[e[:, 1]] + 1
    np.testing.assert_array_equal(bt.bt_count_support(h, e, 60000, nL).astype(np.int64), want)
    assert 4 * bt.bt_build_index(h, e, 60000, nL)["n_butterflies"] == int(want.sum())


def test_skewed_graph(h):
    g = synth.chunglu(9000, 4000, 60000, 2.0, 2.2, seed=5)
    check(h, g.edges, g.nU, g.nL)


# around 81,920 vertices, above which counters go by places in a layer instead of
# ranks; either layer larger, either convention of ids
@pytest.mark.parametrize("flags", [0, bt.BT_TIE_LOWER_FIRST])
@pytest.mark.parametrize("nU,nL", [(61920, 20000), (61921, 20000), (20000, 61921), (3000, 120000), (180000, 3000)])
def test_places_in_a_layer(h, nU, nL, flags):
    g = synth.chunglu(nU, nL, 50000, 2.0, 2.2, seed=nU)
    sup = oracle.support(g.edges, nU, nL)
    np.testing.assert_array_equal(bt.bt_count_support(h, g.edges, nU, nL, flags=flags), sup)
    st = bt.bt_build_index(h, g.edges, nU, nL, flags=flags)
    assert 4 * st["n_butterflies"] == int(sup.sum())


# the pairs of a bloom of many lie about in the order of their middle vertices (the peel
# of dense blooms walks along their edges): a block places 4,096 neighbouring wedges
# at a time, some 30 middle vertices here, where 32 shares of the wedges would
# spread any 32 neighbouring pairs over nearly all 1,000
def test_pairs_of_dense_blooms_in_order(h):
    a, b = 150, 1000
    st = bt.bt_build_index(h, pins.biclique(a, b), a, b)
    k, first, pairs, _ = bt.bt_index_export(h, st, a * b)
    for i in range(len(k) - 100, len(k)):
        mid = pairs[first[i]:first[i] + k[i], 0].astype(np.int64) % b
        assert k[i] == b and len(np.unique(mid)) == b
        assert np.median([np.ptp(mid[j:j + 32]) for j in range(0, b - 32, 32)]) < b / 2
