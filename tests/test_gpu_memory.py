"""Device memory a call may hold: the estimate of bt_estimate_bytes and the server's
admission bound against what calls really take from the GPU."""
import numpy as np
import pytest

from paper_2001_06111_gb300 import bitruss as bt
from paper_2001_06111_gb300 import build, synth
from tests import pins

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def skewed(m, nplant=0):
    g = synth.chunglu(m // 12, m // 30, m, 2.1, 2.4, seed=m, nplant=nplant, plant_lo=250, plant_hi=300, plant_p=0.9)
    return g.edges, g.nU, g.nL


def uniform(nU, nL, m):
    k = np.unique(np.random.default_rng(m).integers(0, nU * nL, int(1.1 * m)))
    k = np.random.default_rng(m).permutation(k)[:m]
    return np.stack([k // nL, k % nL], 1).astype(np.int32), nU, nL


# blooms of many pairs, blooms of few (their state weighs most), skewed graphs by parts
# with and without a dense block, and graphs of many vertices and no blooms
GRAPHS = {
    "biclique": lambda: (pins.biclique(400, 400), 400, 400),
    "uniform": lambda: uniform(20000, 20000, 2000000),
    "skewed": lambda: skewed(600000),
    "planted": lambda: skewed(400000, 2),
    "sparse": lambda: uniform(400000, 100000, 300000),
}


def taken(call):
    """Bytes a call on a fresh handle took (its memory pool keeps what it took)."""
    build.build()
    with bt.bt_create(0) as warm:  # kernels are loaded once
        for small in (pins.biclique(3, 3), pins.biclique(60, 60)):
            bt.bt_decompose_batch(warm, [(small, 60, 60)])
    free = torch.cuda.mem_get_info()[0]
    with bt.bt_create(0) as h:
        call(h)
        return free - torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_estimate_is_an_upper_bound(name):
    e, nU, nL = GRAPHS[name]()
    used = taken(lambda h: bt.bt_decompose(h, e, nU, nL))
    assert used <= bt.bt_estimate_bytes(e, nU, nL)[0]


@pytest.mark.parametrize("name", ["biclique", "skewed", "planted"])
def test_admission_bound_covers_a_batch(name):
    # the counters' share of a batch's bound is charged once, so several requests of
    # one kind must be covered by the rest
    e, nU, nL = GRAPHS[name]()
    n = 4
    used = taken(lambda h: bt.bt_decompose_batch(h, [(e, nU, nL)] * n))
    with bt.Server(0) as srv:
        info, _ = srv.poll(srv.submit(e, nU, nL), wait=True)
        counters = 16 * 152 * (nU + nL)
        assert used <= n * (info["admitted_bytes"] - counters) + counters


def test_a_budget_below_the_bound_still_serves():
    # parts do not fit the budget, the grid's peel does: served as before
    e, nU, nL = pins.biclique(100, 100), 100, 100
    least = 201 * 32 + 10000 * 160 + 1000000 * 32 + (64 << 20) + 16 * 152 * 200
    with bt.Server(0, memory_budget_bytes=least) as srv:
        info, (_, phi) = srv.poll(srv.submit(e, nU, nL), wait=True)
    assert info["status"] == bt.BT_OK and (phi == 99 * 99).all() and info["admitted_bytes"] == least
    with bt.Server(0, memory_budget_bytes=least - 1) as srv:
        info, _ = srv.poll(srv.submit(e, nU, nL), wait=True)
    assert info["status"] == bt.BT_ERR_NOMEM


def test_counters_of_many_vertices_by_fewer_blocks():
    # a block an SM would take 365 GB for emit's arrays: ids spread over 150M + 10M
    # vertices, which changes no vertex's place in the priority order among those
    # with edges
    g = synth.chunglu(3000, 2000, 40000, 2.1, 2.4, seed=8)
    far = g.edges * np.array([[50000, 5000]], dtype=np.int32)
    with bt.bt_create(0) as h:
        near = bt.bt_decompose(h, g.edges, g.nU, g.nL)
        out = bt.bt_decompose(h, far, 150_000_000, 10_000_000)
        np.testing.assert_array_equal(bt.bt_count_support(h, far, 150_000_000, 10_000_000), near[0])
    np.testing.assert_array_equal(out[0], near[0])
    np.testing.assert_array_equal(out[1], near[1])
    assert out[2] == near[2]


def _decompose(h, g):
    return bt.bt_decompose(h, g.edges, g.nU, g.nL)[:2]


def _batch(h, g):
    return [x for r in bt.bt_decompose_batch(h, [(g.edges, g.nU, g.nL)] * 2)[0] for x in r]


def _progressive(h, g):
    return bt.bt_decompose_progressive(h, g.edges, g.nU, g.nL, tau=0.5)[:2]


# a GPU that is full but for a part of what a call takes when it may: the call runs out of
# memory somewhere between its first array and its last, and either says so or,
# where only the parts do not fit, peels by the grid with the same results
@pytest.mark.parametrize("call", [_decompose, _batch, _progressive])
def test_calls_on_a_full_gpu(call):
    g = synth.chunglu(50000, 20000, 600000, 2.1, 2.4, seed=3)
    want = []
    used = taken(lambda h: want.extend(call(h, g)))
    with bt.bt_create(0) as h:
        call(h, g)
        launches = bt.bt_profile_read(h)["launches"]
        bt.bt_set_limits(h, join_cap=1 << 30)
        for a, b in zip(want, call(h, g)):  # (and the grid's kernels are loaded)
            np.testing.assert_array_equal(a, b)
    refused = otherwise = 0
    for share in np.linspace(0.35, 1.1, 13):
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        full = torch.empty(free - int(share * used), dtype=torch.uint8, device="cuda")
        with bt.bt_create(0) as h:
            try:
                out = call(h, g)
            except bt.BitrussError as err:
                assert err.code == bt.BT_ERR_NOMEM
                refused += 1
                out = want
            otherwise += bt.bt_profile_read(h)["launches"] != launches
            for a, b in zip(want, out):
                np.testing.assert_array_equal(a, b)
            del full
            torch.cuda.empty_cache()
            for a, b in zip(want, call(h, g)):  # the handle is as good as before
                np.testing.assert_array_equal(a, b)
    assert 0 < refused < 13 and otherwise > refused
