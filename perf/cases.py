"""What a user of the bitruss library has it do, as timed cases.

Every case is one call sequence through the public binding
(`paper_2001_06111_gb300.bitruss`; its C entry points where a program keeps
its results for many graphs in buffers of its own) on a seeded synthetic bipartite graph of
the repository's own kinds: skewed Chung-Lu graphs, the same with planted
dense bicliques, and the mixed-size graphs of the batch and serving
workloads.  Sizes are those of the repository's workloads and tests, a little
off round numbers so that remainders occur.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2001_06111_gb300 import bitruss as bt

DEV = "cuda"


# ----------------------------------------------------------------- the cases
def listed():
    return [
        # one small graph from host memory, the low end of the batch and
        # serving distributions: latency and launches are everything
        dict(name="decompose-1k", kind="decompose", m=1003, nU=126, nL=84, gU=2.3, gL=2.4, cap=0, plant=0,
             device=False, lower_first=False),
        # the repository's 20,000-edge workload through host buffers
        dict(name="decompose-20k", kind="decompose", m=20000, nU=2000, nL=1500, gU=2.2, gL=2.5, cap=0, plant=0,
             device=False, lower_first=False),
        # the top end of the batch distribution as a single device-resident
        # graph, with the other reading of the id convention
        dict(name="decompose-200k", kind="decompose", m=199999, nU=25000, nL=16667, gU=2.1, gL=2.5, cap=0, plant=0,
             device=True, lower_first=True),
        # the 2M-edge skewed workload (degree cap 20,000), device-resident
        dict(name="decompose-2M", kind="decompose", m=2000000, nU=200000, nL=80000, gU=2.1, gL=2.4, cap=20000,
             plant=0, device=True, lower_first=False),
        # dense planted bicliques in a skewed graph (fraud-ring shape): high
        # supports, deep levels, large blooms; the largest single-graph peel
        dict(name="decompose-planted", kind="decompose", m=2400001, nU=160000, nL=40000, gU=2.0, gL=2.3, cap=0,
             plant=14, device=True, lower_first=False),
        # many uneven graphs in one call, host buffers in and out
        dict(name="batch-384", kind="batch", graphs=384, lo=100, hi=200000),
        # a burst of requests against the request server, all awaited
        dict(name="serve-48", kind="serve", graphs=48, lo=100, hi=200000),
        # butterfly counting alone, inside a caller that owns all device memory
        dict(name="count-static-60k", kind="static", m=60013, nU=7000, nL=5000, gU=2.2, gL=2.4, cap=0, plant=0),
        # butterfly counting alone on the 30M-edge workload's shape
        dict(name="count-30M", kind="count", m=30000000, nU=2000000, nL=500000, gU=2.0, gL=2.3, cap=0, plant=200),
        # the BE-Index alone, kept on the device
        dict(name="index-2M", kind="index", m=1999993, nU=200000, nL=80000, gU=2.1, gL=2.4, cap=20000, plant=0),
        # progressive compression (BiT-PC) with its default step of 0.1
        dict(name="progressive-100k", kind="progressive", m=100003, nU=12500, nL=8334, gU=2.2, gL=2.4, cap=0,
             plant=0, tau=0.1, recount=False),
        # the k-bitruss hierarchy of 30M edges and one H_k of it
        dict(name="hierarchy-30M", kind="hierarchy", m=30000000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sides(rng, m):
    """Layer sizes of a graph of m edges: the batch's m/8 by m/12, or sparser."""
    r = rng.uniform(1.0, 1.6) if m > 1000 else 1.0
    return max(12, int(m / 8 * r) + rng.randrange(3)), max(9, int(m / 12 * r) + rng.randrange(3))


def draw(rng):
    kind = rng.choice(["decompose", "decompose", "decompose", "planted", "batch", "serve", "static", "count",
                       "index", "progressive", "hierarchy"])
    if kind in ("batch", "serve"):
        return dict(kind=kind, graphs=_log(rng, 8, 384 if kind == "batch" else 48), lo=100,
                    hi=_log(rng, 2000, 200000))
    if kind == "hierarchy":
        return dict(kind=kind, m=_log(rng, 1000, 30000000))
    if kind == "planted":
        m = _log(rng, 200000, 2400001)
        return dict(kind="decompose", m=m, nU=m // 15, nL=m // 60, gU=rng.uniform(2.0, 2.2),
                    gL=rng.uniform(2.3, 2.5), cap=0, plant=max(1, m // 172000), device=True,
                    lower_first=rng.random() < 0.3)
    top = {"decompose": 2000000, "static": 260000, "count": 30000000, "index": 2000000, "progressive": 200000}[kind]
    m = _log(rng, 1000, top)
    nU, nL = _sides(rng, m)
    c = dict(kind=kind, m=m, nU=nU, nL=nL, gU=rng.uniform(2.1, 2.6), gL=rng.uniform(2.3, 2.6),
             cap=20000 if m > 300000 else 0, plant=0)
    if kind == "decompose":
        c.update(device=rng.random() < 0.5, lower_first=rng.random() < 0.3)
    if kind == "progressive":
        c.update(tau=rng.choice([0.05, 0.1, 0.2, 0.5]), recount=rng.random() < 0.4)
    return c


# ---------------------------------------------------------------- the inputs
def _weights(n, gamma, m, cap):
    w = (np.arange(n, dtype=np.float64) + 1.0) ** (-1.0 / (gamma - 1.0))
    w *= m / w.sum()
    return np.minimum(w, cap) if cap else w


def _chunglu(nU, nL, m, gU, gL, cap, plant, seed):
    """Chung-Lu bipartite graph with power-law expected degrees, `plant`
    bicliques (sides uniform in [50, 300], density 0.9) placed first, vertex
    ids and edge order shuffled: int32 (m, 2) on the GPU."""
    m = min(m, int(0.9 * nU * nL))
    rng = np.random.default_rng(seed)
    g = torch.Generator(device=DEV)
    g.manual_seed(int(rng.integers(1 << 62)))
    cums = []
    for n, gamma in ((nU, gU), (nL, gL)):
        c = np.cumsum(_weights(n, gamma, m, cap))
        cums.append(torch.from_numpy(c / c[-1]).to(DEV))
    keys = torch.empty(0, dtype=torch.int64, device=DEV)
    for _ in range(plant):
        a, b = int(rng.integers(50, 301)), int(rng.integers(50, 301))
        u = torch.from_numpy(rng.choice(nU, a, replace=False)).to(DEV)
        v = torch.from_numpy(rng.choice(nL, b, replace=False)).to(DEV)
        k = (u[:, None] * nL + v[None, :]).reshape(-1)
        keys = torch.cat([keys, k[torch.rand(k.numel(), generator=g, device=DEV) < 0.9]])
    keys = torch.unique(keys)
    planted = keys
    want = m - int(planted.numel())
    rest = torch.empty(0, dtype=torch.int64, device=DEV)
    n = int(want * 1.3) + 64
    while rest.numel() < want:
        r = torch.rand(2, n, generator=g, device=DEV, dtype=torch.float64)
        u = torch.searchsorted(cums[0], r[0]).clamp_(max=nU - 1)
        v = torch.searchsorted(cums[1], r[1]).clamp_(max=nL - 1)
        k = torch.unique(torch.cat([rest, u * nL + v]))
        if planted.numel():
            at = torch.searchsorted(planted, k).clamp_(max=planted.numel() - 1)
            k = k[planted[at] != k]
        rest = k
        n = min(2 * n, 1 << 26)
    rest = rest[torch.randperm(rest.numel(), generator=g, device=DEV)[:want]]
    keys = torch.cat([planted, rest])
    keys = keys[torch.randperm(keys.numel(), generator=g, device=DEV)]
    pu = torch.randperm(nU, generator=g, device=DEV)
    pl = torch.randperm(nL, generator=g, device=DEV)
    return torch.stack([pu[keys // nL], pl[keys % nL]], dim=1).to(torch.int32).contiguous()


def _graph(case, seed):
    return _chunglu(case["nU"], case["nL"], case["m"], case["gU"], case["gL"], case["cap"], case["plant"], seed)


def _mixed(case, seed):
    """Graphs of the batch and serving workloads on the host: sizes log-uniform,
    exponents uniform in [2.0, 2.6].  The sizes belong to the case, the graphs
    to the seed.  Edge lists and results lie in one host buffer each, as a
    program with many graphs keeps them: (bt_graph array, supports, bitruss
    numbers, what must stay alive)."""
    sizes = np.random.default_rng([case["graphs"], case["hi"]])
    m = np.exp(sizes.uniform(math.log(case["lo"]), math.log(case["hi"]), case["graphs"])).round().astype(np.int64)
    gamma = sizes.uniform(2.0, 2.6, (case["graphs"], 2))
    off = np.concatenate([[0], np.cumsum(m)])
    edges = np.empty((off[-1], 2), dtype=np.int32)
    sup = np.empty(off[-1], dtype=np.int64)
    phi = np.empty(off[-1], dtype=np.int32)
    arr = (bt.Graph * case["graphs"])()
    rng = np.random.default_rng(seed)
    for i in range(case["graphs"]):
        n, o = int(m[i]), int(off[i])
        nU, nL = (n + 7) // 8, (n + 11) // 12
        e = _chunglu(nU, nL, n, gamma[i, 0], gamma[i, 1], 0, 0, int(rng.integers(1 << 62)))
        edges[o:o + n] = e.cpu().numpy()
        arr[i] = bt.Graph(edges.ctypes.data + 8 * o, n, nU, nL, sup.ctypes.data + 8 * o, phi.ctypes.data + 4 * o)
    return arr, sup, phi, edges


def _phi(case, seed):
    """Bitruss numbers as skewed graphs have them (many zeros, a heavy tail), in
    an order that belongs to the seed."""
    m = case["m"]
    x = (torch.arange(m, device=DEV, dtype=torch.float64) + 0.5) / m
    x = ((x.pow_(-0.7) - 1.0) * 4.0).to(torch.int64).to(torch.int32)
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return x[torch.randperm(m, generator=g, device=DEV)].view(torch.uint32)


class _Server(bt.Server):
    """A request server that ends with the state that holds it."""

    def __del__(self):
        self.close()


def prepare(case, seed):
    k = case["kind"]
    st = dict(case=case)
    if k == "hierarchy":
        st["phi"] = _phi(case, seed)
    elif k in ("batch", "serve"):
        st["graphs"] = _mixed(case, seed)
    else:
        e = _graph(case, seed)
        host = k == "progressive" or (k == "decompose" and not case["device"])
        st["edges"] = e.cpu().numpy() if host else e
        if k == "static":
            st["out"] = torch.empty(e.shape[0], dtype=torch.int64, device=DEV)
    torch.cuda.synchronize()
    if k == "serve":
        st["server"] = _Server(0)
    elif k != "static":
        st["h"] = bt.bt_create(0, torch.cuda.current_stream())
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    c = st["case"]
    k = c["kind"]
    if k == "decompose":
        flags = bt.BT_TIE_LOWER_FIRST if c["lower_first"] else 0
        sup, phi, stats = bt.bt_decompose(st["h"], st["edges"], c["nU"], c["nL"], flags=flags)
        return [_ints(sup), _ints(phi), stats]
    if k == "batch":
        arr, sup, phi, _ = st["graphs"]
        stats = bt.BatchStats()
        _ok(bt.load().bt_decompose_batch(st["h"].ptr, arr, len(arr), None, ctypes.byref(stats), 0))
        # the schedule fields say what the autotuner timed best, not a result
        keep = ("graphs", "launches", "edges", "wedges", "rounds", "levels", "support_updates")
        return [sup, phi, {f: int(getattr(stats, f)) for f in keep}]
    if k == "serve":
        lib, ptr = bt.load(), st["server"].ptr
        arr, sup, phi, _ = st["graphs"]
        ids = [ctypes.c_uint64() for _ in arr]
        for g, i in zip(arr, ids):
            _ok(lib.bt_server_submit(ptr, ctypes.byref(g), ctypes.byref(i)))
        info = bt.RequestInfo()
        for i in ids:
            _ok(lib.bt_server_poll(ptr, i.value, 1, ctypes.byref(info)))
            _ok(info.status)
        return [sup, phi]
    if k == "static":
        bt.bt_count_support_static(st["edges"], c["nU"], c["nL"], st["out"])
        return st["out"]
    if k == "count":
        return _ints(bt.bt_count_support(st["h"], st["edges"], c["nU"], c["nL"]))
    if k == "index":
        return bt.bt_build_index(st["h"], st["edges"], c["nU"], c["nL"])
    if k == "progressive":
        sup, phi, stats = bt.bt_decompose_progressive(st["h"], st["edges"], c["nU"], c["nL"], tau=c["tau"],
                                                      flags=bt.BT_PC_RECOUNT if c["recount"] else 0)
        # support_updates counts this library's own work, the rest the method's
        return [_ints(sup), _ints(phi), {f: v for f, v in stats.items() if f != "support_updates"}]
    order, ps = bt.bt_hierarchy(st["h"], st["phi"])
    hk = bt.bt_k_bitruss(st["h"], st["phi"], 5)
    return [_ints(order), _ints(ps), _ints(hk)]


def _ok(status):
    if status != bt.BT_OK:
        raise RuntimeError("bitruss status %d" % status)


def _ints(x):
    """Unsigned results under the signed type of their width (same bits)."""
    if isinstance(x, torch.Tensor):
        return x.view({4: torch.int32, 8: torch.int64}[x.element_size()])
    return x.view({4: np.int32, 8: np.int64}[x.itemsize])


# ---------------------------------------------------- what a pass cannot omit
def work(case):
    """Edge list in, results out; the arithmetic is whole numbers on graphs, so
    no floating-point operations are counted.  The wedges and the index that
    lie between depend on the drawn graph and are left out."""
    k = case["kind"]
    if k == "hierarchy":
        return dict(bytes=case["m"] * (4 + 8 + 4 + 2), flops=0)
    if k in ("batch", "serve"):
        mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        return dict(bytes=int(case["graphs"] * mean) * (8 + 8 + 4), flops=0)
    per = {"decompose": 20, "progressive": 20, "static": 16, "count": 16, "index": 8}[k]
    return dict(bytes=case["m"] * per, flops=0)


# ------------------------------------------------------------ exact answers
def _support(adj, e):
    """Butterflies through each edge: paths of three edges from u to v less
    those that go back over (u, v), in doubles (whole numbers below 2^53)."""
    p = adj @ (adj.T @ adj)
    du, dl = adj.sum(1), adj.sum(0)
    u, v = e[:, 0].long(), e[:, 1].long()
    return (p[u, v] - du[u] - dl[v] + 1).round().long()


def _phi_exact(nU, nL, e):
    """Bitruss numbers by deletion: at each k remove every edge with fewer than
    k + 1 butterflies until none is left below."""
    phi = torch.zeros(e.shape[0], dtype=torch.int64, device=e.device)
    alive = torch.ones(e.shape[0], dtype=torch.bool, device=e.device)
    adj = torch.zeros(nU, nL, dtype=torch.float64, device=e.device)
    adj[e[:, 0].long(), e[:, 1].long()] = 1.0
    k = 0
    while bool(alive.any()):
        sup = _support(adj, e)
        k = max(k, int(sup[alive].min()))
        gone = alive & (sup <= k)
        phi[gone] = k
        alive &= ~gone
        adj[e[gone, 0].long(), e[gone, 1].long()] = 0.0
    return phi.to(torch.int32)


def exact(case, seed):
    k = case["kind"]
    if k == "hierarchy":
        phi = _phi(case, seed).view(torch.int32)  # all below 2^31
        ps, order = torch.sort(phi, descending=True, stable=True)
        return [order.to(torch.int32), ps, torch.nonzero(phi >= 5).reshape(-1).to(torch.int32)]
    if k in ("batch", "serve", "index") or case["nU"] * case["nL"] > 40_000_000:
        return None
    e = _graph(case, seed)
    adj = torch.zeros(case["nU"], case["nL"], dtype=torch.float64, device=DEV)
    adj[e[:, 0].long(), e[:, 1].long()] = 1.0
    sup = _support(adj, e)
    if k in ("static", "count"):
        return sup
    phi = _phi_exact(case["nU"], case["nL"], e) if case["m"] <= 3000 else None
    return [sup, phi, None]
