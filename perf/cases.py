"""Performance cases of the partitioner: the calls a program makes, over the sizes it makes them at.

Every case names a hypergraph shape, its size, an entry point and the entry point's options.  The
shapes are those of the framework's own workloads, drawn on the GPU from the seed alone:

  uniform   N nodes, N hyperedges of 2 to 6 uniform pins, unit weights;
  netlist   N nodes of weight 1 to 4 and 1.2 N nets: 70 % two-pin, a geometric tail up to 64 pins,
            0.1 % high-fanout nets of 1,000 to 10,000 pins, pins local to a window;
  rownet    the row-net hypergraph of an N x N power-law matrix: Zipf(2.1) rows of at least 2
            entries, a fifth of the entries in 1 % hub columns, unit weights.

Entry points ("call"):

  oneshot   create + partition + close: a tool that partitions one hypergraph and exits, from host
            arrays ("source": "host") or from arrays another GPU program left on the device;
  resident  partition_device on a handle that stays: repeated partitions of one design;
  refine    refine_kept: the same hierarchy refined under another imbalance (design-space sweeps);
  batch     partition_batch: many independent hypergraphs at once;
  serve     a burst of requests to a running server, waited for;
  cut       the cut of a k-way partition, through a handle or without allocation.
"""
import math

import numpy as np
import torch

import paper_2012_13618_gb300 as bp

LEVELS = 25


def listed():
    return [
        # the smallest call: a thousand-node hypergraph partitioned once, all latency
        dict(name="oneshot_uniform_1k", call="oneshot", source="host", shape="uniform", n=1000, k=2, eps=0.1,
             policy="LDH", iters=2),
        # a small hypergraph that stays on the GPU and is partitioned again and again
        dict(name="resident_uniform_10k", call="resident", shape="uniform", n=10_000, k=2, eps=0.1, policy="LDH",
             iters=2),
        # a mid-size circuit read from files and partitioned once (copies, checks and level 0 included)
        dict(name="oneshot_netlist_150k", call="oneshot", source="host", shape="netlist", n=150_001, k=2, eps=0.05,
             policy="LDH", iters=2),
        # the headline: one bisection of the 1M-node circuit resident in HBM
        dict(name="resident_netlist_1m", call="resident", shape="netlist", n=1_000_000, k=2, eps=0.05, policy="LDH",
             iters=2),
        # the largest: a 5M x 5M sparse matrix for parallel matrix-vector products
        dict(name="resident_rownet_5m", call="resident", shape="rownet", n=5_000_000, k=2, eps=0.05, policy="LDH",
             iters=2),
        # a sparse matrix assembled on the GPU and partitioned once
        dict(name="oneshot_rownet_400k", call="oneshot", source="device", shape="rownet", n=400_003, k=2, eps=0.05,
             policy="LDH", iters=2),
        # weighted nets with the weight-based policy and parallel-net merging (timing-driven placement)
        dict(name="resident_weighted_90k", call="resident", shape="netlist", n=90_007, k=2, eps=0.05, policy="HWD",
             iters=2, hw=9, merge=True),
        # a 16-way partition by nested bisection, each bisection with its share of the imbalance
        dict(name="resident_kway16_250k", call="resident", shape="netlist", n=250_000, k=16, eps=0.05, policy="LDH",
             iters=2, adaptive=True),
        # one point of a design-space sweep on a kept hierarchy
        dict(name="refine_netlist_500k", call="refine", shape="netlist", n=499_979, k=2, eps=0.03, policy="LDH",
             iters=4),
        # many small circuits at once (k = 2, every eighth one k = 4)
        dict(name="batch_netlist_400", call="batch", shape="netlist", n=1000, n_max=40_000, count=400, k=2, eps=0.05,
             policy="LDH", iters=2),
        # a burst of mixed requests to a server (k cycles through 2, 4, 16)
        dict(name="serve_mix_12", call="serve", shape="mix", n=30_000, n_max=120_000, count=12, k=2, eps=0.05,
             policy="LDH", iters=2),
        # the cut of an 8-way partition that another program computed, arrays on the device
        dict(name="cut_netlist_1m_k8", call="cut", source="device", shape="netlist", n=1_000_000, k=8, hw=4),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    call = rng.choice(["oneshot", "oneshot", "resident", "resident", "resident", "refine", "batch", "serve", "cut"])
    if call == "batch":
        lo = size(1000, 4000)
        return dict(call=call, shape="netlist", n=lo, n_max=lo * rng.randint(2, 12), count=size(20, 400), k=2,
                    eps=rng.choice([0.03, 0.05, 0.1]), policy=rng.choice(["LDH", "HDH", "RAND"]), iters=2)
    if call == "serve":
        lo = size(30_000, 60_000)
        return dict(call=call, shape="mix", n=lo, n_max=2 * lo, count=rng.randint(4, 16), k=2, eps=0.05,
                    policy=rng.choice(["LDH", "RAND"]), iters=2)
    if call == "cut":
        return dict(call=call, source=rng.choice(["device", "handle"]), shape=rng.choice(["netlist", "rownet"]),
                    n=size(1000, 1_000_000), k=rng.randint(2, 64), hw=rng.choice([0, 4]))
    shape = rng.choice(["uniform", "netlist", "netlist", "rownet"])
    c = dict(call=call, shape=shape, n=size(1000, 1_500_000 if shape == "rownet" else 1_000_000), k=2,
             eps=rng.choice([0.03, 0.05, 0.1]), policy=rng.choice(["LDH", "LDH", "HDH", "LWD", "HWD", "RAND"]),
             iters=rng.choice([1, 2, 2, 4]))
    if call == "oneshot":
        c["source"] = rng.choice(["host", "device"])
    if call != "refine" and rng.random() < 0.25:
        c["k"] = rng.choice([3, 4, 8, 16])
        c["n"] = min(c["n"], 250_000)
        c["adaptive"] = rng.random() < 0.5
    if c["policy"] in ("LWD", "HWD"):
        c["hw"] = 9
        c["merge"] = rng.random() < 0.5
    return c


# ------------------------------------------------------------------------------- hypergraphs
def _fanout(n):
    """Range of a netlist's high-fanout nets (clipped on small circuits)."""
    return max(2, min(1000, n // 4)), max(2, min(10_000, n // 2))


def _row_cap(n):
    return max(2, min(100_000, n // 4))


def _csr(deg):
    off = torch.zeros(deg.numel() + 1, dtype=torch.int64, device=deg.device)
    torch.cumsum(deg, 0, out=off[1:])
    net = torch.repeat_interleave(torch.arange(deg.numel(), device=deg.device), deg)
    slot = torch.arange(net.numel(), device=deg.device) - off[net]
    return off, net, slot


def _uniform(n, gen):
    deg = torch.randint(2, 7, (n,), generator=gen, device="cuda")
    off, net, slot = _csr(deg)
    pins = torch.randint(0, n, (net.numel(),), generator=gen, device="cuda")
    return off, pins, None


def _netlist(n, gen):
    e = int(1.2 * n)
    lo, hi = _fanout(n)
    u = torch.rand(e, generator=gen, device="cuda")
    v = torch.rand(e, generator=gen, device="cuda", dtype=torch.float64)
    tail = 3 + torch.floor(torch.log2(1.0 / (1.0 - v).clamp_min(1e-18))).to(torch.int64)
    deg = torch.where(u < 0.7, torch.full_like(tail, 2), tail.clamp_max(64))
    deg = torch.where(u >= 0.999, lo + torch.floor(v * (hi - lo + 1)).to(torch.int64), deg).clamp_max(max(2, n // 2))
    off, net, slot = _csr(deg)
    # distinct pins: a net's slots go through a bijection of its window of 2^m nodes
    m = torch.ceil(torch.log2((2 * deg).clamp_min(4096).double())).to(torch.int64)
    m = m.clamp_max(int(math.floor(math.log2(n))))
    a = torch.randint(0, 1 << 20, (e,), generator=gen, device="cuda") * 2 + 1
    b = torch.randint(0, 1 << 20, (e,), generator=gen, device="cuda")
    base = torch.floor(torch.rand(e, generator=gen, device="cuda", dtype=torch.float64) * (n - (1 << m) + 1)).to(torch.int64)
    mask = ((1 << m) - 1)[net]
    x = (slot * a[net] + b[net]) & mask
    x = x ^ (x >> ((m + 1) // 2)[net])
    x = (x * 0x9E3779B1) & mask
    nw = torch.randint(1, 5, (n,), generator=gen, device="cuda", dtype=torch.int32)
    return off, base[net] + x, nw


def _zipf(n):
    length = torch.arange(2, _row_cap(n) + 1, dtype=torch.float64)
    p = length.pow(-2.1)
    return length, p / p.sum()


def _rownet(n, gen):
    _, p = _zipf(n)
    u = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)
    deg = 2 + torch.searchsorted(torch.cumsum(p, 0).cuda(), u).clamp_max(p.numel() - 1)
    off, net, slot = _csr(deg)
    hubs = torch.randperm(n, generator=gen, device="cuda")[: max(1, n // 100)]
    hub = torch.rand(net.numel(), generator=gen, device="cuda") < 0.2
    pins = torch.randint(0, n, (net.numel(),), generator=gen, device="cuda")
    pick = torch.randint(0, hubs.numel(), (net.numel(),), generator=gen, device="cuda")
    return off, torch.where(hub, hubs[pick], pins), None


def _graph(shape, n, seed, hw=0):
    """One hypergraph as int32 CUDA tensors: (N, hoff, pins, node weights, hyperedge weights)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    off, pins, nw = {"uniform": _uniform, "netlist": _netlist, "rownet": _rownet}[shape](n, gen)
    w = torch.randint(1, hw + 1, (off.numel() - 1,), generator=gen, device="cuda", dtype=torch.int32) if hw else None
    return n, off.to(torch.int32), pins.to(torch.int32), nw, w


def _parts(n, k, seed):
    """Parts in runs of ids with a tenth moved at random: a partition with locality."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 1)
    parts = torch.arange(n, device="cuda") * k // n
    other = torch.randint(0, k, (n,), generator=gen, device="cuda")
    return torch.where(torch.rand(n, generator=gen, device="cuda") < 0.1, other, parts).to(torch.int32)


def _host(g):
    n, off, pins, nw, hw = g
    return dict(N=n, hoff=off.cpu().numpy(), pins=pins.cpu().numpy(),
                nw=None if nw is None else nw.cpu().numpy(), hw=None if hw is None else hw.cpu().numpy())


def _sizes(case):
    """Node counts of a batch's or burst's hypergraphs: spread over the logarithm of the range."""
    c, lo, hi = case["count"], math.log(case["n"]), math.log(case["n_max"])
    return [int(round(math.exp(lo + (hi - lo) * ((7 * i) % c) / max(1, c - 1)))) for i in range(c)]


def _options(case):
    return dict(k=case["k"], eps=case["eps"], policy=case["policy"], levels=LEVELS, iters=case["iters"],
                adaptive_eps=bool(case.get("adaptive")), merge_parallel=bool(case.get("merge")))


def _member_options(case, i):
    """Options of member i of a batch or burst."""
    k = (4 if i % 8 == 7 else 2) if case["call"] == "batch" else (2, 4, 16)[i % 3]
    return dict(k=k, eps=case["eps"], policy=case["policy"], levels=LEVELS, iters=case["iters"])


def _member_shape(case, i):
    return case["shape"] if case["shape"] != "mix" else ("netlist", "rownet")[i % 2]


_running = []  # the server a serving program keeps for its lifetime


def _server():
    if not _running:
        _running.append(bp.Server(hbm_budget_bytes=64 << 30, workers=8))
    return _running[0]


# ------------------------------------------------------------------------------- the interface
def prepare(case, seed):
    call = case["call"]
    s = dict(case=dict(case))
    if call in ("batch", "serve"):
        s["graphs"] = [_host(_graph(_member_shape(case, i), n, seed * 1_000_003 + i))
                       for i, n in enumerate(_sizes(case))]
        s["options"] = [_member_options(case, i) for i in range(len(s["graphs"]))]
        if call == "serve":
            s["server"] = _server()
        return s
    g = _graph(case["shape"], case["n"], seed, case.get("hw", 0))
    n = g[0]
    if call == "oneshot":
        s["graph"] = _host(g) if case["source"] == "host" else g
    elif call == "cut":
        parts = _parts(n, case["k"], seed)
        if case["source"] == "device":
            s.update(graph=g, parts=parts, out=torch.zeros(1, dtype=torch.int64, device="cuda"))
        else:
            s.update(handle=bp.create_device(*g), parts=parts.cpu().numpy())
    else:
        s["handle"] = bp.create_device(*g)
        if call == "refine":
            s["handle"].partition(2, 0.1, case["policy"], LEVELS, 2)
        else:
            s["out"] = torch.empty(n, dtype=torch.int32, device="cuda")
    return s


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "oneshot":
        g = state["graph"]
        h = bp.create_from(g) if case["source"] == "host" else bp.create_device(*g)
        parts, status = h.partition(**_options(case))
        h.close()
        return parts, status
    if call == "resident":
        status = state["handle"].partition_device(state["out"], **_options(case))
        return state["out"], status
    if call == "refine":
        return state["handle"].refine_kept(case["eps"], case["iters"])
    if call == "batch":
        parts, statuses = bp.partition_batch(state["graphs"], state["options"])
        return np.concatenate(parts), statuses
    if call == "serve":
        server = state["server"]
        tickets = [server.submit(g, **o) for g, o in zip(state["graphs"], state["options"])]
        done = [server.wait(t)[:2] for t in tickets]
        return [parts for parts, _ in done], [status for _, status in done]
    if case["source"] == "device":
        n, off, pins, _, hw = state["graph"]
        bp.cut_noalloc(n, off, pins, hw, state["parts"], case["k"], state["out"])
        return state["out"]
    return state["handle"].cut(state["parts"])


def _mean_pins(shape, n):
    """Expected pins of one hypergraph."""
    if shape == "uniform":
        return 4.0 * n
    if shape == "netlist":
        lo, hi = _fanout(n)
        return 1.2 * n * (0.7 * 2 + 0.299 * 4 + 0.001 * (lo + hi) / 2)
    length, p = _zipf(n)
    return n * float((length * p).sum())


def _graph_bytes(shape, n, hw):
    """Arrays of one hypergraph, read once: offsets, pins and the weights it has."""
    e = 1.2 * n if shape == "netlist" else n
    return 4.0 * (e + 1 + _mean_pins(shape, n) + (n if shape == "netlist" else 0) + (e if hw else 0))


def work(case):
    call = case["call"]
    if call in ("batch", "serve"):
        b = sum(_graph_bytes(_member_shape(case, i), n, 0) + 4.0 * n for i, n in enumerate(_sizes(case)))
    else:
        b = _graph_bytes(case["shape"], case["n"], case.get("hw", 0)) + 4.0 * case["n"]
    return {"bytes": b, "flops": 0.0}


def exact(case, seed):
    """The cut by sorting (hyperedge, part) pairs; partitions are whole numbers of the method's own."""
    if case["call"] != "cut":
        return None
    _, off, pins, _, hw = _graph(case["shape"], case["n"], seed, case.get("hw", 0))
    off, pins = off.cpu().numpy().astype(np.int64), pins.cpu().numpy()
    parts = _parts(case["n"], case["k"], seed).cpu().numpy()
    net = np.repeat(np.arange(off.size - 1), np.diff(off))
    pairs = np.unique(net * case["k"] + parts[pins])
    lam = np.bincount(pairs // case["k"], minlength=off.size - 1)
    w = np.ones(off.size - 1, np.int64) if hw is None else hw.cpu().numpy().astype(np.int64)
    cut = int((w * (lam - 1)).sum())
    return torch.tensor([cut]) if case["source"] == "device" else cut
