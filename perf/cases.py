"""The work a user of this library has it do, as measurable cases.

A multilevel partitioner contracts a hypergraph level by level, makes a handle of each level,
refines (and rebalances) its partition there and reads the partition back; a service refines
streams of small hypergraphs; a local-search caller asks for exact gains of move sequences.  Every
case goes through the package's public classes, on seeded synthetic hypergraphs drawn on the GPU
(the recipes of the benchmark: planted hypergraphs with Poisson or Zipf net sizes, and row-net
hypergraphs of banded sparse matrices).

A case's "path" says what one pass does:
  refine      new start partition into a resident handle, LP rounds, partition read into device memory
  level       handle from device arrays, LP rounds, partition into device memory, handle released
  request     handle from host arrays, LP rounds, partition into host memory, handle released
  batch       new start partitions into the members, one batched refinement, all partitions to the host
  rebalance   new (overloaded) start partition, rebalancing passes, partition into device memory
  contract    coarse hypergraph of a clustering, from device arrays into device arrays
  gains       exact gains of a move sequence against a resident handle, from and to host memory
  candidates  the allocation-free gain step over device arrays

All outputs are whole numbers and are the same on every run.
"""
import math

import numpy as np
import torch

from paper_2010_10272_gb300 import HGP, Batch, Coarse
from paper_2010_10272_gb300.native import candidates_noalloc

EPS = 0.03
SUBROUNDS = 4
CHUNK_NETS = 1 << 23
NOALLOC_MAX_NETS = 1 << 18


def listed():
    return [
        # the smallest call: a 10k-vertex bisection (small coarse level), launches and latency
        {"name": "refine-planted-10k", "path": "refine", "shape": "planted", "n": 10_000, "k": 2, "rounds": 5},
        # a small weighted level with uneven nets, an odd size, replayed as a CUDA graph
        {"name": "refine-zipf-30k-graph", "path": "refine", "shape": "zipf", "n": 30_011, "k": 16, "rounds": 5,
         "vertex_w": 4, "graph": True},
        # a sparse matrix's row-net hypergraph (20M pins) into 8 blocks
        {"name": "refine-rownet-2m", "path": "refine", "shape": "rownet", "n": 2_000_000, "k": 8, "rounds": 10},
        # the largest instance: 345M pins, 64 blocks, weighted nets of up to 100,000 pins
        {"name": "refine-powerlaw-50m", "path": "refine", "shape": "powerlaw", "n": 50_000_000, "k": 64, "rounds": 5,
         "net_w": 10},
        # both label-propagation variants on (zero-gain balance moves, reverts of negative moves)
        {"name": "refine-variants-3m", "path": "refine", "shape": "powerlaw", "n": 3_000_001, "k": 32, "rounds": 5,
         "net_w": 10, "balance_moves": True, "revert_negative": True},
        # one level of a multilevel hierarchy: its handle made from device arrays and used once
        {"name": "level-powerlaw-5m", "path": "level", "shape": "powerlaw", "n": 5_000_000, "k": 64, "rounds": 5,
         "net_w": 10},
        # one refinement request as a service gets it, in host memory (500k pins)
        {"name": "request-planted-83k", "path": "request", "shape": "planted", "n": 83_334, "k": 8, "rounds": 3},
        # a batch of uneven instances (1k to 200k vertices, k in {2,4,8,16}) refined together
        {"name": "batch-256", "path": "batch", "shape": "zipf", "count": 256, "n_lo": 1_000, "n_hi": 200_000,
         "k": 16, "vertex_w": 4, "rounds": 5},
        # a partition with a fifth of the vertices moved into one block, brought back into balance
        {"name": "rebalance-powerlaw-5m", "path": "rebalance", "shape": "powerlaw", "n": 5_000_000, "k": 64,
         "net_w": 10, "skew": 0.2, "passes": 16},
        # contraction of a large level by a pair clustering
        {"name": "contract-powerlaw-10m", "path": "contract", "shape": "powerlaw", "n": 10_000_000, "k": 64,
         "net_w": 10},
        # exact gains of 100k moves in sequence on a million vertices
        {"name": "gains-planted-1m", "path": "gains", "shape": "planted", "n": 1_000_000, "k": 16, "moves": 100_000},
        # the gain step without allocations, near its largest size
        {"name": "candidates-zipf-250k", "path": "candidates", "shape": "zipf", "n": 250_000, "k": 16, "vertex_w": 4,
         "net_w": 10},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["refine", "refine", "refine", "refine", "level", "request", "batch", "rebalance", "contract",
                       "gains", "candidates"])
    case = {"path": path, "shape": rng.choice(["planted", "zipf", "powerlaw", "rownet"])}
    top = {"refine": 10_000_000, "level": 5_000_000, "request": 800_000, "batch": 0, "rebalance": 5_000_000,
           "contract": 10_000_000, "gains": 2_000_000, "candidates": 250_000}[path]
    if path == "batch":
        case.update(shape="zipf", count=rng.randint(8, 256), n_lo=1_000, n_hi=_log_int(rng, 2_000, 200_000))
    else:
        case["n"] = _log_int(rng, 1_000, top)
    case["k"] = rng.choice([2, 4, 8, 16]) if path == "batch" else rng.randint(2, 64)
    if rng.random() < 0.5:
        case["vertex_w"] = 4
    if rng.random() < 0.5:
        case["net_w"] = 10
    if path in ("refine", "level", "request", "batch"):
        case["rounds"] = rng.randint(3, 10)
    if path == "refine":
        case["graph"] = rng.random() < 0.4
        if rng.random() < 0.25:
            case["balance_moves"] = True
        if rng.random() < 0.25:
            case["revert_negative"] = True
    if path == "rebalance":
        case.update(skew=round(rng.uniform(0.05, 0.5), 3), passes=16)
    if path == "gains":
        case["moves"] = max(1, int(case["n"] * rng.uniform(0.01, 0.2)))
    return case


# ---------------------------------------------------------------------------------- inputs
def _zipf(gen, count, a, cap, dev):
    """Zipf(a) draws, values above cap counted as cap."""
    p = np.arange(1, cap + 1, dtype=np.float64) ** -a
    tail = cap ** (1.0 - a) / (a - 1.0)          # weight of the values above cap
    cdf = torch.from_numpy(np.cumsum(p) / (p.sum() + tail)).to(dev)
    u = torch.rand(count, generator=gen, device=dev, dtype=torch.float64)
    return torch.clamp(torch.searchsorted(cdf, u) + 1, max=cap)


def _net_sizes(gen, shape, count, n, dev):
    if shape == "zipf":
        s = torch.clamp(2 + _zipf(gen, count, 2.5, 1000, dev), max=1000)
    elif shape == "powerlaw":
        s = torch.clamp(2 + _zipf(gen, count, 2.1, 100_000, dev), max=100_000)
    else:
        base, rate = (1, 9.0) if shape == "rownet" else (2, 4.0)
        s = base + torch.poisson(torch.full((count,), rate, device=dev), generator=gen).to(torch.int64)
    return torch.clamp(s, max=n)


def _hypergraph(case, gen, dev, n=None, k=None):
    """A hypergraph with n nets and its start partition, on `dev`: net_off int64 [n+1], pins int32,
    part int32 [n], vertex_w / net_w int32 [n] or None."""
    n, k, shape = n or case["n"], k or case["k"], case["shape"]
    p_in, f = {"powerlaw": (0.6, 0.4)}.get(shape, (0.8, 0.3))
    perm = torch.randperm(n, generator=gen, device=dev)
    group = torch.empty(n, dtype=torch.int64, device=dev)
    group[perm] = torch.arange(n, device=dev) % k
    gsize = (n - torch.arange(k, device=dev) + k - 1) // k
    sizes, pins = [], []
    for a in range(0, n, CHUNK_NETS):
        cnt = min(CHUNK_NETS, n - a)
        size = _net_sizes(gen, shape, cnt, n, dev)
        local = torch.repeat_interleave(torch.arange(cnt, device=dev), size)
        P = local.numel()
        home = torch.rand(P, generator=gen, device=dev) < (0.7 if shape == "rownet" else p_in)
        v = torch.randint(0, n, (P,), generator=gen, device=dev)
        if shape == "rownet":                    # columns near the diagonal
            band = min(5000, max(1, n // 8))
            near = torch.remainder(local + a + torch.randint(-band, band + 1, (P,), generator=gen, device=dev), n)
        else:                                    # members of the net's hidden group
            g = torch.randint(0, k, (cnt,), generator=gen, device=dev)[local]
            r = torch.rand(P, generator=gen, device=dev, dtype=torch.float64)
            at = torch.minimum((r * gsize[g]).to(torch.int64), gsize[g] - 1)
            near = perm[torch.clamp(g + k * at, max=n - 1)]
        key = torch.unique(local * n + torch.where(home, near, v))      # sorted pins, none twice
        net = key // n
        pins.append((key - net * n).to(torch.int32))
        sizes.append(torch.bincount(net, minlength=cnt))
    off = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    torch.cumsum(torch.cat(sizes), 0, out=off[1:])
    part = group
    if shape != "rownet":                        # the hidden groups, a fraction of them reassigned
        sel = torch.randperm(n, generator=gen, device=dev)[: int(round(f * n))]
        part[sel] = torch.randint(0, k, (sel.numel(),), generator=gen, device=dev)

    def weights(most):
        return torch.randint(1, most + 1, (n,), generator=gen, device=dev, dtype=torch.int32) if most else None
    return {"n": n, "m": n, "k": k, "net_off": off, "pins": torch.cat(pins), "part": part.to(torch.int32),
            "vertex_w": weights(case.get("vertex_w")), "net_w": weights(case.get("net_w"))}


def _generator(seed, dev):
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    return gen


def _handle(hg, **kw):
    return HGP(hg["n"], hg["m"], hg["net_off"], hg["pins"], hg["k"], EPS, hg["part"], hg["vertex_w"], hg["net_w"],
               subrounds=SUBROUNDS, **kw)


def _to_host(hg):
    return {key: v.cpu().numpy() if isinstance(v, torch.Tensor) else v for key, v in hg.items()}


def _clusters(gen, n, dev):
    """About n/2 clusters: a permutation cut into consecutive pairs."""
    perm = torch.randperm(n, generator=gen, device=dev)
    cluster = torch.empty(n, dtype=torch.int32, device=dev)
    cluster[perm] = perm[torch.arange(n, device=dev) // 2 * 2].to(torch.int32)
    return cluster


def _moves(gen, hg, count, dev):
    """count moves (u, from, to) of distinct vertices, each to another block."""
    u = torch.randperm(hg["n"], generator=gen, device=dev)[:count]
    a = hg["part"][u].to(torch.int64)
    b = (a + torch.randint(1, hg["k"], (u.numel(),), generator=gen, device=dev)) % hg["k"]
    return torch.stack([u, a, b], 1).to(torch.int32).cpu().numpy()


def _transpose(hg):
    """Vertex -> nets lists (int32), net ids increasing in each."""
    n, m = hg["n"], hg["m"]
    net = torch.repeat_interleave(torch.arange(m, device=hg["pins"].device), hg["net_off"].diff())
    v = hg["pins"].to(torch.int64)
    inc = (torch.sort(v * m + net)[0] % max(1, m)).to(torch.int32)
    off = torch.zeros(n + 1, dtype=torch.int32, device=v.device)
    off[1:] = torch.cumsum(torch.bincount(v, minlength=n), 0).to(torch.int32)
    return off, inc


class _DeviceArray:
    """A device array of `owner` for torch.as_tensor (no copy); the tensor keeps the owner alive."""

    def __init__(self, owner, ptr, count, typestr):
        self.owner = owner
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": (count,), "typestr": typestr, "version": 3}


def _coarse_arrays(c):
    """The arrays of a Coarse as tensors: (name, tensor)."""
    a = c.device_arrays()
    spec = {"net_off": (c.m + 1, "<i8"), "pins": (c.num_pins, "<i4"), "vertex_w": (c.n, "<i4"), "net_w": (c.m, "<i4"),
            "map": (c.fine_n, "<i4")}
    return [(key, torch.as_tensor(_DeviceArray(c, a[key], n, t), device="cuda")) for key, (n, t) in spec.items() if n]


def prepare(case, seed):
    dev = torch.device("cuda")
    gen = _generator(seed, dev)
    path = case["path"]
    state = {"case": dict(case), "seed": seed}
    if path == "batch":
        rng = np.random.default_rng(case["count"])       # sizes of the members, by the case alone
        hs, parts = [], []
        for _ in range(case["count"]):
            n = int(math.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]))))
            hg = _hypergraph(case, gen, dev, n=n, k=int(rng.choice([k for k in (2, 4, 8, 16) if k <= case["k"]])))
            hs.append(_handle(hg, device=True))
            parts.append(hg["part"])
        state.update(handles=hs, parts=parts, batch=Batch(hs))
        return state
    hg = _hypergraph(case, gen, dev)
    if path in ("refine", "rebalance"):
        if path == "rebalance":
            hg["part"][torch.rand(hg["n"], generator=gen, device=dev) < case["skew"]] = 0
        state["handle"] = _handle(hg, device=True, graph=int(case.get("graph", False)),
                                  balance_moves=case.get("balance_moves", False),
                                  revert_negative=case.get("revert_negative", False))
        state["part"] = hg["part"]
    elif path == "gains":
        state["handle"] = _handle(hg, device=True)
        state["moves"] = _moves(gen, hg, case["moves"], dev)
    elif path == "candidates":
        state["hg"] = {**hg, "net_off": hg["net_off"].to(torch.int32)}
        state["transpose"] = _transpose(hg)
        state["gain"] = torch.empty(hg["n"], dtype=torch.int64, device=dev)
    elif path == "contract":
        state.update(hg=hg, cluster=_clusters(gen, hg["n"], dev))
        # the caller's own buffers for the coarse arrays, sized by the case
        room = {"net_off": hg["n"] + 1, "vertex_w": hg["n"], "net_w": hg["n"], "map": hg["n"],
                "pins": max(hg["pins"].numel(), int(1.5 * _MEAN_SIZE[case["shape"]] * hg["n"]) + 100_000)}
        state["room"] = {key: torch.zeros(size, dtype=torch.int64 if key == "net_off" else torch.int32, device=dev)
                         for key, size in room.items()}
    else:
        state["hg"] = _to_host(hg) if path == "request" else hg
    if path != "request":
        state["out"] = torch.empty(hg["n"], dtype=torch.int32, device=dev)
    return state


# ---------------------------------------------------------------------------------- one pass
def run(state):
    case = state["case"]
    path = case["path"]
    if path == "refine":
        h = state["handle"]
        h.set_partition(state["part"], device=True)
        stats = h.refine(case["rounds"])
        h.partition(out_device=state["out"])
        return {"partition": state["out"], "stats": stats}
    if path == "level":
        with _handle(state["hg"], device=True) as h:
            stats = h.refine(case["rounds"])
            h.partition(out_device=state["out"])
        return {"partition": state["out"], "stats": stats}
    if path == "request":
        with _handle(state["hg"]) as h:
            stats = h.refine(case["rounds"])
            part = h.partition()
        return {"partition": part, "stats": stats}
    if path == "batch":
        for h, p in zip(state["handles"], state["parts"]):
            h.set_partition(p, device=True)
        stats = state["batch"].refine(case["rounds"])
        parts = state["batch"].partitions(range(len(state["handles"])))
        return {"partitions": np.concatenate(parts), "stats": stats}
    if path == "rebalance":
        h = state["handle"]
        h.set_partition(state["part"], device=True)
        stats, phases = h.rebalance(case["passes"])
        h.partition(out_device=state["out"])
        return {"partition": state["out"], "stats": stats, "phases": phases}
    if path == "contract":
        hg, room = state["hg"], state["room"]
        c = Coarse(hg["n"], hg["m"], hg["net_off"], hg["pins"], hg["vertex_w"], hg["net_w"], state["cluster"])
        for key, t in _coarse_arrays(c):
            room[key][: t.numel()].copy_(t)
        return {**room, "n": c.n, "m": c.m, "pin_count": c.num_pins}
    if path == "gains":
        return {"gains": state["handle"].exact_gains(state["moves"])}
    hg = state["hg"]
    rc = candidates_noalloc(hg["n"], hg["m"], hg["net_off"], hg["pins"], *state["transpose"], hg["k"], EPS, hg["part"],
                            state["out"], state["gain"], hg["vertex_w"], hg["net_w"], subrounds=SUBROUNDS,
                            seed=0, s=0, stream=torch.cuda.current_stream())
    return {"status": rc, "target": state["out"], "gain": state["gain"]}


# ---------------------------------------------------------------------------------- least work
_MEAN_SIZE = {"planted": 6.0, "rownet": 10.0, "zipf": 3.9, "powerlaw": 6.9}   # pins of a net, about


def work(case):
    """Bytes each pass reads or writes once, and its additions.  Refinement visits every incidence
    against the state each round left, so the lists count once a round."""
    mean = _MEAN_SIZE[case["shape"]]
    path = case["path"]
    if path == "batch":     # n log-uniform: its mean
        n = case["count"] * (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])
    else:
        n = case["n"]
    P = mean * n
    wv, wn = 4 * n * bool(case.get("vertex_w")), 4 * n * bool(case.get("net_w"))
    lists = 4 * n + 4 * P + wv + wn                  # vertex -> nets lists and weights
    if path in ("refine", "batch"):
        r = case["rounds"]
        return {"bytes": r * lists + 8 * n, "flops": 2 * r * P}
    if path in ("level", "request"):
        r = case["rounds"]
        return {"bytes": r * lists + 8 * n + 8 * n + 4 * P, "flops": 2 * r * P}
    if path == "rebalance":
        return {"bytes": lists + 8 * n, "flops": 2 * P}
    if path == "contract":  # the input, the map and about as many coarse pins and nets
        return {"bytes": 8 * n + 4 * P + wv + wn + 4 * n + 4 * n + 0.9 * (4 * P + 8 * n + 4 * n) + 2 * n, "flops": P}
    if path == "gains":     # the moved vertices' lists and pin counts, moves and gains
        return {"bytes": case["moves"] * (12 + 8 + 8 + mean * (4 + 2)), "flops": 4 * mean * case["moves"]}
    return {"bytes": 2 * (4 * n + 4 * P) + wv + wn + 4 * n + 12 * n, "flops": 2 * P}


# ---------------------------------------------------------------------------------- exact results
def _sub_round(u, r):
    """SplitMix64 output of seed 0 ^ (r << 32 | u), modulo SUBROUNDS (a power of two)."""
    def shift(z, s):
        return (z >> s) & ((1 << (64 - s)) - 1)
    z = u | (r << 32)
    z = (z ^ shift(z, 30)) * (0xBF58476D1CE4E5B9 - (1 << 64))
    z = (z ^ shift(z, 27)) * (0x94D049BB133111EB - (1 << 64))
    return (z ^ shift(z, 31)) & (SUBROUNDS - 1)


class _Plain:
    """The rounds of the default options in plain torch, 64-bit."""

    def __init__(self, hg):
        dev = hg["pins"].device
        self.n, self.m, self.k = hg["n"], hg["m"], hg["k"]
        self.v = hg["pins"].to(torch.int64)
        self.e = torch.repeat_interleave(torch.arange(self.m, device=dev), hg["net_off"].to(torch.int64).diff())
        one = torch.ones(self.n, dtype=torch.int64, device=dev)
        self.c = one if hg["vertex_w"] is None else hg["vertex_w"].to(torch.int64)
        self.w = torch.ones(self.m, dtype=torch.int64, device=dev) if hg["net_w"] is None else hg["net_w"].to(torch.int64)
        self.part = hg["part"].to(torch.int64)
        self.u = torch.arange(self.n, device=dev)
        self.W = torch.zeros_like(one).index_add_(0, self.v, self.w[self.e])
        self.lmax = math.floor((1.0 + EPS) * float(-(-int(self.c.sum()) // self.k)))
        self.count()

    def count(self):
        k = self.k
        self.phi = torch.bincount(self.e * k + self.part[self.v], minlength=self.m * k).view(self.m, k)
        self.bw = torch.zeros(k, dtype=torch.int64, device=self.v.device).index_add_(0, self.part, self.c)
        lam = (self.phi > 0).sum(1)
        return int(((lam - 1).clamp(min=0) * self.w).sum())

    def best(self, active):
        """Best target and gain of every active vertex (target -1: none)."""
        on = active[self.v].nonzero()[:, 0]
        v, e = self.v[on], self.e[on]
        alone = self.phi[e, self.part[v]] == 1
        b = torch.zeros(self.n, dtype=torch.int64, device=v.device).index_add_(0, v, self.w[e] * alone)
        g = torch.zeros(self.n, self.k, dtype=torch.int64, device=v.device)
        g.index_add_(0, v, (self.phi[e] > 0) * self.w[e][:, None])
        g += (b - self.W)[:, None]
        g[self.bw[None, :] + self.c[:, None] > self.lmax] = 0
        g[self.u, self.part] = 0
        key = g * self.k + torch.arange(self.k - 1, -1, -1, device=v.device)     # smallest block on ties
        t = key.argmax(1)
        g = g[self.u, t]
        ok = active & (g > 0)
        return torch.where(ok, t, -1), torch.where(ok, g, 0)

    def round(self, r, moved):
        elig = torch.ones_like(self.u, dtype=torch.bool)
        if moved is not None:
            elig = torch.zeros_like(elig)
            elig[self.v[moved[self.e]]] = True
        sub, now = _sub_round(self.u, r), torch.zeros(self.m, dtype=torch.bool, device=self.v.device)
        cand = appr = pins = 0
        for s in range(SUBROUNDS):
            t, g = self.best(elig & (sub == s))
            x = (t >= 0).nonzero()[:, 0]
            order = x[torch.argsort((t[x] * (1 << 32) - g[x]), stable=True)]     # block, gain desc, id asc
            c = self.c[order]
            run = torch.cumsum(c, 0)
            first = torch.searchsorted(t[order].contiguous(), t[order].contiguous())
            prefix = run - (run - c)[first] if order.numel() else run
            go = order[prefix <= self.lmax - self.bw[t[order]]]
            mask = torch.zeros_like(elig)
            mask[go] = True
            at = mask[self.v]
            now[self.e[at]] = True
            self.part[go] = t[go]
            cand, appr, pins = cand + int(x.numel()), appr + int(go.numel()), pins + int(at.sum())
            obj = self.count()
        return [obj, cand, appr, int(elig.sum()), int(self.bw.max()), pins, 0], now


def exact(case, seed):
    """What run() returns, from the rounds in plain torch; None for the paths whose outputs would take
    too long that way (all outputs are whole numbers, so they are compared bit by bit anyhow)."""
    path = case["path"]
    if path not in ("refine", "level", "request", "candidates") or case.get("balance_moves") or case.get("revert_negative"):
        return None
    if case["n"] * case["k"] * case.get("rounds", 1) > 200_000_000:
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    p = _Plain(_hypergraph(case, _generator(seed, dev), dev))
    if path == "candidates":
        t, g = p.best(_sub_round(p.u, 0) == 0)
        return {"status": 0, "target": t.to(torch.int32), "gain": g}
    stats, moved = [], None
    for r in range(case["rounds"]):
        row, moved = p.round(r, moved)
        stats.append(row)
    part = p.part.to(torch.int32)
    return {"partition": part.cpu().numpy() if path == "request" else part, "stats": np.array(stats, dtype=np.int64)}
