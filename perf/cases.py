"""What a user of this library has it do, as cases that can be timed.

A case is one of five calls:

  update   one batch of capacity updates, then the answer (Solver.update, Solver.query):
           the dynamic max-flow stream, which is what the library is for
  static   the current graph solved again from zero flow (Solver.resolve_static)
  batched  many uneven instances in one launch (maxflow_solve_batched without batches)
  tick     one launch that updates several resident graphs, as the serving loop issues it
  oneshot  a graph in host memory to its minimum cut: Solver(...), query, close

Graphs are drawn on the GPU from the seed: Erdos-Renyi, R-MAT (a/b/c = 0.57/0.19/0.19,
terminals as in workloads.rmat) and the segmentation grid of workloads.GridSegmentation.
A stream of updates has four batches, each followed by the batch that takes it back, so
that its passes are all real changes however often it runs; on the grid it is the
segmentation window that moves over the image.

Every output is a whole number and does not depend on the flow that was found: the value,
the capacity of the minimum cut, and its source side.  The side is the set of vertices that
cannot reach t in the residual graph of a maximum flow, which is the same for all of them.
"""
import math
import random

import numpy as np
import torch

from paper_2511_01235_gb300 import native
from paper_2511_01235_gb300 import workloads as W

DEVICE = "cuda"


def listed():
    """Smallest calls first; sizes are those of bench.py, the tests and the scheduler's families,
    the largest ones cut down to what can be prepared in a few seconds."""
    return [
        # an interactive what-if on the small Erdos-Renyi graph of the tests: a handful of edges change
        {"name": "er4096_b16", "path": "update", "family": "er", "n": 4096, "m": 32768, "cap_hi": 100,
         "batch": 16, "kind": "mixed", "host": True, "cut": True, "gseed": 0},
        # the paper-shaped small stream: 256 mixed updates a batch from host arrays, with the cut certificate
        {"name": "er4096_b256", "path": "update", "family": "er", "n": 4096, "m": 32768, "cap_hi": 100,
         "batch": 256, "kind": "mixed", "host": True, "cut": True, "gseed": 0},
        # a mid-sized sparse graph of odd size whose capacities go up and down (no insertion or deletion)
        {"name": "er60001_b1500", "path": "update", "family": "er", "n": 60001, "m": 480013, "cap_hi": 500,
         "batch": 1500, "kind": "reweight", "host": False, "cut": True, "gseed": 0},
        # a power-law graph that fits in L2, batches already on the device
        {"name": "rmat16_b1000", "path": "update", "family": "rmat", "scale": 16, "ef": 16, "cap_hi": 1000,
         "batch": 1000, "kind": "mixed", "host": False, "cut": False, "gseed": 0},
        # a large batch on a mid-sized power-law graph: 100 000 updates, 2.5 % of the edges
        {"name": "rmat18_b100k", "path": "update", "family": "rmat", "scale": 18, "ef": 16, "cap_hi": 1000,
         "batch": 100000, "kind": "mixed", "host": False, "cut": False, "gseed": 0},
        # bench.py's headline: a million vertices, 16 M edges, 10 000 mixed updates a batch
        {"name": "rmat20_b10k", "path": "update", "family": "rmat", "scale": 20, "ef": 16, "cap_hi": 1000,
         "batch": 10000, "kind": "mixed", "host": False, "cut": False, "gseed": 0},
        # interactive segmentation: the t-links of a 128 x 128 window of a megapixel image are drawn anew
        {"name": "grid1024_w128", "path": "update", "family": "grid", "side": 1024, "window": 128,
         "host": True, "cut": False, "gseed": 0},
        # the comparator: a whole re-solve of a power-law graph ...
        {"name": "rmat18_static", "path": "static", "family": "rmat", "scale": 18, "ef": 16, "cap_hi": 1000,
         "cut": True, "gseed": 0},
        # ... and of a segmentation grid, where the flow travels far
        {"name": "grid512_static", "path": "static", "family": "grid", "side": 512, "cut": True, "gseed": 0},
        # 64 uneven small instances (Erdos-Renyi, layered, geometric) in one launch
        {"name": "batched64", "path": "batched", "count": 64, "n_lo": 1000, "n_hi": 20000, "cap_hi": 500,
         "gseed": 0},
        # one tick of the server: a waiting batch for each of six resident power-law graphs
        {"name": "tick6", "path": "tick", "scales": "14,15,15,16,16,17", "ef": 16, "cap_hi": 1000,
         "batch_lo": 10, "batch_hi": 20000, "host": True, "gseed": 0},
        # a graph that is solved once: edge list in host memory to its minimum cut
        {"name": "oneshot_rmat16", "path": "oneshot", "family": "rmat", "scale": 16, "ef": 16, "cap_hi": 1000,
         "cut": True, "gseed": 0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any call, any family, sizes over the whole range on a log scale (odd ones too)."""
    path = rng.choice(["update", "update", "update", "static", "batched", "tick", "oneshot"])
    c = {"path": path, "gseed": rng.randrange(1, 1 << 16)}
    if path == "batched":
        c.update(count=rng.randrange(5, 65), n_lo=1000, n_hi=_log_int(rng, 1500, 20000), cap_hi=500)
        return c
    if path == "tick":
        k = rng.randrange(2, 7)
        c.update(scales=",".join(str(rng.randrange(13, 18)) for _ in range(k)), ef=rng.randrange(8, 17),
                 cap_hi=1000, batch_lo=10, batch_hi=_log_int(rng, 500, 20000), host=bool(rng.randrange(2)))
        return c
    c["cut"] = bool(rng.randrange(2))
    family = c["family"] = rng.choice(["er", "rmat", "grid"])
    if family == "er":
        n = _log_int(rng, 1001, 200000)
        c.update(n=n, m=int(n * rng.uniform(4, 12)), cap_hi=rng.choice([100, 500, 1000]))
        edges = c["m"]
    elif family == "rmat":
        top = {"update": 19, "static": 18, "oneshot": 16}[path]
        c.update(scale=rng.randrange(12, top + 1), ef=rng.randrange(8, 17), cap_hi=1000)
        edges = c["ef"] << c["scale"]
    else:
        top = {"update": 800, "static": 512, "oneshot": 300}[path]
        c.update(side=_log_int(rng, 65, top))
        edges = 6 * c["side"] ** 2
    if path == "update":
        c["host"] = bool(rng.randrange(2))
        if family == "grid":
            c["window"] = rng.randrange(16, min(128, c["side"] // 2) + 1)
        else:
            c.update(batch=min(_log_int(rng, 10, 100000), edges // 16), kind=rng.choice(["mixed", "reweight"]))
    return c


# ---- graphs, drawn on the GPU ----------------------------------------------------


def _gen(seed, salt):
    g = torch.Generator(device=DEVICE)
    g.manual_seed((int(seed) * 1000003 + int(salt) * 7919 + 17) & 0x7FFFFFFFFFFF)
    return g


def _ints(g, lo, hi, size):
    """Uniform whole numbers in [lo, hi]."""
    return torch.randint(lo, hi + 1, (size,), generator=g, device=DEVICE)


class _Drawn:
    """n, the sorted keys u * n + v of the edges, their capacities, and the terminals."""

    def __init__(self, n, keys, cap, s, t):
        self.n, self.keys, self.cap, self.s, self.t = n, keys, cap, s, t

    def host(self):
        """(n, src, dst, cap, s, t) as a user's program has them: int32 arrays in host memory."""
        u, v = self.keys // self.n, self.keys % self.n
        return (self.n, u.int().cpu().numpy(), v.int().cpu().numpy(), self.cap.int().cpu().numpy(), self.s, self.t)


def _er(n, m, cap_hi, g):
    keys = torch.empty(0, dtype=torch.int64, device=DEVICE)
    while keys.numel() < m:
        k = m - keys.numel() + (m >> 6) + 64
        u, v = _ints(g, 0, n - 1, k), _ints(g, 0, n - 1, k)
        keys = torch.unique(torch.cat([keys, (u * n + v)[u != v]]))
    if keys.numel() > m:
        keys = keys[torch.randperm(keys.numel(), generator=g, device=DEVICE)[:m]].sort().values
    return _Drawn(n, keys, _ints(g, 1, cap_hi, m), 0, n - 1)


def _reached(n, src, dst, root, both):
    """Breadth-first level of every vertex from root (-1: not reached)."""
    lev = torch.full((n,), -1, dtype=torch.int64, device=DEVICE)
    lev[root] = 0
    L = 0
    while True:
        hit = dst[(lev[src] == L) & (lev[dst] < 0)]
        if both:
            hit = torch.cat([hit, src[(lev[dst] == L) & (lev[src] < 0)]])
        if hit.numel() == 0:
            return lev
        L += 1
        lev[hit] = L


def _rmat(scale, ef, cap_hi, g, a=0.57, b=0.19, c=0.19):
    n, M = 1 << scale, ef << scale
    u = torch.zeros(M, dtype=torch.int64, device=DEVICE)
    v = torch.zeros(M, dtype=torch.int64, device=DEVICE)
    for _ in range(scale):
        low = torch.rand(M, generator=g, device=DEVICE) >= a + b
        thr = torch.where(low, c / (1 - a - b), a / (a + b))
        right = torch.rand(M, generator=g, device=DEVICE) >= thr
        u, v = 2 * u + low, 2 * v + right
    keys = torch.unique((u * n + v)[u != v])
    u, v = keys // n, keys % n
    deg = torch.bincount(u, minlength=n) + torch.bincount(v, minlength=n)
    # the terminals: the vertex of highest degree, and the highest one that it reaches in the far half
    # of an undirected breadth-first order from it
    s = int(deg.argmax())
    lev = _reached(n, u, v, s, True)
    order = torch.argsort(torch.where(lev < 0, 1 << 40, lev), stable=True)[:int((lev >= 0).sum())]
    far = order[order.numel() // 2:]
    far = far[(_reached(n, u, v, s, False)[far] >= 0) & (far != s)]
    t = int(far[deg[far].argmax()])
    return _Drawn(n, keys, _ints(g, 1, cap_hi, keys.numel()), s, t)


def _layered(n, cap_hi, g, layers=16, fanout=8):
    """s to layer 0, every vertex to `fanout` vertices of the next layer, the last layer to t."""
    inner = max(n - 2, layers)
    first = torch.tensor([inner * i // layers for i in range(layers + 1)], device=DEVICE)
    v = torch.arange(inner, device=DEVICE)
    at = torch.searchsorted(first, v, right=True) - 1
    mid = v[at < layers - 1].repeat_interleave(fanout)
    nxt = at[mid] + 1
    size = first[nxt + 1] - first[nxt]
    to = first[nxt] + (torch.rand(mid.numel(), generator=g, device=DEVICE) * size).long().clamp(max=int(size.max()) - 1)
    to = torch.minimum(to, first[nxt + 1] - 1)
    s, t, nn = inner, inner + 1, inner + 2
    keys = torch.cat([mid * nn + to, s * nn + v[at == 0], v[at == layers - 1] * nn + t])
    keys = torch.unique(keys)
    return _Drawn(nn, keys, _ints(g, 1, cap_hi, keys.numel()), s, t)


def _graph(case, seed):
    g = _gen(seed, case["gseed"])
    if case["family"] == "er":
        return _er(case["n"], case["m"], case["cap_hi"], g)
    return _rmat(case["scale"], case["ef"], case["cap_hi"], g)


def _grid(case, seed):
    side, w = case["side"], case.get("window", 16)
    at = max(0, (side - w) // 2)
    step = max(1, min(8, (side - w - at) // 8))       # 8 px a batch, as far as the image reaches
    return W.GridSegmentation(side=side, seed=int(seed) * 31 + case["gseed"] + 3, window=w, origin=(at, at), step=step)


def _mixed_pair(d, B, kind, g, inc_hi=50):
    """A batch and the batch that takes it back.  mixed: 40 % raised by U[1, 50], 40 % lowered to
    U[0, c], 10 % new pairs, 10 % deleted; reweight: half raised, half lowered."""
    n, m = d.n, d.keys.numel()
    n_ins = B // 10 if kind == "mixed" else 0
    n_del = B // 10 if kind == "mixed" else 0
    n_inc = (B - n_ins - n_del) // 2
    idx = torch.randperm(m, generator=g, device=DEVICE)[:B - n_ins]
    old = d.cap[idx]
    new = torch.floor(torch.rand(idx.numel(), generator=g, device=DEVICE) * (old + 1)).long().clamp(max=1 << 30)
    new = torch.minimum(new, old)
    new[:n_inc] = old[:n_inc] + _ints(g, 1, inc_hi, n_inc)
    if n_del:
        new[idx.numel() - n_del:] = 0
    keys = d.keys[idx]
    if n_ins:
        fresh = torch.empty(0, dtype=torch.int64, device=DEVICE)
        while fresh.numel() < n_ins:
            u, v = _ints(g, 0, n - 1, 2 * n_ins + 16), _ints(g, 0, n - 1, 2 * n_ins + 16)
            lo, hi = torch.minimum(u, v), torch.maximum(u, v)
            k = (lo * n + hi)[lo != hi]
            there = torch.zeros(k.numel(), dtype=torch.bool, device=DEVICE)
            for q in (k, (k % n) * n + k // n):
                p = torch.searchsorted(d.keys, q).clamp(max=m - 1)
                there |= d.keys[p] == q
            fresh = torch.unique(torch.cat([fresh, k[~there]]))
        fresh = fresh[torch.randperm(fresh.numel(), generator=g, device=DEVICE)[:n_ins]]
        keys = torch.cat([keys, fresh])
        old = torch.cat([old, torch.zeros(n_ins, dtype=torch.int64, device=DEVICE)])
        new = torch.cat([new, _ints(g, 1, int(d.cap.max()), n_ins)])
    p = torch.randperm(keys.numel(), generator=g, device=DEVICE)
    keys, old, new = keys[p], old[p], new[p]
    u, v = (keys // n).int(), (keys % n).int()
    return [(u, v, new.int()), (u, v, old.int())]


def _as_user(batches, host):
    """Device batches are int32 tensors; host batches are int32 arrays in pageable memory."""
    return [tuple(x.cpu().numpy() if host else x for x in b) for b in batches]


def _stream(d, case, seed, count=4):
    out = []
    for k in range(count):
        out += _mixed_pair(d, case["batch"], case["kind"], _gen(seed, 100 + k))
    return _as_user(out, case["host"])


def _instances(case, seed):
    sizes, r = random.Random(case["gseed"]), random.Random(int(seed) * 131 + case["gseed"])
    out = []
    for i in range(case["count"]):
        n = _log_int(sizes, case["n_lo"], case["n_hi"])
        g = _gen(seed, 1000 * case["gseed"] + i)
        if i % 3 == 0:
            out.append(_er(n, 8 * n, case["cap_hi"], g).host())
        elif i % 3 == 1:
            out.append(_layered(n, case["cap_hi"], g).host())
        else:
            q = W.geometric(n, seed=r.randrange(1 << 30), cap_hi=case["cap_hi"])
            out.append((q.n, q.src, q.dst, q.cap, q.s, q.t))
    return out


# ---- what a user's program has in hand, and the call --------------------------------


def prepare(case, seed):
    path = case["path"]
    if path == "batched":
        return {"path": path, "S": [native.Solver(*h) for h in _instances(case, seed)]}
    if path == "tick":
        r = random.Random(int(seed) * 17 + case["gseed"])
        solvers, ticks = [], [[] for _ in range(8)]
        for i, scale in enumerate(int(x) for x in case["scales"].split(",")):
            d = _rmat(scale, case["ef"], case["cap_hi"], _gen(seed, 10 * case["gseed"] + i))
            solvers.append(native.Solver(*d.host()))
            for k in range(4):
                B = min(_log_int(r, case["batch_lo"], case["batch_hi"]), d.keys.numel() // 8)
                pair = _as_user(_mixed_pair(d, B, "mixed", _gen(seed, 1000 + 10 * i + k)), case["host"])
                ticks[2 * k].append(pair[0])
                ticks[2 * k + 1].append(pair[1])
        return {"path": path, "S": solvers, "ticks": ticks, "i": 0}
    if case["family"] == "grid":
        gs = _grid(case, seed)
        q = gs.graph()
        host = (q.n, q.src, q.dst, q.cap, q.s, q.t)
    else:
        d = _graph(case, seed)
        host = d.host()
    if path == "oneshot":
        return {"path": path, "host": host, "cut": case["cut"]}
    state = {"path": path, "S": native.Solver(*host), "cut": case["cut"], "i": 0}
    if path == "update":
        if case["family"] == "grid":
            dev = [tuple(torch.from_numpy(x).to(DEVICE) for x in (b.u, b.v, b.cap))
                   for b in (gs.window_batch(k) for k in range(8))]
            state["batches"] = _as_user(dev, case["host"])
        else:
            state["batches"] = _stream(d, case, seed)
    return state


def _answer(S, cut):
    value, side, cap = S.query(side=True, cut=cut)
    return [value, side, cap] if cut else [value, side]


def run(state):
    path = state["path"]
    if path == "oneshot":
        S = native.Solver(*state["host"])
        out = _answer(S, state["cut"])
        S.close()
        return out
    S = state["S"]
    if path == "batched":
        native.maxflow_solve_batched(S)
        got = [s.query(side=True) for s in S]
        return [np.array([g[0] for g in got]), np.concatenate([g[1] for g in got])]
    if path == "static":
        S.resolve_static()
        return _answer(S, state["cut"])
    todo = state["ticks"] if path == "tick" else state["batches"]
    b = todo[state["i"] % len(todo)]
    state["i"] += 1
    if path == "tick":
        native.maxflow_solve_batched(S, b)
        return [np.array([s.value for s in S])] + [s.query(side=True)[1] for s in S]
    S.update(*b)
    return _answer(S, state["cut"])


# ---- the least that a pass has to move ------------------------------------------------


def _sizes(case):
    """Vertices, and slots of the residual graph (two for every joined pair; R-MAT loses the
    duplicates among its draws, some 2 to 20 %, which is left out here)."""
    f = case["family"]
    if f == "er":
        return case["n"], 2 * case["m"]
    if f == "rmat":
        return 1 << case["scale"], 2 * (case["ef"] << case["scale"])
    return case["side"] ** 2 + 2, 8 * case["side"] ** 2


def work(case):
    """An update has to read its records (12 bytes each) and, for each, read and write both slots of its pair
    (capacity and residual, 32 bytes), and to read a label and write a side for each vertex.  A solve from
    zero flow reads head and capacity of every slot once and writes every residual (12 bytes a slot), and
    writes an excess, a label and a side for each vertex; a graph that comes from the host is read once on
    top (12 bytes an edge).  Whole-number work only: no floating operations."""
    path = case["path"]
    if path == "batched":
        mean = (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])
        n, slots = case["count"] * mean, case["count"] * mean * 16
    elif path == "tick":
        scales = [int(x) for x in case["scales"].split(",")]
        n = sum(1 << s for s in scales)
        per = (case["batch_hi"] - case["batch_lo"]) / math.log(case["batch_hi"] / case["batch_lo"])
        return {"bytes": 44 * per * len(scales) + 5 * n, "flops": 0}
    else:
        n, slots = _sizes(case)
    if path == "update":
        B = 2 * case["window"] ** 2 if case["family"] == "grid" else case["batch"]
        return {"bytes": 44 * B + 5 * n, "flops": 0}
    return {"bytes": 12 * slots + 13 * n + (6 * slots if path == "oneshot" else 0), "flops": 0}


# ---- the same answers without this repository's code ------------------------------------


def exact(case, seed):
    """The answer of the first pass by plain augmenting paths (whole numbers of any size) for the
    Erdos-Renyi graphs that Python gets through in seconds; None for the others."""
    if case["path"] == "tick" or case["path"] == "batched" or case["family"] != "er" or case["m"] > 40000:
        return None
    d = _graph(case, seed)
    cap = dict(zip(d.keys.tolist(), d.cap.tolist()))
    if case["path"] == "update":
        u, v, c = _mixed_pair(d, case["batch"], case["kind"], _gen(seed, 100))[0]
        cap.update(zip((u.long() * d.n + v.long()).tolist(), c.tolist()))
    value, side = _augment(d.n, cap, d.s, d.t)
    return [value, side, value] if case["cut"] else [value, side]


def _augment(n, cap, s, t):
    """Dinic's algorithm on {u * n + v: capacity}: the value, and the vertices that cannot reach t at the end."""
    to, res, adj = [], [], [[] for _ in range(n)]
    for k, c in cap.items():
        u, v = divmod(k, n)
        adj[u].append(len(to))
        adj[v].append(len(to) + 1)
        to += [v, u]
        res += [c, 0]
    value = 0
    while True:
        # levels towards t over residual edges, then paths that go down one level at a time
        lev = [-1] * n
        lev[t] = 0
        queue = [t]
        for x in queue:
            for e in adj[x]:
                y = to[e]
                if res[e ^ 1] > 0 and lev[y] < 0:
                    lev[y] = lev[x] + 1
                    queue.append(y)
        if lev[s] < 0:
            return value, np.array([l < 0 for l in lev])
        at, path, x = [0] * n, [], s
        while True:
            if x == t:
                push = min(res[e] for e in path)
                value += push
                for e in path:
                    res[e] -= push
                    res[e ^ 1] += push
                path, x = [], s
                continue
            while at[x] < len(adj[x]):
                e = adj[x][at[x]]
                if res[e] > 0 and lev[to[e]] == lev[x] - 1:
                    break
                at[x] += 1
            if at[x] < len(adj[x]):
                path.append(adj[x][at[x]])
                x = to[path[-1]]
            elif path:
                e = path.pop()
                x = to[e ^ 1]
                at[x] += 1
            else:
                break
