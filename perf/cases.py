"""The work that a program built on this framework has it do, as measurable cases.

A case names a flow network (``kind`` and its sizes), how the resident graph
is set up (``mode``, ``kc``, ``policy``) and what one pass does with it
(``act``):

* ``repair``     the next ``batches`` update batches of ``k`` entries of a
                 stream, the flow value read after each one (the dynamic
                 max-flow use); with ``cut`` the minimum cut is read too
* ``recompute``  the same stream, every batch answered by a static recompute
* ``solve``      one static solve of a resident graph, its value and its cut
* ``oneshot``    one graph from host CSR arrays: build, solve, value, cut
* ``serve``      requests for several resident graphs through the server

A stream is much longer than a pass, so that most passes bring batches that
the graph has not met: its first half changes edge sets drawn afresh for every
batch, its second half puts them back in reverse order, and then it starts
over.  Every batch holds raises and cuts in equal parts (grids: the terminal
capacities of a square).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2511_05895_gb300 as mf

MODES = {"data-driven": mf.MF_MODE_DATA_DRIVEN, "topology": mf.MF_MODE_TOPOLOGY, "push-pull": mf.MF_MODE_PUSH_PULL}


def _case(kind, act, *, n=0, m=0, scale=0, w=0, h=0, left=0, right=0, mode="data-driven", kc=0, policy="fixed",
          k=0, batches=8, host=False, delta=False, cut=False, name=None):
    c = dict(kind=kind, act=act, n=n, m=m, scale=scale, w=w, h=h, left=left, right=right, mode=mode, kc=kc,
             policy=policy, k=k, batches=batches, host=host, delta=delta, cut=cut)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a small network re-solved after every handful of changes: the latency of one call
        _case("random", "repair", name="small_50", n=1000, m=8000, k=50, host=True),
        # a mid-size social graph fed small batches from host memory
        _case("rmat", "repair", name="rmat16_1k_pp", scale=16, m=16 << 16, mode="push-pull", kc=4, k=1000, host=True),
        # the topology-driven mode of the paper (no worklist), ordinary size
        _case("rmat", "repair", name="rmat18_10k_topo", scale=18, m=16 << 18, mode="topology", kc=4, k=10_000),
        # the benchmark's graph under a small batch: most of the work is finding out what did not change
        _case("rmat", "repair", name="rmat20_1k_dd", scale=20, m=16 << 20, kc=4, k=1000),
        # the benchmark's own step, in the plain and in the push-pull method
        _case("rmat", "repair", name="rmat20_100k_dd", scale=20, m=16 << 20, kc=4, k=100_000),
        _case("rmat", "repair", name="rmat20_100k_pp", scale=20, m=16 << 20, mode="push-pull", kc=4, k=100_000),
        # the static recompute that the dynamic repair is compared with
        _case("rmat", "recompute", name="rmat20_100k_static", scale=20, m=16 << 20, kc=4, k=100_000, batches=4),
        # assignment: unit capacities, +-1 changes given as deltas, the learned policy choosing per batch
        _case("bipartite", "repair", name="assign18_10k_learned", left=1 << 18, right=1 << 18, m=1 << 22,
              mode="push-pull", kc=4, policy="learned", k=10_000, delta=True),
        # interactive segmentation: a rectangle of an odd-sized image changes, the new mask is read
        _case("grid", "repair", name="grid1023_rect_dd_cut", w=1023, h=769, kc=4, k=2 * 96 * 96, cut=True),
        # the same on a large image, values only
        _case("grid", "repair", name="grid2048_rect_pp", w=2048, h=2048, mode="push-pull", kc=4, k=2 * 256 * 256),
        # one network solved once, from host arrays
        _case("random", "oneshot", name="oneshot_64k", n=65_537, m=1_000_003),
        # four resident graphs served together
        _case("mix", "serve", name="serve_mix", scale=16, w=512, h=512, left=1 << 14, right=1 << 14, k=20_000,
              mode="push-pull", kc=4, batches=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["random", "rmat", "rmat", "grid", "bipartite"])
    # (a static solve of an assignment graph is left to the others: its value is nearly always the smaller side)
    act = rng.choice(["repair", "repair", "repair", "recompute", "recompute" if kind == "bipartite" else "solve"])
    c = _case(kind, act, mode=rng.choice(["data-driven", "data-driven", "push-pull", "topology"]),
              kc=rng.choice([0, 2, 4, 4, 7]), host=rng.random() < 0.4, cut=rng.random() < 0.2)
    if kind == "random":
        c["n"] = _log_int(rng, 300, 300_000)
        c["m"] = int(c["n"] * rng.uniform(3.0, 12.0)) | 1
    elif kind == "rmat":
        c["scale"] = rng.randint(12, 20)
        c["m"] = int((1 << c["scale"]) * rng.uniform(6.0, 16.0)) | 1
    elif kind == "grid":
        c["w"], c["h"] = _log_int(rng, 96, 1400), _log_int(rng, 96, 1400)
        if c["mode"] == "topology":
            c["mode"] = "data-driven"
    else:
        c["left"], c["right"] = _log_int(rng, 1 << 10, 1 << 18), _log_int(rng, 1 << 10, 1 << 18)
        c["m"] = int(max(c["left"], c["right"]) * rng.uniform(4.0, 16.0)) | 1
        c["delta"] = rng.random() < 0.5
    if c["mode"] == "push-pull" and act == "repair" and rng.random() < 0.4:
        c["policy"] = "learned"
    if kind == "grid":
        side = _log_int(rng, 16, max(17, min(c["w"], c["h"], 300) // 2))
        c["k"] = 2 * side * side
    else:
        c["k"] = _log_int(rng, 40, max(41, min(100_000, _edges(c) // 16)))
    if act == "solve":
        c["k"], c["batches"], c["cut"], c["policy"], c["delta"] = 0, 1, True, "fixed", False
    elif act == "recompute":
        c["batches"], c["cut"] = 2, False
    return c


def _edges(c):
    if c["kind"] == "grid":
        return 2 * (c["w"] * (c["h"] - 1) + c["h"] * (c["w"] - 1)) + 2 * c["w"] * c["h"]
    return c["m"] + (c["left"] + c["right"] if c["kind"] == "bipartite" else 0)


def _vertices(c):
    return {"random": c["n"], "rmat": 1 << c["scale"], "grid": c["w"] * c["h"] + 2,
            "bipartite": c["left"] + c["right"] + 2}[c["kind"]]


def _parts(c):
    """The graphs of a case: one, or the four of the served mix."""
    if c["kind"] != "mix":
        return [c]
    return [dict(c, kind="rmat", m=16 << c["scale"]), dict(c, kind="rmat", scale=c["scale"] - 2, m=16 << (c["scale"] - 2)),
            dict(c, kind="grid"), dict(c, kind="bipartite", m=16 * c["left"])]


def work(case):
    """One pass: the resident structure of the residual graph (head and residual of every arc; row offset and excess
    read and height written for every vertex) is read once per answered batch, a batch entry with what it changes
    (id, capacity, its arc, both residuals and the capacities) moves 32 bytes, and each value or cut is written once.
    A solve also writes the residual, a build reads the edges and writes the arcs with their reverse and capacity."""
    total = 0
    for c in _parts(case):
        n, m = _vertices(c), _edges(c)
        arcs = 2 * m if c["kind"] != "grid" else m + 2 * c["w"] * c["h"]
        state = 8 * arcs + 16 * n
        per = state + 32 * c["k"] + 8 + (n if c["cut"] else 0)
        if c["act"] == "solve":
            total += state + 8 * arcs + n + 8
        elif c["act"] == "oneshot":
            total += 8 * m + 8 * n + 16 * arcs + state + 8 * arcs + n + 8
        elif c["act"] == "recompute":
            total += c["batches"] * (per + 8 * arcs)
        else:
            total += c["batches"] // (4 if case["act"] == "serve" else 1) * per
    return {"bytes": total, "flops": 0}


# ------------------------------------------------------------ flow networks --
def _csr(n, tails, heads, caps):
    """CSR arrays (CUDA) of an edge list, edges ordered by tail."""
    order = torch.argsort(tails, stable=True)
    row = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row[1:] = torch.bincount(tails, minlength=n).cumsum(0)
    return row, heads[order].to(torch.int32), caps[order].to(torch.int32)


def _ints(g, count, lo, hi):
    return torch.randint(lo, hi + 1, (count,), generator=g, device="cuda")


def _random(c, g):
    """Uniform directed graph with a guaranteed path 0 -> 1 -> 2 -> n-1, capacities U[1, 100]."""
    n, m = c["n"], c["m"]
    u = _ints(g, m - 3, 0, n - 1)
    v = (u + 1 + _ints(g, m - 3, 0, n - 2)) % n
    fix = torch.tensor([[0, 1, 2], [1, 2, n - 1]], device="cuda")
    return (n, *_csr(n, torch.cat([fix[0], u]), torch.cat([fix[1], v]), _ints(g, m, 1, 100)), 0, n - 1)


def _rmat(c, g):
    """Power-law graph by the RMAT recursion (.57, .19, .19, .05), vertex ids permuted, self-loops dropped,
    capacities U[1, 1000]; s and t are the vertices of highest out-degree."""
    n = 1 << c["scale"]
    u = torch.zeros(c["m"], dtype=torch.int64, device="cuda")
    v = torch.zeros_like(u)
    for _ in range(c["scale"]):
        x = torch.rand(c["m"], generator=g, device="cuda")
        bu = x >= 0.76
        bv = ((x >= 0.57) & ~bu) | (x >= 0.95)
        u = 2 * u + bu
        v = 2 * v + bv
    perm = torch.randperm(n, generator=g, device="cuda")
    u, v = perm[u], perm[v]
    keep = u != v
    u, v = u[keep], v[keep]
    top = torch.argsort(torch.bincount(u, minlength=n), descending=True, stable=True)[:2].tolist()
    return (n, *_csr(n, u, v, _ints(g, u.numel(), 1, 1000)), top[0], top[1])


def _bipartite(c, g):
    """Assignment: s -> left -> right -> t, unit capacities."""
    nl, nr, m = c["left"], c["right"], c["m"]
    s, t = nl + nr, nl + nr + 1
    lo, hi = torch.arange(nl, device="cuda"), nl + torch.arange(nr, device="cuda")
    tails = torch.cat([torch.full((nl,), s, device="cuda"), _ints(g, m, 0, nl - 1), hi])
    heads = torch.cat([lo, nl + _ints(g, m, 0, nr - 1), torch.full((nr,), t, device="cuda")])
    return (t + 1, *_csr(t + 1, tails, heads, torch.ones_like(tails)), s, t)


def _blobs(w, h, g, count):
    y, x = torch.arange(h, device="cuda", dtype=torch.float64)[:, None], torch.arange(w, device="cuda", dtype=torch.float64)
    p = torch.rand((count, 4), generator=g, device="cuda", dtype=torch.float64).tolist()
    img = torch.full((h, w), 40.0, dtype=torch.float64, device="cuda")
    for a, b, c, d in p:
        rad = (1 / 32 + c * (1 / 6 - 1 / 32)) * min(w, h)
        img += (60 + 100 * d) * torch.exp(-((x - a * w) ** 2 + (y - b * h) ** 2) / (2 * rad * rad))
    return img


def _terminals(img):
    """Capacities to the source and from the sink: Gaussian negative log-likelihoods of the background (50, 30) and
    foreground (175, 30) models, scaled to [0, 1000]."""
    nll_b, nll_f = ((0.5 * ((img - mu) / 30.0) ** 2 + math.log(30.0)) for mu in (50.0, 175.0))
    top = 0.5 * ((255.0 - 50.0) / 30.0) ** 2 + math.log(30.0)
    return (torch.round(1000 * nll_b / top).clamp(0, 1000).long(), torch.round(1000 * nll_f / top).clamp(0, 1000).long())


def _grid(c, g):
    """Image segmentation: 4-connected pixels with contrast capacities round(100 exp(-dI^2 / 200)) and terminal arcs."""
    w, h = c["w"], c["h"]
    img = (_blobs(w, h, g, 24) + 10 * torch.rand((h, w), generator=g, device="cuda", dtype=torch.float64) - 5).clamp(0, 255)
    pix = torch.arange(w * h, device="cuda").view(h, w)
    s, t = w * h, w * h + 1
    tails, heads, caps = [], [], []
    for a, b, da in ((pix[:, :-1], pix[:, 1:], img[:, :-1] - img[:, 1:]), (pix[:-1], pix[1:], img[:-1] - img[1:])):
        cc = torch.round(100 * torch.exp(-da * da / 200)).long().reshape(-1)
        tails += [a.reshape(-1), b.reshape(-1)]
        heads += [b.reshape(-1), a.reshape(-1)]
        caps += [cc, cc]
    cs, ct = _terminals(img)
    p = pix.reshape(-1)
    tails += [p, torch.full_like(p, s)]
    heads += [torch.full_like(p, t), p]
    caps += [ct.reshape(-1), cs.reshape(-1)]
    row, col, cap = _csr(t + 1, torch.cat(tails), torch.cat(heads), torch.cat(caps))
    return (t + 1, row, col, cap, s, t), img


# ------------------------------------------------------------------ batches --
_STREAM = 64   # batches before a stream turns back


def _mixed(c, g, cap):
    """Disjoint random edge sets, half of each raised, half cut by U[1, 500] (unit graphs by 1), then put back."""
    k, m = c["k"], cap.numel()
    half = min(_STREAM, m // (2 * k))
    step = 1 if c["kind"] == "bipartite" else 500
    ids = torch.randperm(m, generator=g, device="cuda")[: half * k].view(half, k)
    old = cap[ids].long()
    amount = _ints(g, half * k, 1, step).view(half, k)
    amount[:, (k + 1) // 2:] *= -1
    new = (old + amount).clamp_min(0)
    there, back = (new - old, old - new) if c["delta"] else (new, old)
    return [(ids[j], there[j]) for j in range(half)] + [(ids[j], back[j]) for j in reversed(range(half))]


def _rects(c, g, row, cap, img):
    """Squares of the image re-drawn (a new blob each), the terminal capacities of their pixels rewritten, then put
    back in reverse order (squares may overlap)."""
    w, h = c["w"], c["h"]
    sw, sh = min(math.isqrt(c["k"] // 2), w), min(math.isqrt(c["k"] // 2), h)
    img, cap = img.clone(), cap.clone()
    there, back = [], []
    y = torch.arange(sh, device="cuda", dtype=torch.float64)[:, None] - sh / 2
    x = torch.arange(sw, device="cuda", dtype=torch.float64) - sw / 2
    for r in torch.rand((_STREAM // 2, 4), generator=g, device="cuda", dtype=torch.float64).tolist():
        x0, y0 = int(r[0] * (w - sw + 1)), int(r[1] * (h - sh + 1))
        rad = max(sw, sh) / 3
        blob = (40 + 80 * r[2]) * (1 if r[3] < 0.5 else -1) * torch.exp(-(x * x + y * y) / (2 * rad * rad))
        sub = img[y0:y0 + sh, x0:x0 + sw]
        sub.copy_((sub + blob).clamp(0, 255))
        p = (torch.arange(y0, y0 + sh, device="cuda")[:, None] * w + torch.arange(x0, x0 + sw, device="cuda")).reshape(-1)
        ids = torch.cat([row[w * h] + p, row[p + 1] - 1])   # s -> p, and p -> t (the last edge of a pixel)
        back.append((ids, cap[ids].long()))
        there.append((ids, torch.cat([v.reshape(-1) for v in _terminals(sub)])))
        cap[ids] = there[-1][1].to(torch.int32)
    return there + back[::-1]


def _graph_and_batches(c, g):
    img = None
    if c["kind"] == "grid":
        net, img = _grid(c, g)
    else:
        net = {"random": _random, "rmat": _rmat, "bipartite": _bipartite}[c["kind"]](c, g)
    batches = []
    if c["k"]:
        made = _rects(c, g, net[1], net[3], img) if c["kind"] == "grid" else _mixed(c, g, net[3])
        for ids, caps in made:
            b = (ids.to(torch.int32).contiguous(), caps.to(torch.int32).contiguous())
            batches.append(tuple(x.cpu().numpy() for x in b) if c["host"] or c["kind"] == "mix" or c["act"] == "serve" else b)
    return net, batches


def _resident(c, net):
    G = mf.MaxFlowGraph(*net, kernel_cycles=c["kc"], mode=MODES[c["mode"]])
    if c["policy"] == "learned":
        from paper_2511_05895_gb300 import policy
        G.set_policy(mf.MF_POLICY_LEARNED, policy.load_default_params())
    G.solve()
    G.flow_value()
    return G


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * seed + 17)
    if case["act"] == "serve":
        server, plan = mf.Server(), []
        for c in _parts(case):
            net, batches = _graph_and_batches(dict(c, k=min(c["k"], _edges(c) // 64) if c["kind"] != "grid"
                                                   else 2 * 64 * 64), g)
            at = server.add_graph(_resident(c, net), case["k"])
            plan.append([(at, *b) for b in batches])
        return dict(case=case, server=server, plan=plan, turn=0)
    net, batches = _graph_and_batches(case, g)
    if case["act"] == "oneshot":
        return dict(case=case, net=tuple(x.cpu().numpy() if isinstance(x, torch.Tensor) else x for x in net))
    return dict(case=case, graph=_resident(case, net), batches=batches, turn=0)


def _next(state, batches, count):
    """The next `count` batches of a stream."""
    at = state["turn"] * count
    return [batches[(at + j) % len(batches)] for j in range(count)]


def run(state):
    c = state["case"]
    if c["act"] == "serve":
        S = state["server"]
        parts = [_next(state, p, c["batches"] // len(state["plan"])) for p in state["plan"]]
        state["turn"] += 1
        tickets = [S.submit(*r) for turn in zip(*parts) for r in turn]
        S.drain()
        return [S.poll(t)[1] for t in tickets]
    if c["act"] == "oneshot":
        with mf.MaxFlowGraph(*state["net"], kernel_cycles=c["kc"], mode=MODES[c["mode"]]) as G:
            G.solve()
            return [G.flow_value(), G.min_cut()]
    G = state["graph"]
    if c["act"] == "solve":
        G.solve()
        return [G.flow_value(), G.min_cut()]
    values, cuts = [], []
    todo = _next(state, state["batches"], c["batches"])
    state["turn"] += 1
    for ids, caps in todo:
        G.apply_updates(ids, caps, delta=c["delta"], recompute=c["act"] == "recompute")
        values.append(G.flow_value())
        if c["cut"]:
            cuts.append(G.min_cut())
    return [np.array(values, np.int64), *cuts]


def _max_flow(n, tails, heads, caps, s, t):
    """Value and minimal-sink-side minimum cut (1 = source side) by Dinic's method, in Python's whole numbers."""
    adj = [[] for _ in range(n)]
    to, left = [], []
    for u, v, cap in zip(tails, heads, caps):
        if u != v:
            adj[u].append(len(to))
            adj[v].append(len(to) + 1)
            to += [v, u]
            left += [cap, 0]
    value = 0
    while True:
        # distances to t; the vertices that cannot reach it are the source side
        dist = [-1] * n
        dist[t] = 0
        todo = [t]
        for v in todo:
            for a in adj[v]:
                if left[a ^ 1] and dist[to[a]] < 0:
                    dist[to[a]] = dist[v] + 1
                    todo.append(to[a])
        if dist[s] < 0:
            return value, np.array([d < 0 for d in dist], np.uint8)
        at, path, u = [0] * n, [], s
        while True:
            if u == t:
                d = min(left[a] for a in path)
                for a in path:
                    left[a] -= d
                    left[a ^ 1] += d
                value, path, u = value + d, [], s
            while at[u] < len(adj[u]) and not (left[adj[u][at[u]]] and dist[to[adj[u][at[u]]]] == dist[u] - 1):
                at[u] += 1
            if at[u] < len(adj[u]):
                path.append(adj[u][at[u]])
                u = to[path[-1]]
            elif u == s:
                break
            else:
                dist[u] = -1
                u = to[path.pop() ^ 1]


def exact(case, seed):
    if case["act"] not in ("repair", "recompute") or _edges(case) > 20_000:
        return None
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * seed + 17)
    (n, row, col, cap, s, t), batches = _graph_and_batches(case, g)
    tails = torch.repeat_interleave(torch.arange(n, device="cuda"), row.diff()).tolist()
    heads, caps = col.tolist(), cap.tolist()
    values, cuts = [], []
    for ids, new in batches[: case["batches"]]:
        for e, x in zip(ids.tolist(), new.tolist()):
            caps[e] = max(0, caps[e] + x) if case["delta"] else x
        value, cut = _max_flow(n, tails, heads, caps, s, t)
        values.append(value)
        cuts += [cut] if case["cut"] else []
    return [np.array(values, np.int64), *cuts]
