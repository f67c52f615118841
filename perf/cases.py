"""The calls whose speed counts: one pass of each of the package's main entry points, over the sizes
that its users bring -- from a few thousand edges, where latency and launches are the time, to the
1.07 G-edge dense graph of the benchmark, which streams 8.6 GB.

Graphs are synthetic and made from the seed alone, on the GPU: dense clusters joined by a tree of
single edges, some further edges between clusters, and pendant paths (bridges hang off dense
cores, the shape of the small, mid and large benchmark workloads); sparse random multigraphs
(many components, thousands of bridges); R-MAT graphs (skewed degrees, too many vertices for
16-bit labels); batches and request streams of small graphs.  Lists come shuffled, or sorted by
their ends as graph files usually hold them.  Every output is whole numbers and unique, so
everything is compared exactly.
"""
import math

import numpy as np
import torch

import paper_2108_07346_gb300 as pb

DEV = "cuda"


def listed():
    return [
        # a topology check on a handful of nodes: launches and latency only
        _find("tiny", clusters=2, core=224, pendant=32, extra=2, edges=2_000),
        # the small benchmark workload's shape: 8 clusters of 256, density 1/2
        _find("small", clusters=8, core=2048, pendant=40, extra=20, edges=130_507),
        # a sparse network: average degree 3, thousands of bridges to sort
        dict(name="sparse", kind="find", shape="sparse", core=20_000, edges=30_001, order="shuffled", skip=0),
        # the mid benchmark workload's shape: 64 clusters of 512, density 0.3, pendant paths
        _find("mid", clusters=64, core=32_768, pendant=4_379, extra=500, edges=2_509_163),
        # the same graph as a file holds it, sorted by its ends
        _find("mid sorted", clusters=64, core=32_768, pendant=4_379, extra=500, edges=2_509_163, order="sorted"),
        # the large benchmark workload's shape: one dense core of 65,536 vertices, density 1/2
        _find("large", clusters=1, core=65_536, pendant=8_183, extra=128, edges=1_073_698_874),
        # a web-like graph: skewed degrees, a million vertices
        dict(name="rmat", kind="find", shape="rmat", scale=20, edges=16_777_216, order="shuffled", skip=0),
        # a list in pinned host memory: copy and compute
        _find("host", clusters=1, core=12_288, pendant=1_024, extra=16, edges=40_000_003, kind="host"),
        # cut vertices
        _find("articulation", clusters=64, core=32_768, pendant=4_379, extra=500, edges=2_509_163, kind="articulation"),
        # many graphs in one call: V log-uniform in 64..4,096, density 0.1..0.9
        dict(name="batched", kind="batched", graphs=1024, vmin=64, vmax=4096),
        # a resident graph, new links added, bridges and 2-edge-connected components asked for
        _find("incremental", clusters=64, core=32_768, pendant=4_379, extra=500, edges=2_509_163, kind="incremental",
              added=1_000),
        # a burst of queries to the server: V log-uniform in 256..65,536, density 0.05..0.6
        dict(name="served", kind="served", requests=24, vmin=256, vmax=65_536),
    ]


def _find(name, clusters, core, pendant, extra, edges, order="shuffled", skip=0, kind="find", **more):
    c = dict(kind=kind, shape="clusters", clusters=clusters, core=core, pendant=pendant, extra=extra, edges=edges,
             order=order, skip=skip, **more)
    return dict(c, name=name) if name else c


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["find"] * 6 + ["articulation"] * 2 + ["host", "batched", "incremental", "served"])
    if kind == "batched":
        vmin = _log(rng, 32, 512)
        return dict(kind=kind, graphs=_log(rng, 17, 2048), vmin=vmin, vmax=_log(rng, vmin * 2, 4096))
    if kind == "served":
        vmin = _log(rng, 64, 4096)
        return dict(kind=kind, requests=rng.randint(2, 48), vmin=vmin, vmax=_log(rng, vmin * 2, 65_536))
    order = rng.choice(["shuffled", "shuffled", "sorted"])
    skip = rng.choice([0, 0, 0, 1])  # a slice of a longer list: its start is not 16-byte aligned
    shape = rng.choice(["clusters"] * 4 + ["sparse", "rmat"]) if kind == "find" else "clusters"
    if shape == "sparse":
        v = _log(rng, 100, 100_000)
        return dict(kind=kind, shape=shape, core=v, edges=int(v * rng.uniform(0.6, 3.0)), order=order, skip=skip)
    if shape == "rmat":
        scale = rng.randint(14, 21)
        return dict(kind=kind, shape=shape, scale=scale, edges=int((1 << scale) * rng.uniform(4, 24)), order=order,
                    skip=skip)
    core = _log(rng, 96, 65_536)
    clusters = rng.choice([1, 1, 2, max(1, core // 512), max(1, core // 128)])
    size = core // clusters
    core = size * clusters
    most = min(300e6, 0.3 * core * size) if kind != "host" else min(60e6, 0.3 * core * size)
    edges = _log(rng, 4 * core, max(5 * core, most))
    return _find(None, clusters, core, rng.randint(1, max(1, core // 8)), rng.randint(1, max(1, core // 64)), edges,
                 order, skip, kind, **(dict(added=_log(rng, 1, 10_000)) if kind == "incremental" else {}))


# ---- inputs ----------------------------------------------------------------------------------

def _vertices(c):
    if c["shape"] == "rmat":
        return 1 << c["scale"]
    return c["core"] + c.get("pendant", 0)


def _structure(c, g):
    """The edges between clusters and the pendant paths: (u, v) int32 arrays of vertex numbers before
    relabelling (clusters first, pendant vertices last)."""
    k, core, pend = c["clusters"], c["core"], c["pendant"]
    size = core // k
    inside = lambda cl: cl * size + g.integers(0, size, cl.shape[0])  # noqa: E731
    child = np.arange(1, k)
    up = (g.random(k - 1) * child).astype(np.int64)  # a random earlier cluster
    us, vs = [inside(child)], [inside(up)]
    if c["extra"] > 0:
        us.append(g.integers(0, core, c["extra"]))
        vs.append(g.integers(0, core, c["extra"]))
    if pend > 0:
        x = core + np.arange(pend)
        start = g.random(pend) < 1 / 4.5  # paths of 4.5 vertices on average
        start[0] = True
        us.append(x)
        vs.append(np.where(start, g.integers(0, core, pend), x - 1))
    return np.concatenate(us).astype(np.int32), np.concatenate(vs).astype(np.int32)


def _pairs(n_clusters, size, u, v, gen):
    """Fills u, v with random pairs of different vertices of one random cluster each."""
    for i in range(0, u.numel(), 1 << 26):
        n = min(1 << 26, u.numel() - i)
        a = torch.randint(0, size, (n,), generator=gen, dtype=torch.int32, device=DEV)
        b = torch.randint(1, size, (n,), generator=gen, dtype=torch.int32, device=DEV).add_(a).remainder_(size)
        if n_clusters > 1:
            cl = torch.randint(0, n_clusters, (n,), generator=gen, dtype=torch.int32, device=DEV).mul_(size)
            a.add_(cl)
            b.add_(cl)
        u[i:i + n] = a
        v[i:i + n] = b


def _rmat(scale, u, v, gen):
    for i in range(0, u.numel(), 1 << 25):
        n = min(1 << 25, u.numel() - i)
        a = torch.zeros(n, dtype=torch.int32, device=DEV)
        b = torch.zeros(n, dtype=torch.int32, device=DEV)
        for _ in range(scale):  # quadrants 0.57 / 0.19 / 0.19 / 0.05
            r = torch.rand(n, generator=gen, device=DEV)
            a.mul_(2).add_((r >= 0.76).to(torch.int32))
            b.mul_(2).add_((((r >= 0.57) & (r < 0.76)) | (r >= 0.95)).to(torch.int32))
        u[i:i + n] = a
        v[i:i + n] = b


def _graph(c, seed):
    """(u, v, V): the case's edge list on the GPU."""
    gen = torch.Generator(device=DEV).manual_seed(seed * 1_000_003 + 17)
    g = np.random.default_rng(seed * 7919 + 5)
    V, E = _vertices(c), c["edges"]
    u = torch.empty(E, dtype=torch.int32, device=DEV)
    v = torch.empty(E, dtype=torch.int32, device=DEV)
    if c["shape"] == "sparse":
        u.copy_(torch.randint(0, V, (E,), generator=gen, dtype=torch.int32, device=DEV))
        v.copy_(torch.randint(0, V, (E,), generator=gen, dtype=torch.int32, device=DEV))
    elif c["shape"] == "rmat":
        _rmat(c["scale"], u, v, gen)
    else:
        su, sv = _structure(c, g)
        n = su.shape[0]
        _pairs(c["clusters"], c["core"] // c["clusters"], u, v, gen)
        at = torch.from_numpy(np.unique(g.integers(0, E, 2 * n + 64))).to(DEV)  # the structure's places in the list
        at = at[torch.randperm(at.numel(), generator=gen, device=DEV)][:n]
        if at.numel() < n:
            at = torch.arange(n, device=DEV)
        u[at] = torch.from_numpy(su).to(DEV)
        v[at] = torch.from_numpy(sv).to(DEV)
    if c["shape"] != "sparse":  # vertex numbers say nothing about the structure
        name = torch.randperm(V, generator=gen, device=DEV).to(torch.int32)
        for i in range(0, E, 1 << 26):
            u[i:i + (1 << 26)] = name[u[i:i + (1 << 26)].long()]
            v[i:i + (1 << 26)] = name[v[i:i + (1 << 26)].long()]
    if c["order"] == "sorted":
        lo, hi = torch.minimum(u, v).long(), torch.maximum(u, v).long()
        key = (lo * V + hi).sort().values
        u, v = (key // V).to(torch.int32), (key % V).to(torch.int32)
    return u, v, V


def _skipped(u, v, skip):
    if not skip:
        return u, v
    z = torch.zeros(skip, dtype=torch.int32, device=u.device)
    return torch.cat([z, u])[skip:], torch.cat([z, v])[skip:]


def _small_specs(c, n, dmin, dmax, span):
    """Sizes of n small graphs: vertices log-uniform in [vmin, vmax], density uniform inside clusters
    (of the case alone; what the graphs hold comes from the seed)."""
    g = np.random.default_rng(11)
    V = np.exp(g.uniform(np.log(c["vmin"]), np.log(c["vmax"]), n)).astype(np.int64)
    d = g.uniform(dmin, dmax, n)
    specs = []
    for i in range(n):
        v = int(V[i])
        k = max(1, v // span) if span else int(g.integers(1, 5))
        pend = int(g.integers(1, max(2, min(32, v // 4))))
        size = max(2, (v - pend) // k)
        specs.append(dict(clusters=k, core=size * k, pendant=pend, extra=max(1, v // 64),
                          edges=int(d[i] * k * size * (size - 1) / 2) + 4 * k + 2 * pend + v // 32 + 4))
    return specs


def _many(specs, seed):
    """The edge lists of many clustered graphs in one pair of arrays, and where each begins."""
    gen = torch.Generator(device=DEV).manual_seed(seed * 1_000_003 + 29)
    g = np.random.default_rng(seed * 7919 + 31)
    off = np.concatenate([[0], np.cumsum([s["edges"] for s in specs])]).astype(np.int64)
    n = int(off[-1])
    u = torch.empty(n, dtype=torch.int32, device=DEV)
    v = torch.empty(n, dtype=torch.int32, device=DEV)
    count = torch.tensor([s["edges"] for s in specs], device=DEV)
    size = torch.repeat_interleave(torch.tensor([s["core"] // s["clusters"] for s in specs], device=DEV), count)
    k = torch.repeat_interleave(torch.tensor([s["clusters"] for s in specs], device=DEV), count)
    a = (torch.rand(n, generator=gen, device=DEV) * size).long().clamp_(max=size - 1)
    b = (torch.rand(n, generator=gen, device=DEV) * (size - 1)).long().clamp_(max=size - 2).add_(a + 1).remainder_(size)
    base = (torch.rand(n, generator=gen, device=DEV) * k).long().clamp_(max=k - 1).mul_(size)
    u.copy_(a.add_(base))
    v.copy_(b.add_(base))
    del a, b, base, size, k
    su, sv, at = [], [], []
    for i, s in enumerate(specs):  # the structure's places: distinct, spread over the graph's own list
        x, y = _structure(s, g)
        su.append(x)
        sv.append(y)
        at.append(off[i] + (np.arange(x.shape[0]) * s["edges"]) // x.shape[0])
    at = torch.from_numpy(np.concatenate(at)).to(DEV)
    u[at] = torch.from_numpy(np.concatenate(su)).to(DEV)
    v[at] = torch.from_numpy(np.concatenate(sv)).to(DEV)
    return u, v, off


def _pairs_buffer(V, **how):
    """Room for the bridges of a graph of V vertices, kept by the caller; its unused end stays zero."""
    return torch.zeros(2 * max(V - 1, 1), dtype=torch.int32, **how)


def prepare(case, seed):
    c = case
    if c["kind"] == "batched":
        specs = _small_specs(c, c["graphs"], 0.1, 0.9, 0)
        u, v, off = _many(specs, seed)
        Vs = np.array([s["core"] + s["pendant"] for s in specs], np.int32)
        out = torch.zeros(int((2 * np.maximum(Vs.astype(np.int64) - 1, 0)).sum()), dtype=torch.int32, device=DEV)
        counts = torch.zeros(len(specs), dtype=torch.int64, device=DEV)
        return dict(case=c, ctx=pb.Context(), u=u, v=v, off=off, Vs=Vs, out=out, counts=counts)
    if c["kind"] == "served":
        specs = _small_specs(c, c["requests"], 0.05, 0.6, 512)
        u, v, off = _many(specs, seed)
        graphs = []
        for i, s in enumerate(specs):
            V = s["core"] + s["pendant"]
            graphs.append((u[off[i]:off[i + 1]].clone(), v[off[i]:off[i + 1]].clone(), V, _pairs_buffer(V, device=DEV)))
        return dict(case=c, server=pb.Server(), graphs=graphs)
    u, v, V = _graph(c, seed)
    if c["kind"] == "host":
        hu, hv = (torch.empty(t.numel() + c["skip"], dtype=torch.int32, pin_memory=True)[c["skip"]:] for t in (u, v))
        hu.copy_(u)
        hv.copy_(v)
        return dict(case=c, ctx=pb.Context(), u=hu, v=hv, V=V, out=_pairs_buffer(V, pin_memory=True))
    u, v = _skipped(u, v, c["skip"])
    if c["kind"] == "incremental":
        inc = pb.Incremental()
        inc.reset(u, v, V)
        gen = torch.Generator(device=DEV).manual_seed(seed * 31 + 7)
        a = torch.randint(0, V, (c["added"],), generator=gen, dtype=torch.int32, device=DEV)
        b = torch.randint(0, V, (c["added"],), generator=gen, dtype=torch.int32, device=DEV)
        # every new link is a pair of lines, so adding the same ones again changes nothing
        return dict(case=c, inc=inc, a=torch.cat([a, a]), b=torch.cat([b, b]), out=_pairs_buffer(V, device=DEV))
    if c["kind"] == "articulation":
        return dict(case=c, ctx=pb.Context(), u=u, v=v, V=V, out=torch.zeros(V, dtype=torch.int32, device=DEV))
    return dict(case=c, ctx=pb.Context(), u=u, v=v, V=V, out=_pairs_buffer(V, device=DEV))


def run(state):
    """One call.  The results are in the caller's buffers, whole, and their number is returned."""
    s, kind = state, state["case"]["kind"]
    if kind == "find":
        n = s["ctx"].find(s["u"], s["v"], s["V"], out=s["out"]).shape[0]
        return {"bridges": s["out"], "count": n}
    if kind == "host":
        n = s["ctx"].find_host(s["u"], s["v"], s["V"], out=s["out"]).shape[0]
        return {"bridges": s["out"], "count": n}
    if kind == "articulation":
        n = s["ctx"].articulation_points(s["u"], s["v"], s["V"], out=s["out"]).shape[0]
        return {"points": s["out"], "count": n}
    if kind == "batched":
        s["ctx"].find_batched(s["u"], s["v"], s["off"], s["Vs"], out=s["out"], counts=s["counts"])
        return {"bridges": s["out"], "counts": s["counts"]}
    if kind == "incremental":
        bridges = s["inc"].add(s["a"], s["b"])
        s["out"][: bridges.numel()] = bridges.view(-1)
        n, labels = s["inc"].two_edge_components()
        return {"bridges": s["out"], "count": bridges.shape[0], "components": n, "labels": labels}
    tickets = [s["server"].submit(u, v, V, out=out) for u, v, V, out in s["graphs"]]
    counts = [s["server"].wait(t)[0].shape[0] for t in tickets]
    return {"bridges": [g[3] for g in s["graphs"]], "counts": np.array(counts)}


def work(case):
    """Each edge read once (8 bytes); each bridge that the construction plants written once (8 bytes).
    A comparison per edge and forest at the least: 2 operations."""
    c = case
    if c["kind"] in ("batched", "served"):
        # expected sizes: V log-uniform, half the density of all pairs (inside clusters of 512 when served)
        n = c["graphs"] if c["kind"] == "batched" else c["requests"]
        lo, hi = c["vmin"], c["vmax"]
        span = math.log(hi / lo)
        if c["kind"] == "batched":
            edges = n * 0.5 * 0.5 * 0.5 * (hi * hi - lo * lo) / (2 * span)
        else:
            edges = n * 0.325 * 0.5 * 512 * (hi - lo) / span
        return {"bytes": 8 * edges + 16 * 8 * n, "flops": 2 * edges}
    V = _vertices(c)
    if c["kind"] == "incremental":  # the resident certificate (at most 2V edges), the new links, the labels
        return {"bytes": 16 * V + 16 * c["added"] + 4 * V, "flops": 4 * V + 4 * c["added"]}
    return {"bytes": 8 * c["edges"] + 8 * c.get("pendant", 0), "flops": 2 * c["edges"]}


def tolerance(case):
    return "exact"


def exact(case, seed):
    """The bridges by one depth-first search on the host, for lists short enough for it."""
    if case["kind"] != "find" or case["edges"] > 200_000:
        return None
    u, v, V = _graph(case, seed)
    u, v = u.cpu().numpy(), v.cpu().numpy()
    E = u.shape[0]
    ends = np.concatenate([u, v])
    order = np.argsort(ends, kind="stable")
    first = np.concatenate([[0], np.cumsum(np.bincount(ends, minlength=V))]).tolist()
    other = np.concatenate([v, u])[order].tolist()
    edge = np.concatenate([np.arange(E), np.arange(E)])[order].tolist()
    disc, low, found, clock = [-1] * V, [0] * V, [], 0
    at = first[:-1]
    for root in range(V):
        if disc[root] >= 0:
            continue
        disc[root] = low[root] = clock
        clock += 1
        path = [(root, -1)]
        while path:
            x, by = path[-1]
            if at[x] < first[x + 1]:
                y, e = other[at[x]], edge[at[x]]
                at[x] += 1
                if e == by or y == x:
                    continue
                if disc[y] < 0:
                    disc[y] = low[y] = clock
                    clock += 1
                    path.append((y, e))
                else:
                    low[x] = min(low[x], disc[y])
            else:
                path.pop()
                if path:
                    p = path[-1][0]
                    low[p] = min(low[p], low[x])
                    if low[x] > disc[p]:
                        found.append((min(p, x), max(p, x)))
    found.sort()
    out = _pairs_buffer(V)
    out[: 2 * len(found)] = torch.tensor(found, dtype=torch.int32).view(-1)
    return {"bridges": out, "count": len(found)}
