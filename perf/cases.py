"""Performance cases of the connected-components library: what its users run,
through the public Python entry points (``Graph``, ``Batch``, ``Server`` and
the ``cc_*`` calls), from a few thousand edges to 2^32.

A case is a dict of plain values:
  api    coo     Graph.run on a device-resident edge list
         csr     cc_run_csr on device-resident offsets and neighbours
         host    cc_run_host on pinned host edges, labels back to the host
         packed  cc_run_host_packed: the same with 3-byte ids
         stream  a resident graph, then insert batches, query batches, labels
         batch   many small graphs in one Batch.run
         serve   one graph's life in a Server: admission with labels, insert
                 batches, query batches, a snapshot, the drop
  graph  rmat    skewed degrees, one giant component; scrambled vertex ids
         uniform independent uniform pairs: no hub
         grid    2D lattice, each edge kept with probability 0.9, row-major
  n, edges       vertices and edges (grid: width x height; about 1.8 edges a vertex)
  order          "random" as generated, or "source": sorted by first endpoint
  shift          the edge buffer starts 8 bytes past a 16-byte boundary
  mode, label_space, root_select: the library's options of those names

Inputs are made on the GPU from the seed alone. ``exact`` gives the labels that
the definition demands (each component named by its smallest vertex).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2507_03695_gb300 as cc

DEV = "cuda"
CHUNK = 1 << 27
# R-MAT quadrants 0.57 / 0.19 / 0.19 / 0.05, as thresholds on 31 random bits
T_A, T_AB, T_ABC = (int(p * (1 << 31)) for p in (0.57, 0.76, 0.95))


def listed():
    return [
        # the smallest call a program makes: launches and their gaps decide it
        coo("coo_rmat12_small", "rmat", 1 << 12, 3 * (1 << 12) + 1),
        # one small graph under Algorithm 1 (f = id): R-MAT 16, edge factor 16
        coo("coo_rmat16_identity", "rmat", 1 << 16, 1 << 20, mode=cc.CC_ROOT_IDENTITY),
        # an ordinary graph with odd sizes, read from a slice of a larger
        # buffer: the vertex count is no power of two, the edges are not
        # 16-byte aligned, the count is odd
        coo("coo_rmat20_ragged", "rmat", 1_000_003, 15_999_999, shift=True),
        # a large skewed graph whose parent array fits the L2 cache
        coo("coo_rmat24", "rmat", 1 << 24, 1 << 28),
        # a large graph without a hub: equal degrees, no locality
        coo("coo_uniform24", "uniform", 1 << 24, 1 << 26),
        # road-like: high diameter, many components, edges in row order
        dict(name="coo_grid8192", api="coo", graph="grid", width=8192, height=8192, **OPTIONS),
        # the largest: 2^32 edges resident in HBM, parent array beyond L2
        coo("coo_rmat28", "rmat", 1 << 28, 1 << 32),
        # the compressed-row layout that graph files are kept in
        dict(coo("csr_rmat24", "rmat", 1 << 24, 1 << 28), api="csr"),
        # edges in host memory, labels wanted there: the copies count
        dict(coo("host_rmat22", "rmat", 1 << 22, 1 << 26), api="host"),
        # incremental use: a resident graph, ten insert batches of 10^3 to
        # 10^6 uniform pairs, a batch of 10^4 queries after each, then labels
        dict(coo("stream_rmat20", "rmat", 1 << 20, 1 << 22), api="stream", batches=10, largest=1_000_000, queries=10_000),
        # thousands of independent small graphs, 2^8 to 2^18 vertices, mixed
        # uniform / R-MAT / grid
        dict(name="batch_4096_mixed", api="batch", graphs=4096),
        # the serving runtime: a graph admitted, grown, queried, dropped
        dict(coo("serve_rmat20", "rmat", 1 << 20, 1 << 24), api="serve", batches=16, largest=100_000, queries=10_000),
    ]


OPTIONS = dict(mode=cc.CC_ROOT_MAXDEG, label_space=cc.CC_LABEL_MIN_ID, root_select=cc.CC_ROOT_SELECT_EXACT,
               order="random", shift=False)


def coo(name, graph, n, edges, **options):
    return dict(name=name, api="coo", graph=graph, n=n, edges=edges, **{**OPTIONS, **options})


def draw(rng):
    api = rng.choice(["coo"] * 5 + ["csr"] * 2 + ["host", "packed", "stream", "batch", "serve"])
    if api == "batch":
        return dict(api=api, graphs=int(2 ** rng.uniform(0, 12)))
    options = dict(mode=rng.choice([cc.CC_ROOT_MAXDEG] * 3 + [cc.CC_ROOT_IDENTITY]),
                   label_space=rng.choice([cc.CC_LABEL_MIN_ID] * 3 + [cc.CC_LABEL_ROOT_VALUE]),
                   root_select=rng.choice([cc.CC_ROOT_SELECT_EXACT] * 4 + [cc.CC_ROOT_SELECT_SAMPLED]),
                   order=rng.choice(["random", "random", "source"]), shift=rng.random() < 0.25)
    graph = rng.choice(["rmat", "rmat", "rmat", "uniform", "grid"])
    if graph == "grid":
        return dict(api="coo" if api in ("packed", "stream", "serve") else api, graph=graph,
                    width=int(2 ** rng.uniform(8, 13)), height=int(2 ** rng.uniform(8, 13)), **options)
    large = {"coo": 26, "csr": 25, "host": 24, "packed": 24, "stream": 24, "serve": 22}[api]
    n = int(2 ** rng.uniform(12 if api in ("stream", "serve") else 8, large))
    if rng.random() < 0.3:
        n = 1 << (n.bit_length() - 1)
    # uniform graphs stay below the density that joins every vertex
    factor = 2 ** (rng.uniform(0, 5) if graph == "rmat" else rng.uniform(-1, 2 if n >= 1 << 18 else 1))
    case = dict(api=api, graph=graph, n=n, edges=min(int(n * factor), 1 << (29 if api == "coo" else 27)), **options)
    if api in ("stream", "serve"):
        case.update(batches=rng.randint(1, 24), largest=int(n * 2 ** rng.uniform(-6, -2)), queries=int(10 ** rng.uniform(1, 6)))
    return case


# ------------------------------------------------------------------- inputs

def n_vertices(case):
    return case["width"] * case["height"] if case["graph"] == "grid" else case["n"]


def n_edges(case):
    if case["graph"] == "grid":
        w, h = case["width"], case["height"]
        return int(0.9 * (2 * w * h - w - h))
    return case["edges"]


def generator(seed, salt=0):
    return torch.Generator(DEV).manual_seed(seed * 1009 + salt)


def rmat_columns(scale, count, gen):
    """Both endpoint columns of `count` R-MAT edges, as int32 (scale <= 30)."""
    u = torch.zeros(count, dtype=torch.int32, device=DEV)
    v = torch.zeros_like(u)
    r = torch.empty_like(u)
    for _ in range(scale):
        r.random_(generator=gen)  # 31 bits
        low = r >= T_AB
        u.mul_(2).add_(low)
        v.mul_(2).add_((low ^ (r >= T_A)) | (r >= T_ABC))
    return u, v


def scramble(x, scale, seed):
    """A bijection of [0, 2^scale) in place, so that hubs get ids of any size."""
    mask = (1 << scale) - 1
    mix = np.random.RandomState(seed & 0x7FFFFFFF)
    for _ in range(2):
        x.mul_(int(mix.randint(0, 1 << 30)) | 1).add_(int(mix.randint(0, 1 << 30))).bitwise_and_(mask)
        x.bitwise_xor_(x >> ((scale + 1) // 2))
    return x


def edge_list(case, seed):
    """The case's edges as an (E, 2) int32 tensor."""
    gen = generator(seed)
    if case["graph"] == "grid":
        w, h = case["width"], case["height"]
        cell = torch.arange(w * h, dtype=torch.int32, device=DEV)
        both = torch.stack([torch.stack([cell, cell + 1], 1), torch.stack([cell, cell + w], 1)], 1)  # cell, direction, end
        keep = torch.rand((w * h, 2), generator=gen, device=DEV) < 0.9
        keep[:, 0] &= cell % w != w - 1
        keep[:, 1] &= cell < w * (h - 1)
        found = both[keep]
        edges = buffer(found.shape[0], case["shift"])
        edges.copy_(found)
        return edges  # already in source order
    n, total = case["n"], case["edges"]
    scale = max(1, (n - 1).bit_length())
    edges = buffer(total, case["shift"])
    for a in range(0, total, CHUNK):
        b = min(total, a + CHUNK)
        if case["graph"] == "uniform":
            edges[a:b].random_(0, n, generator=gen)
        else:
            for k, x in enumerate(rmat_columns(scale, b - a, gen)):
                x = scramble(x, scale, seed)
                edges[a:b, k] = x if n == 1 << scale else x % n
    if case["order"] == "source":
        edges.copy_(edges[torch.sort(edges[:, 0], stable=True).indices])
    return edges


def buffer(count, shift):
    flat = torch.empty(2 * count + 2, dtype=torch.int32, device=DEV)
    return flat[2:].view(count, 2) if shift else flat[: 2 * count].view(count, 2)


def pairs(n, count, seed, salt):
    return torch.randint(0, n, (count, 2), generator=generator(seed, salt), dtype=torch.int32, device=DEV)


def batch_sizes(case, largest):
    """Sizes from 1000 (or the largest, if smaller) up to the largest, evenly in the logarithm."""
    count = case["batches"]
    low = min(1000, largest)
    return [int(round(low * (largest / low) ** (i / max(1, count - 1)))) for i in range(count)]


def mixed_batch(case, seed):
    """Many graphs: 40% uniform, 40% R-MAT, 20% grid; 2^8 to 2^18 vertices, evenly in the logarithm;
    average degree 2 to 32. Edges hold graph-local ids, graph after graph. The shapes belong to the case, the
    edges to the seed."""
    count = case["graphs"]
    mix = np.random.RandomState(count)
    kind = mix.choice(3, count, p=[0.4, 0.4, 0.2])
    n = np.exp2(mix.uniform(8, 18, count)).astype(np.int64)
    m = np.where(kind == 2, (1.8 * n).astype(np.int64), (n * mix.uniform(1, 16, count)).astype(np.int64))
    vtx_off = torch.from_numpy(np.concatenate([[0], np.cumsum(n)])).to(DEV)
    edge_off = np.concatenate([[0], np.cumsum(m)])
    n_d, m_d, kind_d = (torch.from_numpy(x).to(DEV) for x in (n, m, kind))
    width = n_d.double().sqrt().long()
    scale = torch.from_numpy(np.ceil(np.log2(n)).astype(np.int32)).to(DEV)
    first = torch.from_numpy(edge_off[:-1]).to(DEV)
    gen = generator(seed)
    total = int(edge_off[-1])
    edges = torch.empty((total, 2), dtype=torch.int32, device=DEV)
    g0 = 0
    while g0 < count:
        g1 = max(g0 + 1, int(np.searchsorted(edge_off, edge_off[g0] + CHUNK // 2, "right")) - 1)
        a, b = int(edge_off[g0]), int(edge_off[g1])
        g = torch.repeat_interleave(torch.arange(g0, g1, device=DEV), m_d[g0:g1])
        vertices = n_d[g]
        # R-MAT columns of 18 levels; a graph of fewer vertices takes its last levels
        mask = (1 << scale[g].long()) - 1
        u, v = rmat_columns(18, b - a, gen)
        u, v = (u & mask) % vertices, (v & mask) % vertices
        uni = torch.rand((b - a, 2), generator=gen, device=DEV, dtype=torch.float64) * vertices[:, None]
        # grid: edge e of its graph takes one slot (cell, direction) near e / 0.9
        e = torch.arange(a, b, device=DEV) - first[g]
        slot = ((e + torch.rand(b - a, generator=gen, device=DEV, dtype=torch.float64)) / 0.9).long()
        cell = torch.minimum(slot >> 1, vertices - 1)
        w = width[g]
        right = torch.where(cell % w != w - 1, cell + 1, cell)
        other = torch.where(slot % 2 == 0, right, cell + w)
        other = torch.where(other < vertices, other, cell)
        k = kind_d[g]
        edges[a:b, 0] = torch.where(k == 0, uni[:, 0].long(), torch.where(k == 1, u, cell))
        edges[a:b, 1] = torch.where(k == 0, uni[:, 1].long(), torch.where(k == 1, v, other))
        g0 = g1
    return vtx_off, torch.from_numpy(edge_off).to(DEV), edges


def csr(n, edges):
    source, order = torch.sort(edges[:, 0], stable=True)
    offsets = torch.searchsorted(source, torch.arange(n + 1, dtype=torch.int32, device=DEV))
    return offsets, edges[:, 1][order].contiguous()


def pack(edges):
    """3-byte little-endian ids."""
    ids = edges.reshape(-1, 1)
    return torch.cat([ids & 255, (ids >> 8) & 255, (ids >> 16) & 255], 1).to(torch.uint8).reshape(-1)


# ------------------------------------------------------- prepare, run, work

def prepare(case, seed):
    """The inputs in place and the handle open, as a program keeps them."""
    api, state = case["api"], {"api": case["api"]}
    if api == "batch":
        state["vtx_off"], state["edge_off"], state["edges"] = mixed_batch(case, seed)
        state["labels"] = torch.empty(int(state["vtx_off"][-1]), dtype=torch.int32, device=DEV)
        state["graphs"], state["batch"] = case["graphs"], cc.Batch(case["graphs"])
        return state
    n, edges = n_vertices(case), edge_list(case, seed)
    state.update(n=n, edges=edges, labels=torch.empty(n, dtype=torch.int32, device=DEV))
    if api in ("stream", "serve"):
        sizes = batch_sizes(case, case["largest"])
        state["inserts"] = [pairs(n, k, seed, 1 + i) for i, k in enumerate(sizes)]
        state["queries"] = [pairs(n, case["queries"], seed, 101 + i) for i in range(len(sizes))]
        state["answers"] = [torch.empty(case["queries"], dtype=torch.uint8, device=DEV) for _ in sizes]
    if api == "serve":
        # twice the graph's parent array, logs and label copies
        state["first_labels"] = torch.empty_like(state["labels"])
        state["server"] = cc.Server(hbm_budget_bytes=(64 << 20) + 64 * n, idle_timeout_us=1000, mode=case["mode"],
                                    label_space=case["label_space"])
        return state
    if api == "csr":
        state["offsets"], state["neighbors"] = csr(n, edges)
        state["edges"] = None
    elif api in ("host", "packed"):
        flat = pack(edges) if api == "packed" else edges
        state["edges"] = torch.empty(flat.shape, dtype=flat.dtype, pin_memory=True)
        state["edges"].copy_(flat)
        state["labels"] = torch.empty(n, dtype=torch.int32, pin_memory=True)
        state["count"] = edges.shape[0]
    state["graph"] = cc.Graph(n, edges.shape[0] if api in ("host", "packed") else 0, mode=case["mode"],
                              label_space=case["label_space"], root_select=case["root_select"])
    return state


def run(state):
    api, labels = state["api"], state["labels"]
    if api == "batch":
        return state["batch"].run(state["graphs"], state["vtx_off"], state["edge_off"], state["edges"], labels)
    if api == "serve":
        server = state["server"]
        ticket, graph = server.new_graph(state["n"], state["edges"], state["first_labels"])
        tickets = [ticket]
        tickets += server.insert_many(graph, state["inserts"])
        tickets += server.query_many(graph, state["queries"], state["answers"])
        tickets += [server.snapshot(graph, labels), server.drop(graph)]
        for t in tickets:
            if server.wait(t) != cc.CC_OK:
                raise RuntimeError("a request failed")
        return [state["first_labels"], *state["answers"], labels]
    graph = state["graph"]
    if api == "coo":
        return graph.run(state["edges"], labels)
    if api == "csr":
        cc.cc_run_csr(graph.h, state["offsets"], state["neighbors"], L_out=labels)
    elif api == "host":
        cc.cc_run_host(graph.h, state["edges"], L_out_host=labels)
    elif api == "packed":
        cc.cc_run_host_packed(graph.h, state["edges"], state["count"], 3, labels)
    else:
        graph.run(state["edges"])
        for batch, queries, answers in zip(state["inserts"], state["queries"], state["answers"]):
            graph.insert(batch)
            graph.connected(queries, answers)
        graph.labels(labels)
        return [*state["answers"], labels]
    return labels


def work(case):
    """Each edge read once and each label written once; CSR reads its offsets
    and neighbours, a batch its offsets; 3-byte ids take 6 bytes an edge. No
    arithmetic is counted: the work is lookups."""
    if case["api"] == "batch":
        vertices = case["graphs"] * (2 ** 18 - 2 ** 8) / math.log(2 ** 10)
        return {"bytes": vertices * (8 * 0.8 * 8.5 + 8 * 0.2 * 1.8 + 4) + 16 * case["graphs"], "flops": 0}
    n, m = n_vertices(case), n_edges(case)
    size = {"csr": 8 * (n + 1) + 4 * m, "packed": 6 * m}.get(case["api"], 8 * m) + 4 * n
    if case["api"] in ("stream", "serve"):
        size += 8 * sum(batch_sizes(case, case["largest"])) + 9 * case["batches"] * case["queries"]
        size += 4 * n if case["api"] == "serve" else 0
    return {"bytes": size, "flops": 0}


# -------------------------------------------------------------------- exact

def min_labels(n, edges):
    """The smallest vertex of every vertex's component: each vertex takes the
    smallest label across its edges, then labels are followed to their ends,
    until nothing changes."""
    label = torch.arange(n, device=DEV)
    changed = True
    while changed:
        before = label.clone()
        for a in range(0, edges.shape[0], CHUNK // 4):
            u, v = edges[a:a + CHUNK // 4].long().unbind(1)
            lu, lv = before[u], before[v]
            low = torch.minimum(lu, lv)
            for x in (u, v, lu, lv):
                label.scatter_reduce_(0, x, low, "amin")
        while True:
            nearer = label[label]
            if torch.equal(nearer, label):
                break
            label = nearer
        changed = not torch.equal(before, label)
    return label


def exact(case, seed):
    if case["api"] == "batch":
        vtx_off, edge_off, edges = mixed_batch(case, seed)
        if edges.shape[0] > 1 << 28:
            return None
        graphs = torch.arange(case["graphs"], device=DEV)
        base = torch.repeat_interleave(vtx_off[:-1][graphs], edge_off.diff())
        label = min_labels(int(vtx_off[-1]), edges + base[:, None])
        return label - torch.repeat_interleave(vtx_off[:-1], vtx_off.diff())
    if n_edges(case) > 1 << 28 or (case["label_space"] == cc.CC_LABEL_ROOT_VALUE and case["mode"] == cc.CC_ROOT_MAXDEG):
        return None  # the root value of a label depends on which vertex was planted
    n, edges = n_vertices(case), edge_list(case, seed)
    if case["api"] not in ("stream", "serve"):
        return min_labels(n, edges).cpu() if case["api"] in ("host", "packed") else min_labels(n, edges)
    sizes = batch_sizes(case, case["largest"])
    label = first = min_labels(n, edges)
    answers = []
    vertices = torch.arange(n, device=DEV)
    for i, k in enumerate(sizes):
        label = min_labels(n, torch.cat([torch.stack([vertices, label], 1), pairs(n, k, seed, 1 + i)]))
        answers.append(label[pairs(n, case["queries"], seed, 101 + i).long()])
    if case["api"] == "serve":  # the inserts run together, then every query
        answers = [label[pairs(n, case["queries"], seed, 101 + i).long()] for i in range(len(sizes))]
    answers = [(a[:, 0] == a[:, 1]).long() for a in answers]
    return [first, *answers, label] if case["api"] == "serve" else [*answers, label]
