"""What a user of the matcher has it do, as cases that can be timed: single
queries, batches of every size, pages of the first answers, projections,
count-only runs, a burst of served requests, matching through a compressed
graph and k-hop exploration, on graphs of 10,000 to 16 million vertices.

The graphs have the shape of the repository's own workloads (power-law
out-degree, Zipf types and relations, uniform targets) and are drawn on the
GPU.  A query is a random walk over the undirected view of its graph plus 30%
of the other triples among the walked vertices, so it has at least one match,
or one of the unbound cycles, cliques and trees of the output-heavy workload.
Graphs are loaded and queries are packed beforehand, as in a program that
answers queries over a resident graph; nothing is tuned.

Every output is a whole number: counts, fingerprints, row numbers, rows in
query order, levels.
"""
import ctypes
import math
import time

import numpy as np
import torch

import paper_1807_08804_gb300 as gs
from paper_1807_08804_gb300 import inputs

TYPES, RELS, DMAX = 64, 34, 1000


def _match(name, V, E, n, kmin, kmax, bind, cap, var=0.0, project=0):
    return dict(name=name, kind="match", V=V, E=E, n=n, kmin=kmin, kmax=kmax, bind=bind, cap=cap, var=var,
                project=project)


def listed():
    return [
        # one interactive question over a small domain graph: launches and latency
        _match("one-10k", 10_000, 60_000, 1, 3, 6, 0.2, 1 << 20),
        # one question over a knowledge graph of a million concepts
        _match("one-1m", 1_000_000, 8_000_000, 1, 4, 10, 0.2, 1 << 22),
        # a form's worth of questions over the small graph
        _match("batch-10k", 10_000, 60_000, 100, 3, 6, 0.2, 1 << 20),
        # an ordinary batch over the million-vertex graph
        _match("batch-1m", 1_000_000, 8_000_000, 1000, 4, 10, 0.2, 1 << 22),
        # questions whose relations are partly unknown, of which only two vertices are wanted back
        _match("variable-1m", 1_000_000, 8_000_000, 301, 4, 10, 0.2, 1 << 16, var=0.3, project=2),
        # the first page of the answers to each of many questions over the 4M-vertex graph
        _match("page-4m", 4_000_000, 32_000_000, 2001, 3, 12, 0.2, 1 << 10),
        # thousands of questions of uneven size at once, every embedding wanted: the headline load
        _match("batch-4m", 4_000_000, 32_000_000, 5000, 3, 12, 0.1, 1 << 20),
        # graph mining: how often do unbound cycles, cliques and trees occur in the largest graph
        dict(name="shapes-count-16m", kind="shapes", V=16_000_000, E=200_000_000, n=200, cap=0),
        # the same shapes with up to 65,536 of the embeddings of each: output-heavy
        dict(name="shapes-rows-4m", kind="shapes", V=4_000_000, E=50_000_000, n=100, cap=1 << 16),
        # a burst of requests to the serving loop (continuous batching), until every answer is there
        dict(name="serve-1m", kind="serve", V=1_000_000, E=8_000_000, n=500, kmin=3, kmax=12, bind=0.2, cap=1 << 20),
        # a batch through the multi-level compressed graph (three levels, concept families)
        dict(name="compressed-10k", kind="compressed", V=10_000, E=60_000, n=100, kmin=3, kmax=6, bind=0.2,
             cap=1 << 20),
        # a domain's concepts: everything within four hops of 16 seeds of the largest graph
        dict(name="khop-16m", kind="khop", V=16_000_000, E=200_000_000, n=16, levels=4),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["match"] * 6 + ["shapes", "shapes", "serve", "compressed", "khop"])
    if kind == "match":
        V = log(10_000, 4_000_000)
        kmin = rng.randint(3, 5)
        var = rng.choice([0.0, 0.0, 0.0, 0.3])
        cap = 1 << rng.choice([10, 16] if var else [10, 16, 20, 22])
        most = 300 if var else 2000 if cap < 1 << 16 else 4000
        return dict(kind=kind, V=V, E=int(V * rng.uniform(6, 8)), n=log(1, most), kmin=kmin,
                    kmax=rng.randint(kmin + 1, 10 if var else 12), bind=rng.choice([0.1, 0.2]), cap=cap, var=var,
                    project=rng.choice([0, 0, 2]))
    if kind == "shapes":
        cap = rng.choice([0, 1 << 16])
        V = log(100_000, 4_000_000 if cap else 16_000_000)
        return dict(kind=kind, V=V, E=int(V * 12.5), n=rng.randint(4, 100 if cap else 200), cap=cap)
    if kind == "serve":
        V = log(10_000, 1_000_000)
        return dict(kind=kind, V=V, E=int(V * rng.uniform(6, 8)), n=log(1, 500), kmin=3, kmax=rng.randint(4, 12),
                    bind=0.2, cap=1 << 20)
    if kind == "compressed":
        V = rng.randint(2_000, 10_000)
        return dict(kind=kind, V=V, E=6 * V, n=log(1, 100), kmin=3, kmax=rng.randint(4, 6), bind=0.2, cap=1 << 20)
    V = log(10_000, 16_000_000)
    return dict(kind=kind, V=V, E=int(V * rng.uniform(6, 12.5)), n=log(1, 64), levels=rng.randint(2, 4))


# ------------------------------------------------------------------ inputs
def _zipf(labels, s, count, gen):
    cdf = torch.cumsum(torch.arange(1, labels + 1, dtype=torch.float64, device="cuda") ** -s, 0)
    u = torch.rand(count, dtype=torch.float64, device="cuda", generator=gen) * cdf[-1]
    return torch.searchsorted(cdf, u).clamp_(max=labels - 1).int()


def _graph(V, E, gen):
    """A directed graph as an out-CSR on the GPU: Pareto out-degrees (density
    exponent 2.1) scaled to sum to E, uniform targets."""
    x = (1 - torch.rand(V, dtype=torch.float64, device="cuda", generator=gen)) ** (-1 / 1.1)

    def degrees(c):
        return torch.floor(c * x + 0.5).clamp_(1, DMAX)

    lo, hi = 0.0, float(DMAX)
    for _ in range(60):
        c = 0.5 * (lo + hi)
        lo, hi = (c, hi) if int(degrees(c).sum()) <= E else (lo, c)
    deg = degrees(lo).long()
    more = torch.randint(V, (E - int(deg.sum()),), device="cuda", generator=gen)
    deg.index_add_(0, more, torch.ones_like(more))
    off = torch.zeros(V + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(deg, 0, out=off[1:])
    src = torch.repeat_interleave(torch.arange(V, dtype=torch.int32, device="cuda"), deg)
    dst = torch.randint(V - 1, (E,), dtype=torch.int32, device="cuda", generator=gen)
    dst += dst >= src
    rel = _zipf(RELS, 1.1, E, gen)
    while True:  # repeated triples are redrawn
        triple, at = torch.sort((src.long() * V + dst) * RELS + rel)
        at = at[1:][triple[1:] == triple[:-1]].sort()[0]
        if not at.numel():
            break
        new = torch.randint(V - 1, (at.numel(),), dtype=torch.int32, device="cuda", generator=gen)
        dst[at] = new + (new >= src[at])
    del triple, at
    return dict(V=V, E=E, off=off, src=src, dst=dst, rel=rel, type=_zipf(TYPES, 1.0, V, gen))


def _load(g):
    torch.cuda.synchronize()  # the loader reads the arrays on a stream of its own
    return gs.DeviceGraph(num_vertices=g["V"], num_edges=g["E"], row_offsets=g["off"].data_ptr(),
                          col_targets=g["dst"].data_ptr(), edge_rel=g["rel"].data_ptr(),
                          vertex_type=g["type"].data_ptr(), num_types=TYPES, num_rels=RELS, device_ptrs=True)


def _walks(g, n, kmin, kmax, bind, var, gen):
    """n queries walked at once: tree edges are the traversed data edges, each
    other data edge between two walked vertices joins with probability 0.3."""
    V, off, src, dst, rel = (g[k] for k in ("V", "off", "src", "dst", "rel"))
    order = torch.argsort(dst, stable=True)
    ioff = torch.zeros(V + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.bincount(dst, minlength=V), 0, out=ioff[1:])
    k = torch.randint(kmin, kmax + 1, (n,), device="cuda", generator=gen)
    ids = torch.full((n, kmax), -1, dtype=torch.int64, device="cuda")
    esrc, edst, erel = (torch.full((n, kmax), -1, dtype=torch.int64, device="cuda") for _ in range(3))
    cur = torch.randint(V, (n,), device="cuda", generator=gen)
    ids[:, 0] = cur
    have = torch.ones_like(k)
    for _ in range(8 * kmax):
        outs, ins = off[cur + 1] - off[cur], ioff[cur + 1] - ioff[cur]
        pick = (torch.rand(n, dtype=torch.float64, device="cuda", generator=gen) * (outs + ins)).long()
        fwd = pick < outs
        e = torch.where(fwd, off[cur] + pick, order[torch.where(fwd, 0, ioff[cur] + pick - outs)])
        nxt = torch.where(fwd, dst[e], src[e]).long()
        new = (ids != nxt[:, None]).all(1) & (have < k)
        q, here, there = new.nonzero()[:, 0], (ids == cur[:, None]).int().argmax(1)[new], have[new]
        ids[q, there] = nxt[new]
        esrc[q, there] = torch.where(fwd[new], here, there)
        edst[q, there] = torch.where(fwd[new], there, here)
        erel[q, there] = rel[e[new]].long()
        have += new
        more = have < k
        cur = torch.where(more, nxt, cur)
        if not bool(more.any()):
            break
    # one data edge of every ordered pair of walked vertices, if there is any
    pair, at = torch.sort(src.long() * V + dst)
    want = torch.where((ids[:, :, None] >= 0) & (ids[:, None, :] >= 0), ids[:, :, None] * V + ids[:, None, :], -1)
    found = torch.searchsorted(pair, want.reshape(-1)).clamp_(max=g["E"] - 1)
    close = (pair[found] == want.reshape(-1)) & (torch.rand(found.numel(), device="cuda", generator=gen) < 0.3)
    close = close.reshape(n, kmax, kmax)
    q, there = (esrc >= 0).nonzero(as_tuple=True)
    close[q, esrc[q, there], edst[q, there]] = False  # tree edges are there already
    q, a, b = close.nonzero(as_tuple=True)
    r = rel[at[found.reshape(n, kmax, kmax)[q, a, b]]]
    extra = {}
    for row in torch.stack([q, a, b, r.long()], 1).tolist():
        extra.setdefault(row[0], []).append(row[1:])
    del pair, at
    bound = torch.rand((n, kmax), device="cuda", generator=gen) < bind
    types = torch.where(bound, gs.ANY, g["type"][ids.clamp_min(0)].long())
    binds = torch.where(bound, ids, gs.UNBOUND)
    erel = torch.where(torch.rand((n, kmax), device="cuda", generator=gen) < var, gs.ANY, erel)
    have, types, binds, esrc, edst, erel = (t.cpu().numpy() for t in (have, types, binds, esrc, edst, erel))
    out = []
    for i in range(n):
        m, add = int(have[i]), np.array(extra.get(i, []), np.int64).reshape(-1, 3)
        out.append(inputs.Query(types[i, :m].astype(np.uint32), binds[i, :m].astype(np.uint32),
                                *(np.concatenate([t[i, 1:m], add[:, j]]).astype(np.uint32)
                                  for j, t in enumerate((esrc, edst, erel)))))
    return out


def prepare(case, seed):
    gen = torch.Generator("cuda")
    gen.manual_seed(seed)
    c = dict(case)
    if c["kind"] != "khop":
        c["rows"] = np.zeros(min(c["n"] * c["cap"] * (c.get("project") or c.get("kmax", 6)), 1 << 27), np.int32)
    if c["kind"] == "compressed":
        g = inputs.make_graph(c["V"], c["E"], seed=seed, target_s=1.3, copy_p=0.8)
        return dict(c, graph=gs.CompressedGraph(g, [0.8, 0.7, 0.7]),
                    queries=inputs.make_walk_queries(g, c["n"], c["kmin"], c["kmax"], p_bind=c["bind"], seed=seed))
    g = _graph(c["V"], c["E"], gen)
    graph = _load(g)
    if c["kind"] == "khop":
        seeds = torch.randint(c["V"], (c["n"],), dtype=torch.int32, device="cuda", generator=gen)
        s = dict(c, graph=graph, seeds=seeds, level=torch.empty(c["V"], dtype=torch.uint8, device="cuda"))
    else:
        if c["kind"] == "shapes":  # over the most frequent relations and types
            few = inputs.Graph(1, None, None, g["rel"][:1_000_000].cpu().numpy(), g["type"][:1_000_000].cpu().numpy(),
                               TYPES, RELS)
            queries = inputs.make_shape_queries(few, c["n"], seed=seed)
        else:
            queries = _walks(g, c["n"], c["kmin"], c["kmax"], c["bind"], c.get("var", 0.0), gen)
        s = dict(c, graph=graph, queries=queries, pack=gs.QueryPack(queries))
        if c["kind"] == "serve":
            s["server"] = gs.Server(graph)
    del g
    torch.cuda.empty_cache()  # the library allocates beside torch
    return s


# --------------------------------------------------------------------- run
# A program takes the rows of all its queries, in query order, into a buffer
# of its own (zeros past the last row).
def _answers(s, res, block):
    """Results of the C ABI call."""
    n, buf = s["n"], s["rows"]
    a = np.frombuffer(res, gs.RES_DTYPE, n).copy()
    if int((a["num_rows"] * a["k"]).sum()) > buf.size:
        raise RuntimeError("more rows than the buffer holds")
    gs.check(gs.lib().gs_results_copy_rows(res, n, buf.ctypes.data_as(ctypes.c_void_p)))
    gs.lib().gs_results_free(res, n)
    if block:
        gs.lib().gs_rows_release(block)
    return dict(count=a["count"].view(np.int64), fingerprint=a["fingerprint"].view(np.int64),
                num_rows=a["num_rows"].view(np.int64), truncated=a["truncated"].astype(np.int32),
                status=a["status"].astype(np.int32), rows=buf)


def _results(s, got):
    """Results of the Python calls, a list of MatchResult."""
    rows = [r.rows for r in got]
    total = sum(r.size for r in rows)
    if total > s["rows"].size:
        raise RuntimeError("more rows than the buffer holds")
    np.concatenate([r.reshape(-1) for r in rows], out=s["rows"][:total].view(np.uint32))
    return dict(count=np.array([r.count for r in got], np.int64),
                fingerprint=np.array([r.fingerprint for r in got], np.uint64).view(np.int64),
                num_rows=np.array([r.shape[0] for r in rows], np.int64), rows=s["rows"])


def run(state):
    s = state
    if s["kind"] == "khop":
        _, counts, scanned = gs.khop(s["graph"], None, s["levels"],
                                     device=(s["seeds"].data_ptr(), s["n"], s["level"].data_ptr()))
        return dict(level=s["level"], counts=counts.view(np.int64), scanned=scanned)
    if s["kind"] == "compressed":
        return _results(s, s["graph"].match_batch(s["queries"], cap=s["cap"]))
    if s["kind"] == "serve":
        tickets = [s["server"].submit_packed(s["pack"], i, cap=s["cap"]) for i in range(s["n"])]
        got = []
        for t in tickets:
            r = s["server"].poll(t)
            while r is None:
                time.sleep(50e-6)
                r = s["server"].poll(t)
            got.append(r[0])
        return _results(s, got)
    if s["n"] == 1:
        return _results(s, [gs.match(s["graph"], s["queries"][0], cap=s["cap"], project=range(s.get("project", 0)))])
    n, res, block = s["n"], (gs.ResultDesc * s["n"])(), gs.P()
    o = gs.match_opts(cap=s["cap"], mode=gs.GS_ENUMERATE if s["cap"] else gs.GS_COUNT_ONLY,
                      project=range(s.get("project", 0)))
    gs.check(gs.lib().gs_match_batch_shared(s["graph"]._h, s["pack"].arr, n, ctypes.byref(o), res,
                                            ctypes.byref(block)))
    return _answers(s, res, block)


# -------------------------------------------------------------------- work
def work(case):
    """Bytes that one pass cannot do without.  How much of the graph a query
    touches and how many rows it has vary from draw to draw, so these are
    means: per walked query the degree test of its rarest type's vertices, 20
    adjacency rows per query vertex, and the rows measured on these graphs."""
    c = case
    V, E, n, d = c["V"], c["E"], c["n"], 2 * c["E"] / c["V"]
    graph = 8 * E + 18 * V  # both directions' entries and offsets, types, one degree count per vertex
    if c["kind"] == "khop":
        # each hop's frontier is some d times the one before, more where hubs are in it
        scanned = sum(min(0.4 * E, n * d * (2.5 * d) ** hop) for hop in range(c["levels"]))
        return dict(bytes=V * 1.125 + 4 * scanned + 20 * min(V, scanned), flops=0)
    if c["kind"] == "shapes":
        # the lists of the query edges between frequent types, and a row list per query
        return dict(bytes=min(graph, n * 0.02 * graph) + n * 16 + 0.3 * n * c["cap"] * 20, flops=0)
    k = 0.5 * (c["kmin"] + c["kmax"])
    touched = min(graph, n * (0.008 * V * 5 + k * 20 * (16 + 4 * d)))
    rows = min(c["cap"], 100 if V <= 1_000_000 else 1000) * (20 if c.get("var") else 1)
    return dict(bytes=touched + n * (20 * k + 32) + n * rows * 4 * (c.get("project") or k), flops=0)


def exact(case, seed):
    return None  # outputs are whole numbers, the same for every correct program
