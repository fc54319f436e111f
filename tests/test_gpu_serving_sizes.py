"""Serving bursts whose queries are all as large as queries get: a micro-batch
holds as many of them as a slot's vertices and edges allow."""
import time

import numpy as np
import pytest

import paper_1807_08804_gb300 as gs
from paper_1807_08804_gb300 import inputs as I
from tests.helpers import complete_digraph_triples, graph_from_triples, query

pytestmark = pytest.mark.gpu


def drain(srv, tickets, timeout_s=120.0):
    out, t0 = {}, time.time()
    while len(out) < len(tickets):
        assert time.time() - t0 < timeout_s, "serving did not finish in time"
        for t in tickets:
            if t not in out:
                r = srv.poll(t)
                if r is not None:
                    out[t] = r[0]
        time.sleep(0.0005)
    return [out[t] for t in tickets]


@pytest.mark.parametrize("max_batch", [4, 64, 256])
def test_bursts_of_large_queries(max_batch):
    g = I.make_graph(10_000, 60_000, seed=31)
    qs = I.make_walk_queries(g, 300, 11, 12, p_bind=0.3, seed=32)
    dg = gs.DeviceGraph(g)
    want = gs.match_batch(dg, qs, cap=1 << 10)
    srv = gs.Server(dg, slots=2, max_batch=max_batch)
    got = drain(srv, [srv.submit(q, cap=1 << 10) for q in qs])
    for r, a in zip(got, want):
        assert (r.status, r.count, r.fingerprint) == (0, a.count, a.fingerprint)
        np.testing.assert_array_equal(r.rows, a.rows)
    srv.close()
    dg.free()


@pytest.mark.parametrize("max_batch", [1, 3, 9])
def test_queries_of_many_edges(max_batch):
    """Cliques of five vertices over every pair, in both directions, some with
    each edge given twice."""
    dg = gs.DeviceGraph(graph_from_triples(7, complete_digraph_triples(7)))
    edges = [(a, b, 0) for a in range(5) for b in range(5) if a != b]
    qs = [query(5, edges), query(5, edges * 2), query(2, [(0, 1, 0)])] * 8
    want = gs.match_batch(dg, qs, cap=1 << 12)
    assert want[0].count == 7 * 6 * 5 * 4 * 3
    srv = gs.Server(dg, slots=2, max_batch=max_batch)
    for r, a in zip(drain(srv, [srv.submit(q, cap=1 << 12) for q in qs]), want):
        assert (r.status, r.count, r.fingerprint) == (0, a.count, a.fingerprint)
        np.testing.assert_array_equal(r.rows, a.rows)
    srv.close()
    dg.free()
