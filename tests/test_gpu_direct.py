"""The one-kernel matcher (calls with default options) at the sizes where its
buffers and tasks end: runs around one load of a lane, a row batch and the
next-candidate buffer, lists kept beside sets, level and root buffers, dense
and sparse sets, steps cut into tasks, batches of one and of many queries.
Every result equals the oracle's, and the staged pipeline's."""
import numpy as np
import pytest

import oracle as O
import paper_1807_08804_gb300 as gs
from paper_1807_08804_gb300 import inputs as I
from tests.helpers import complete_digraph_triples, graph_from_triples, query, random_tiny

pytestmark = pytest.mark.gpu


def check(g, qs, cap=1 << 12, project=None):
    og = O.OracleGraph.from_graph(g)
    dg = gs.DeviceGraph(g)
    got = gs.match_batch(dg, qs, cap=cap, project=project)
    staged = gs.match_batch(dg, qs, cap=cap, project=project, max_refine_rounds=1)
    count = gs.match_batch(dg, qs, cap=0, mode=gs.GS_COUNT_ONLY)
    for i, q in enumerate(qs):
        o = O.match(og, q, cap=cap, project=project)
        for r in (got[i], staged[i]):
            assert r.status == 0 and (r.count, r.fingerprint) == (o.count, o.fingerprint), i
            np.testing.assert_array_equal(r.rows, o.rows, err_msg=str(i))
        assert (count[i].count, count[i].fingerprint) == (o.count, o.fingerprint), i
    dg.free()


@pytest.mark.parametrize("leaves", [1, 2, 7, 8, 9, 31, 32, 33, 80, 81, 255, 256, 257, 511, 513, 1023, 1024, 1025, 2049])
def test_hubs(leaves):
    """A hub with out-leaves over relation 1 and others over 0 and 2 around
    them, and in-leaves: runs of every length, shared by all partial rows."""
    tr = [(0, 1, 1 + i) for i in range(leaves)] + [(0, 0, leaves + 1), (0, 2, leaves + 2)]
    tr += [(leaves + 3 + i, 1, 0) for i in range(40)]
    V = leaves + 43
    g = graph_from_triples(V, tr, [0] + [1 + v % 2 for v in range(1, V)], 3, 3)
    few = leaves <= 300
    qs = [query(2, [(0, 1, 1)]), query(3, [(0, 1, 1), (0, 2, 1)]), query(3, [(1, 0, 1), (0, 2, 1)]),
          query(2, [(0, 1, I.ANY)]), query(3, [(0, 1, 0), (0, 2, 1)], vtype=[I.ANY, I.ANY, 1]),
          query(3, [(0, 1, 1), (2, 0, 1)], vbind=[0, I.UNBOUND, I.UNBOUND])]
    if few:
        qs.append(query(4, [(0, 1, 1), (0, 2, 1), (3, 0, 1)], vtype=[0, 1, 2, I.ANY]))
    check(g, qs)
    check(g, qs, project=[0, 1])


@pytest.mark.parametrize("V", [2, 31, 33, 1023, 1025, 5000, 33_000])
def test_whole_sets(V):
    """Untyped vertices, so a set is the whole graph: dense sets, root
    candidates past the root buffer, queries of one vertex."""
    rng = np.random.default_rng(V)
    src = rng.integers(0, V, 3 * V)
    dst = rng.integers(0, V, 3 * V)
    tr = sorted({(int(s), int(r), int(d)) for s, r, d in zip(src, rng.integers(0, 2, 3 * V), dst) if s != d})
    g = graph_from_triples(V, tr, rng.integers(0, 3, V), 3, 2)
    qs = [query(1, []), query(1, [], vtype=[1]), query(1, [], vbind=[V - 1]), query(2, [(0, 1, 0)]),
          query(3, [(0, 1, 0), (1, 2, 1)]), query(3, [(0, 1, 0), (1, 2, 1), (2, 0, 0)]),
          query(3, [(0, 1, I.ANY), (1, 2, 0)], vtype=[0, I.ANY, 2])]
    check(g, qs, cap=5000)


@pytest.mark.parametrize("n", [5, 9, 12])
def test_cliques(n):
    """Several edges per joined vertex: the shortest run drives, the others
    are probed; levels pass their buffers."""
    g = graph_from_triples(n, complete_digraph_triples(n))
    qs = [query(k, [(i, j, 0) for i in range(k) for j in range(i + 1, k)]) for k in (3, 4, 5)]
    qs += [query(4, [(i, (i + 1) % 4, 0) for i in range(4)]), query(5, [(0, i, 0) for i in range(1, 5)])]
    check(g, qs, cap=1 << 10)


@pytest.mark.parametrize("copies", [1, 3, 700])
def test_batches_of_one_and_many(copies):
    """Few queries (every step may be cut into tasks) and more queries than
    tasks are worth; each copy gives the same result."""
    g = I.make_graph(20_000, 160_000, seed=5)
    qs = I.make_walk_queries(g, 12, 3, 7, p_bind=0.1, seed=9)
    og, dg = O.OracleGraph.from_graph(g), gs.DeviceGraph(g)
    want = [O.match(og, q, cap=1 << 16) for q in qs]
    for _ in range(3):  # the queue and counters start over with each run
        got = gs.match_batch(dg, qs * copies, cap=1 << 16)
        for i, r in enumerate(got):
            o = want[i % len(qs)]
            assert (r.status, r.count, r.fingerprint) == (0, o.count, o.fingerprint), i
            np.testing.assert_array_equal(r.rows, o.rows)
    dg.free()


def test_random_instances():
    rng = np.random.default_rng(123)
    for case in range(60):
        g, q = random_tiny(rng, n_max=9, k_max=6, p_any=0.2)
        check(g, [q, q], cap=1 << 10)


def test_join_sizes_without_refinement():
    """A batch asked to run without refinement takes the one-kernel matcher;
    its partial-embedding sizes lie between the refined and the unpruned."""
    g = I.make_graph(10_000, 60_000, seed=3)
    qs = I.make_walk_queries(g, 60, 3, 6, p_bind=0.1, seed=4)
    dg = gs.DeviceGraph(g)
    b = gs.Batch(dg, qs, cap=1 << 12)
    size = {}
    for graph in (True, False):
        b.configure(use_graph=graph, group=32, refine_rounds=gs.GS_ROUNDS_NONE)
        b.run()
        b.finish()
        size[graph] = b.join_sizes()[0].sum(), [(r.count, r.fingerprint) for r in b.fetch()]
    assert size[True][1] == size[False][1]
    assert 0 < size[True][0] <= size[False][0]
    b.close()
    dg.free()


def test_buckets_that_overflow_take_the_merge_path():
    """17.3 million rows of one query: more than 4,096 samples can cut into
    buckets of 4,096, so the call sorts it by merge passes after all.  The
    first call finds the output pool too small and finishes on the chunked
    path; the later ones, with the pool enlarged, give the same rows."""
    from math import perm
    n, k, cap = 14, 7, 1 << 21
    dg = gs.DeviceGraph(graph_from_triples(n, complete_digraph_triples(n)))
    q = query(k, [(i, i + 1, 0) for i in range(k - 1)])
    first = gs.match(dg, q, cap=cap)
    assert first.count == perm(n, k) and first.rows.shape == (cap, k)
    want = np.array([0, 1, 2, 3, 4, 5, 6], np.uint32)
    np.testing.assert_array_equal(first.rows[0], want)
    for _ in range(2):
        r = gs.match(dg, q, cap=cap)
        assert (r.count, r.fingerprint) == (first.count, first.fingerprint)
        np.testing.assert_array_equal(r.rows, first.rows)
    dg.free()
