"""The one-kernel matcher where its limits meet: rows that share a relation
run longer than the next-candidate buffer while work is handed to others,
settings that find no memory for their pools, outputs past what the device
keeps, outputs that find room in a second pass, and a work queue of a few
places whose workers leave early."""
from math import perm

import numpy as np
import pytest

import paper_1807_08804_gb300 as gs
from paper_1807_08804_gb300 import inputs as I
from tests.helpers import complete_digraph_triples, graph_from_triples, query

pytestmark = pytest.mark.gpu


def hub(leaves, few=0):
    """Vertex 0 with `leaves` out-neighbours over relation 0 and `few` others
    over relation 1."""
    tr = [(0, 0, 1 + i) for i in range(leaves)] + [(0, 1, 1 + leaves + i) for i in range(few)]
    return graph_from_triples(1 + leaves + few, tr, R=2)


def star(rels):
    return query(len(rels) + 1, [(0, i + 1, r) for i, r in enumerate(rels)])


@pytest.mark.parametrize("leaves", [1025, 1100, 1300])
def test_long_run_shared_by_many_rows(leaves):
    """Stars over a hub: every partial embedding draws on one run of more than
    1,024 entries, which is taken in parts, and workers run out of work of
    their own while others are between two parts."""
    dg = gs.DeviceGraph(hub(leaves))
    q = star([0, 0, 0])
    n = leaves * (leaves - 1) * (leaves - 2)
    want = gs.match(dg, q, cap=0, mode=gs.GS_COUNT_ONLY, max_refine_rounds=1)
    assert want.count == n
    for _ in range(4):
        r = gs.match(dg, q, cap=0, mode=gs.GS_COUNT_ONLY)
        assert (r.count, r.fingerprint) == (n, want.fingerprint)
    dg.free()


def test_long_run_in_a_batch_that_runs_dry():
    """More queries than workers, so that workers go from busy to idle while
    hub stars are joined; and a variant with rows returned."""
    leaves, few = 1100, 12
    dg = gs.DeviceGraph(hub(leaves, few))
    qs = [star([0, 0]), star([1, 0, 0])]
    ns = [leaves * (leaves - 1), few * leaves * (leaves - 1)]
    want = [gs.match(dg, q, cap=0, mode=gs.GS_COUNT_ONLY, max_refine_rounds=1) for q in qs]
    assert [w.count for w in want] == ns
    for q, w, copies in ((qs[0], want[0], 4500), (qs[1], want[1], 700)):
        for _ in range(2):
            got = gs.match_batch(dg, [q] * copies, cap=0, mode=gs.GS_COUNT_ONLY)
            assert {(r.status, r.count, r.fingerprint) for r in got} == {(0, w.count, w.fingerprint)}
    first = np.array([[0, 1 + leaves, 1, 2 + i] for i in range(100)], np.uint32)
    for _ in range(3):
        r = gs.match(dg, qs[1], cap=100)
        assert (r.count, r.fingerprint) == (want[1].count, want[1].fingerprint)
        np.testing.assert_array_equal(r.rows, first)
    dg.free()


@pytest.mark.parametrize("first,second", [(0, gs.GS_ROUNDS_NONE), (gs.GS_ROUNDS_NONE, 2)])
def test_settings_without_memory_leave_the_batch_as_it_was(first, second):
    """gs_batch_set to the other pipeline, whose pools it makes: an allocation
    that fails leaves the batch with the settings and pools it had, and
    nothing allocated."""
    import torch
    g = I.make_graph(10_000, 60_000, seed=41)
    qs = I.make_walk_queries(g, 30, 3, 6, p_bind=0.2, seed=42)
    dg = gs.DeviceGraph(g)
    want = [(r.count, r.fingerprint) for r in gs.match_batch(dg, qs, cap=1 << 10)]
    gs.tune_set(dg, 0, first)
    b = gs.Batch(dg, qs, cap=1 << 10)
    b.run()
    b.finish()
    free0 = torch.cuda.mem_get_info()[0]
    for after in range(64):
        gs.debug_fail_alloc(after)
        try:
            b.configure(refine_rounds=second)
        except gs.GSError as e:
            assert e.status == gs.GS_ERR_OOM
            assert torch.cuda.mem_get_info()[0] >= free0
        else:
            break
        finally:
            gs.debug_fail_alloc(-1)
        b.run()
        b.finish()
        assert [(r.count, r.fingerprint) for r in b.fetch()] == want
    assert 5 <= after < 63
    b.run()
    b.finish()
    assert [(r.count, r.fingerprint) for r in b.fetch()] == want
    b.close()
    dg.free()


def paths(k):
    return query(k, [(i, i + 1, 0) for i in range(k - 1)])


def test_large_outputs_leave_the_others_their_room():
    """Two queries of 19.5 million embeddings, more than the device keeps,
    among 300 of 342 rows and four of 93,024: only those two finish on the
    chunked path, on the first run and on later ones."""
    dg = gs.DeviceGraph(graph_from_triples(19, complete_digraph_triples(19)))
    qs = [paths(2)] * 150 + [paths(6)] + [paths(4)] * 4 + [paths(6)] + [paths(2)] * 150
    cap = 1 << 10
    want = {q.k: gs.match(dg, q, cap=cap, max_refine_rounds=1) for q in (paths(2), paths(4), paths(6))}
    assert [want[k].count for k in (2, 4, 6)] == [perm(19, k) for k in (2, 4, 6)]
    b = gs.Batch(dg, qs, cap=cap)
    b.configure(refine_rounds=gs.GS_ROUNDS_NONE)
    for _ in range(2):
        b.run()
        b.finish()
        assert b.counters()["fallback_queries"] == 2
        for q, r in zip(qs, b.fetch()):
            w = want[q.k]
            assert (r.status, r.count, r.fingerprint) == (0, w.count, w.fingerprint)
            np.testing.assert_array_equal(r.rows, w.rows)
    words = b.join_sizes()[0]  # of every query, whichever pass it was in
    assert {q.k: int(x) for q, x in zip(qs, words)} == {2: 19, 4: 19 + 2 * 342 + 3 * 5814,
                                                       6: 19 + 2 * 342 + 3 * 5814 + 4 * 93024 + 5 * 1395360}
    b.finish()  # once more without a run: the same results
    assert [r.count for r in b.fetch()] == [want[q.k].count for q in qs]
    np.testing.assert_array_equal(b.fetch()[-1].rows, want[2].rows)
    b.close()
    dg.free()


@pytest.mark.parametrize("cap,project", [(50, None), (50, [0, 2]), (1 << 20, [0, 2])])
def test_rows_that_find_room_in_a_second_pass(cap, project):
    """More rows than the pools of a first run hold: whole rows and distinct
    tuples of two of three vertices, cut to cap or not, come from a second
    pass over the batch, and from one pass once the pools have grown."""
    dg = gs.DeviceGraph(graph_from_triples(120, complete_digraph_triples(120)))
    qs = [paths(3)] * 12
    b = gs.Batch(dg, qs, cap=cap, project=project)
    b.configure(refine_rounds=gs.GS_ROUNDS_NONE)
    w = gs.match(dg, qs[0], cap=cap, project=project, max_refine_rounds=1)
    assert w.count == perm(120, 3)
    for _ in range(2):
        b.run()
        b.finish()
        assert b.counters()["fallback_queries"] == 0
        for r in b.fetch():
            assert (r.status, r.count, r.fingerprint, r.truncated) == (0, w.count, w.fingerprint, w.truncated)
            np.testing.assert_array_equal(r.rows, w.rows)
    b.close()
    dg.free()


@pytest.fixture(scope="module")
def mixed():
    """A graph with hubs, queries of every size that the matcher cuts into
    tasks, and their results from the staged pipeline."""
    g = I.make_graph(30_000, 240_000, seed=51)
    qs = I.make_walk_queries(g, 60, 2, 6, p_bind=0.05, seed=52)
    qs += [I.Query(np.full(q.k, I.ANY, np.uint32), q.vbind, q.esrc, q.edst, q.erel)
           for q in I.make_walk_queries(g, 8, 3, 3, p_bind=0.0, seed=53)]
    dg = gs.DeviceGraph(g)
    want = gs.match_batch(dg, qs, cap=1 << 12, max_refine_rounds=1)
    assert all(w.status == 0 for w in want) and max(w.count for w in want) > 100_000
    yield dg, qs, want
    dg.free()


def runs_with(mixed, copies, **queue):
    dg, qs, want = mixed
    b = gs.Batch(dg, qs * copies, cap=1 << 12)
    b.configure(refine_rounds=gs.GS_ROUNDS_NONE)
    for what, value in queue.items():
        b.set_queue(getattr(gs, what), value)
    for _ in range(3):
        b.run()
        b.finish()
        for i, r in enumerate(b.fetch()):
            w = want[i % len(qs)]
            assert (r.status, r.count, r.fingerprint) == (0, w.count, w.fingerprint), i
            np.testing.assert_array_equal(r.rows, w.rows)
    b.close()


@pytest.mark.parametrize("copies", [1, 20])
@pytest.mark.parametrize("polls", [1, 2, 16])
def test_workers_that_leave_early(mixed, copies, polls):
    """Workers give up waiting after a few polls, while others still cut steps
    into tasks for them: no task is lost."""
    runs_with(mixed, copies, GS_QUEUE_IDLE_POLLS=polls)


def test_queue_settings_are_checked(mixed):
    dg, qs, _ = mixed
    b = gs.Batch(dg, qs)
    with pytest.raises(gs.GSError):  # the staged pipeline
        b.set_queue(gs.GS_QUEUE_IDLE_POLLS, 1)
    b.configure(refine_rounds=gs.GS_ROUNDS_NONE)
    with pytest.raises(gs.GSError):
        b.set_queue(99, 1)
    b.close()


@pytest.mark.parametrize("copies", [1, 20])
@pytest.mark.parametrize("slots", [32, 64, 4096])
def test_ring_of_few_slots(mixed, copies, slots):
    """Many more tasks than the ring has slots: slots are used again within a
    run, and with none free workers do their work themselves."""
    runs_with(mixed, copies, GS_QUEUE_TASKS=slots)


@pytest.mark.parametrize("copies", [1, 20])
@pytest.mark.parametrize("pieces", [1, 2, 64])
def test_few_pieces_of_shared_rows(mixed, copies, pieces):
    """More tasks that start from rows than there are places for rows: a place
    is used again once its task is done, and rows without one stay."""
    runs_with(mixed, copies, GS_QUEUE_PIECES=pieces)


def test_few_of_everything(mixed):
    runs_with(mixed, 3, GS_QUEUE_PIECES=4, GS_QUEUE_TASKS=32, GS_QUEUE_IDLE_POLLS=2)


def test_table_of_row_segments_grows(mixed):
    """More segments of rows than the table holds: the rows of the others come
    from a second pass, and later runs find a larger table."""
    dg, qs, want = mixed
    b = gs.Batch(dg, qs, cap=1 << 12)
    b.configure(refine_rounds=gs.GS_ROUNDS_NONE)
    b.set_queue(gs.GS_QUEUE_SEGMENTS, 8)
    launches = []
    for _ in range(3):
        n0 = b.counters()["kernel_launches"]
        b.run()
        b.finish()
        launches.append(b.counters()["kernel_launches"] - n0)
        assert b.counters()["fallback_queries"] == 0
        for r, w in zip(b.fetch(), want):
            assert (r.status, r.count, r.fingerprint) == (0, w.count, w.fingerprint)
            np.testing.assert_array_equal(r.rows, w.rows)
    assert launches[0] > launches[1] == launches[2]
    b.set_queue(gs.GS_QUEUE_SEGMENTS, 0)  # no more than the table holds by now
    b.run()
    b.finish()
    assert [r.fingerprint for r in b.fetch()] == [w.fingerprint for w in want]
    b.close()


def test_tuned_rounds_reach_batches_made_before():
    """A call after gs_tune_set runs with its settings, also where the call
    takes a batch made before: refinement needs the staged pipeline's pools."""
    import torch
    g = I.make_graph(20_000, 120_000, seed=8)
    qs = I.make_walk_queries(g, 20, 3, 5, p_bind=0.1, seed=8)
    dg = gs.DeviceGraph(g)
    want = gs.match_batch(dg, qs, cap=64)
    free0 = torch.cuda.mem_get_info()[0]
    gs.tune_set(dg, 8, 4)
    got = gs.match_batch(dg, qs, cap=64)
    assert free0 - torch.cuda.mem_get_info()[0] > 16 << 20
    for a, r in zip(want, got):
        assert (r.status, r.count, r.fingerprint) == (0, a.count, a.fingerprint)
        np.testing.assert_array_equal(r.rows, a.rows)
    dg.free()


def test_call_without_memory_drops_the_batches_kept_for_others():
    """Batches kept for later calls go when a call's own finds no memory."""
    import torch
    g = I.make_graph(20_000, 120_000, seed=9)
    qs = I.make_walk_queries(g, 20, 3, 5, p_bind=0.1, seed=9)
    dg = gs.DeviceGraph(g)
    want = gs.match_batch(dg, qs, cap=64)
    gs.match_batch(dg, qs, cap=65)
    gs.debug_fail_alloc(0)
    got = gs.match_batch(dg, qs, cap=66)
    gs.debug_fail_alloc(-1)
    for a, r in zip(want, got):
        assert (r.status, r.count, r.fingerprint) == (0, a.count, a.fingerprint)
        np.testing.assert_array_equal(r.rows[:64], a.rows)
    free0 = torch.cuda.mem_get_info()[0]
    gs.match_batch(dg, qs, cap=64)  # was dropped: its pools are made again
    assert free0 - torch.cuda.mem_get_info()[0] > 16 << 20
    dg.free()
    dg = gs.DeviceGraph(g)
    gs.debug_fail_alloc(0)  # nothing to drop: refused as ever
    with pytest.raises(gs.GSError) as e:
        gs.match_batch(dg, qs, cap=64)
    gs.debug_fail_alloc(-1)
    assert e.value.status == gs.GS_ERR_OOM
    assert [r.count for r in gs.match_batch(dg, qs, cap=64)] == [a.count for a in want]
    dg.free()


def test_bound_on_waits_outlives_new_scan_scratch(mixed):
    """A bound set while the batch runs the one-kernel matcher holds for the
    staged pipeline, whose scans get a scratch of their own."""
    dg, qs, want = mixed
    gs.tune_set(dg, 0, gs.GS_ROUNDS_NONE)  # made without the staged pipeline's pools
    b = gs.Batch(dg, qs, cap=1 << 12)
    gs.tune_set(dg, 0, 0)
    b.set_wait(64, withhold_first_tile=True)
    b.configure(refine_rounds=2)
    b.run()
    with pytest.raises(gs.GSError) as e:
        b.finish()
    assert e.value.status == gs.GS_ERR_TIMEOUT
    b.set_wait(0)
    b.run()
    b.finish()
    for r, w in zip(b.fetch(), want):
        assert (r.status, r.count, r.fingerprint) == (0, w.count, w.fingerprint)
    b.close()


def test_statistics_count_each_launch_once(mixed):
    """Pools that grow after a timed run take the captured graphs with them:
    the run's launches are not counted again."""
    dg, qs, _ = mixed
    b = gs.Batch(dg, qs, cap=1 << 12)
    b.configure(refine_rounds=gs.GS_ROUNDS_NONE)
    b.set_queue(gs.GS_QUEUE_SEGMENTS, 8)
    b.stats_enable(True)
    b.run()
    b.finish()  # a second pass, then a larger table: two runs of the matcher
    assert b.stats()["explore"]["launches"] == 2
    b.run()
    b.finish()
    assert b.stats()["explore"]["launches"] == 3
    b.close()
