"""Which vertices a synchronous sweep scans once little changes: the rules that
choose between scanning every vertex and a frontier affect speed only, so the
labels and change counts stay the oracle's, and the entries that lpa_run reports
as scanned tell which of the two a sweep took.
"""
import numpy as np
import pytest

import lpa_inputs as L
import oracle as O


def _trace(g, sweeps):
    """Per sweep t = 1..sweeps of the oracle: dN, entries of the changed vertices,
    entries of their neighbours (the next sweep's frontier); and the last labels."""
    deg = np.diff(g.off)
    row = np.repeat(np.arange(g.n), deg)
    prev, out = np.arange(g.n), []
    for t in range(1, sweeps + 1):
        lab = O.lpa_sync(g.off, g.idx, g.w, 0.0, t)[0]
        moved = lab != prev
        front = np.zeros(g.n, dtype=bool)
        front[g.idx[moved[row]]] = True
        out.append((int(moved.sum()), int(deg[moved].sum()), int(deg[front].sum())))
        prev = lab
    return out, prev


@pytest.fixture(scope="module")
def cycle():
    """R-MAT 16: from the fourth sweep on 65 vertices go back and forth."""
    g = L.rmat(16, 8, seed=1)
    return g, *_trace(g, 14)


def test_the_cycle_graph_is_one(cycle):
    g, trace, _ = cycle
    assert trace[1][1] > g.nnz / 10                          # sweep 2 changes a good part of the entries
    assert all(0 < dn and ent < g.nnz / 1000 and front < g.nnz / 500 for dn, ent, front in trace[3:])


@pytest.mark.gpu
def test_small_graph_takes_frontiers_in_a_long_tail(cycle):
    import torch

    import paper_2312_08140_gb300 as lpa
    g, trace, ref = cycle
    with lpa.Graph(torch.from_numpy(g.off).cuda(), torch.from_numpy(g.idx).cuda()) as G:
        labels, info = G.run("sync", 0.0, len(trace))
    assert np.array_equal(labels.cpu().numpy(), ref)
    assert info["changed"] == [dn for dn, _, _ in trace]
    # sweep 4 changes less than a thousandth, so sweep 5 marks and sweep 6 on
    # scans the neighbours of the vertices that changed
    assert info["scanned"][5:] == [front for _, _, front in trace[4:-1]]
    assert info["scanned"][1] == info["scanned"][2] == g.nnz


@pytest.mark.gpu
def test_serving_through_a_tail_and_back(cycle):
    """A request in its tail (frontiers) is joined by others (every vertex again):
    each result is the oracle's."""
    import time

    import paper_2312_08140_gb300 as lpa
    g, trace, _ = cycle
    cap = 60
    others = [L.planted_partition(3000, 6, seed=2), L.rmat(12, 16, seed=9)]
    srv = lpa.lpa_serve_create(1 << 30, 1 << 18, 1 << 23, 8, "sync", 0.0, cap)
    try:
        todo = {lpa.lpa_serve_submit(srv, g.n, g.nnz, g.off, g.idx, g.w): g}
        for q in others:
            before = lpa.lpa_serve_stats(srv)["cycles"]
            t0 = time.time()
            while lpa.lpa_serve_stats(srv)["cycles"] < before + 12 and time.time() - t0 < 0.02:
                time.sleep(0.0002)
            todo[lpa.lpa_serve_submit(srv, q.n, q.nnz, q.off, q.idx, q.w)] = q
        done, t0 = set(), time.time()
        while len(done) < len(todo):
            done.update(lpa.lpa_serve_poll(srv))
            assert time.time() - t0 < 60, "serving did not finish"
            time.sleep(0.0005)
        for ticket, q in todo.items():
            labels, info = lpa.lpa_serve_fetch(srv, ticket, q.n)
            ref, it, changed = O.lpa_sync(q.off, q.idx, q.w, 0.0, cap)
            assert info.iterations == it and list(info.changed[:it]) == changed.tolist()[:it]
            assert np.array_equal(labels, ref)
    finally:
        lpa.lpa_serve_destroy(srv)
