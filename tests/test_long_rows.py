"""Synchronous rows that a lane cannot sort (more than 64 slots): shared out over
idle warps on small graphs, scanned by the warp that meets them on larger ones,
by a kernel of their own where the weights wait in shared memory (fp32; integers
whose label and weight leave 32 bits), and with them the key layouts of the lane
kernel at the numbers of vertices where they change.

Labels and counts must equal the CPU oracle's.  Every weight is a multiple of 1/4
below 2^17 and every row's sum stays below 2^24, so the sums are exact.
"""
import numpy as np
import pytest

import lpa_inputs as L
import oracle as O

pytestmark = pytest.mark.gpu

TOP = {"byte": 4, "byte255": 255, "word": 131_071, "quarter": 40}       # largest weight (quarter: of 1/4)


@pytest.fixture(scope="module")
def lpa():
    import paper_2312_08140_gb300 as m
    m.load()
    return m


def weights(g, kind, top=None):
    """Symmetric: a hash of the vertex pair; the largest weight occurs."""
    top = top or TOP.get(kind)
    if kind == "unit":
        return None
    row = np.repeat(np.arange(g.n), np.diff(g.off))
    pair = (np.minimum(row, g.idx).astype(np.uint64) * np.uint64(g.n) + np.maximum(row, g.idx).astype(np.uint64))
    w = 1 + ((pair * np.uint64(0x9E3779B97F4A7C15)) >> np.uint64(33)).astype(np.int64) % top
    w[row + g.idx == row[0] + g.idx[0]] = top
    return w.astype(np.float32) / (4 if kind == "quarter" else 1)


def around_64(n, seed=1, low=20, step=25):
    """Communities of 200 with degrees around twice low .. low + step: rows on both
    sides of 64 entries, starting anywhere in a 16-byte vector."""
    rng = np.random.default_rng(seed)
    src = np.repeat(np.arange(n), low + np.arange(n) % step)
    dst = (src // 200) * 200 + rng.integers(0, 200, src.shape[0])
    far = rng.random(src.shape[0]) < 0.3
    dst[far] = rng.integers(0, n, int(far.sum()))
    return L.from_edges(n, src, np.minimum(dst, n - 1))


def check(lpa, g, w, sweeps=4):
    import torch
    off, idx = torch.from_numpy(g.off).cuda(), torch.from_numpy(g.idx).cuda()
    wd = None if w is None else torch.from_numpy(w).cuda()
    out = torch.empty(g.n, dtype=torch.int32, device="cuda")
    h = lpa.lpa_graph_create(g.n, g.nnz, off, idx, wd, lpa.LPA_DEVICE_PTRS)
    try:
        for mode, ns in (("sync", False), ("sync+nonstrict", True)):
            ref, it, changed = O.lpa_sync(g.off, g.idx, w, 0.0, sweeps, nonstrict=ns)
            for profiled in (False, True):                   # captured (kernels side by side) and host-launched
                if profiled:
                    info, _ = lpa.lpa_run_profiled(h, mode, 0.0, sweeps, out)
                else:
                    info = lpa.lpa_run(h, mode, 0.0, sweeps, out)
                got = out.cpu().numpy()
                assert list(info.changed[:info.iterations]) == changed.tolist()[:it]
                assert np.array_equal(got, ref), (mode, np.flatnonzero(got != ref)[:5])
    finally:
        lpa.lpa_graph_destroy(h)


# 17-bit weights fill 32 bits with the labels of 2^15 - 1 vertices
@pytest.mark.parametrize("n", [900, 32_767, 32_768, 50_000])
@pytest.mark.parametrize("kind", ["unit", "byte", "word", "quarter"])
def test_rows_around_64_entries(lpa, kind, n):
    g = around_64(n)
    deg = np.diff(g.off)
    assert (deg > 64).sum() > n // 8 and (deg <= 61).sum() > n // 8
    check(lpa, g, weights(g, kind))


def test_byte_weights_beyond_the_packed_labels(lpa):
    """2^24 vertices, 8-bit weights: the key holds the place in the row."""
    g0 = around_64(6_000, seed=5)
    n = 1 << 24
    off = np.concatenate([g0.off, np.full(n - g0.n, g0.nnz, dtype=np.int64)])
    g = L.Graph(off, g0.idx, None)
    check(lpa, g, weights(g, "byte255"), sweeps=3)


def test_batch_of_fp32_graphs_that_end_apart(lpa):
    """Longer rows of graphs that are done keep their labels."""
    import torch
    graphs = [around_64(n, seed=n, low=lo) for n, lo in ((300, 34), (2_000, 20), (5_000, 30), (1_000, 5))]
    graphs = [L.Graph(g.off, g.idx, weights(g, "quarter")) for g in graphs]
    vtx, edge, off, idx, w = L.pack(graphs)
    local = (idx - np.repeat(vtx[:-1], np.diff(edge))).astype(np.int32)
    h = lpa.lpa_batch_create(len(graphs), vtx, edge, off, local, w)
    try:
        out = torch.empty(int(vtx[-1]), dtype=torch.int32, device="cuda")
        infos = lpa.lpa_batch_run(h, len(graphs), "sync", 0.05, 20, out)
        got = out.cpu().numpy()
        ends = set()
        for k, g in enumerate(graphs):
            ref, it, changed = O.lpa_sync(g.off, g.idx, g.w, 0.05, 20)
            ends.add(it)
            assert infos[k].iterations == it and list(infos[k].changed[:it]) == changed.tolist()[:it]
            assert np.array_equal(got[vtx[k]:vtx[k + 1]], ref)
        assert len(ends) > 1
    finally:
        lpa.lpa_batch_destroy(h)
