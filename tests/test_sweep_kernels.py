"""The synchronous lane-per-vertex sweep, the majority kernels and the
modularity kernels at the sizes where their parts meet: row lengths around the
32 and 64 slots of a sorted half and a lane's row, rows that start anywhere in
a 16-byte vector, every key layout (label; label and weight; label and place;
none), rows that a dominating label settles or just does not, rows listed for
the sliced modularity pass, and communities beyond a block's cached ones.

Labels and counts must equal the CPU oracle's.  Every weight here is a multiple
of 1/4 below 2^17 and every row's sum stays below 2^23, so fp32 and integer sums
are exact in any order.
"""
import numpy as np
import pytest

import lpa_inputs as L
import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lpa():
    import paper_2312_08140_gb300 as m
    m.load()
    return m


def _mixed_degrees(n=2600, top=150, seed=3):
    """Symmetric graph with duplicates and self-loops whose degrees run from 1
    to beyond `top`."""
    rng = np.random.default_rng(seed)
    want = 1 + np.arange(n) % top
    src = np.repeat(np.arange(n), (want + 1) // 2)
    dst = rng.integers(0, n, src.shape[0])
    near = rng.random(src.shape[0]) < 0.6                       # communities of 100
    dst[near] = (src[near] // 100) * 100 + rng.integers(0, 100, int(near.sum()))
    return L.from_edges(n, src, np.minimum(dst, n - 1), dedup=False, drop_self=False)


def _weights(g, kind, seed=5):
    rng = np.random.default_rng(seed)
    if kind == "unit":
        return None
    row = np.repeat(np.arange(g.n), np.diff(g.off))
    pair = np.minimum(row, g.idx).astype(np.int64) * g.n + np.maximum(row, g.idx)
    draw = rng.integers(0, 1 << 31, 4096)[pair % 4093]
    top = {"byte": 5, "byte255": 256, "word": 100_000, "quarter": 40}[kind]
    w = (draw % top).astype(np.float32)
    return w / 4 if kind == "quarter" else w


def _gpu(lpa, g, w, mode, iters, cfg=None, borrow_offset=None):
    import torch
    off, idx = torch.from_numpy(g.off).cuda(), torch.from_numpy(g.idx).cuda()
    flags, wd = lpa.LPA_DEVICE_PTRS, None if w is None else torch.from_numpy(w).cuda()
    if borrow_offset is not None:
        buf = torch.zeros(g.nnz + 8, dtype=torch.float32, device="cuda")
        buf[borrow_offset:borrow_offset + g.nnz] = wd
        wd = buf[borrow_offset:borrow_offset + g.nnz]
        flags |= lpa.LPA_BORROW
    h = lpa.lpa_graph_create(g.n, g.nnz, off, idx, wd, flags)
    try:
        if cfg:
            lpa.lpa_graph_set_config(h, lpa.LpaConfig(*cfg))
        out = torch.full((g.n,), -7, dtype=torch.int32, device="cuda")
        info = lpa.lpa_run(h, mode, 0.0, iters, out)
        return out.cpu().numpy(), list(info.changed[:info.iterations])
    finally:
        lpa.lpa_graph_destroy(h)


@pytest.mark.parametrize("cfg", [None, (1, 16, 256, 1024, 500), (8, 256, 512, 2048, 1001)], ids=["default", "narrow", "wide"])
@pytest.mark.parametrize("kind", ["unit", "byte", "byte255", "word", "quarter"])
def test_lane_sweep_row_lengths(lpa, kind, cfg):
    g = _mixed_degrees()
    w = _weights(g, kind)
    for mode, ns in (("sync", False), ("sync_full+nonstrict", True)):
        ref, it, changed = O.lpa_sync(g.off, g.idx, w, 0.0, 5, nonstrict=ns)
        got, ch = _gpu(lpa, g, w, mode, 5, cfg)
        assert ch == changed.tolist()[:it]
        assert np.array_equal(got, ref), (kind, mode, np.flatnonzero(got != ref)[:5])


@pytest.mark.parametrize("offset", [0, 1, 4])
def test_lane_sweep_borrowed_weights_at_any_alignment(lpa, offset):
    g = _mixed_degrees(n=700)
    w = _weights(g, "quarter")
    ref, it, changed = O.lpa_sync(g.off, g.idx, w, 0.0, 5)
    got, ch = _gpu(lpa, g, w, "sync", 5, borrow_offset=offset)
    assert ch == changed.tolist()[:it] and np.array_equal(got, ref)


def _hubs(n=40_000, hubs=1500, spread=3000, seed=11):
    """Hub rows of about `spread` + entries (over 4 M entries in the last bin),
    leaves that see about a hundred hubs each, and pairs of leaves."""
    rng = np.random.default_rng(seed)
    src = np.repeat(np.arange(hubs), spread)
    dst = rng.integers(hubs, n, src.shape[0])
    a = rng.integers(hubs, n, 3 * n)
    b = np.minimum(a + rng.integers(1, 4, a.shape[0]), n - 1)
    return L.from_edges(n, np.concatenate([src, a]), np.concatenate([dst, b]))


@pytest.mark.parametrize("kind", ["unit", "byte", "quarter"])
def test_majority_rows_match_the_oracle(lpa, kind):
    g = _hubs()
    w = _weights(g, kind)
    deg = np.diff(g.off)
    assert deg[deg > 2048].sum() >= 4 << 20
    for mode, ns in (("sync", False), ("sync_full+nonstrict", True)):
        ref, it, changed = O.lpa_sync(g.off, g.idx, w, 0.0, 4, nonstrict=ns)
        got, ch = _gpu(lpa, g, w, mode, 4)
        assert ch == changed.tolist()[:it]
        assert np.array_equal(got, ref), (kind, mode, int((got != ref).sum()))
    labels, _ = _gpu(lpa, g, w, "async", 4)
    assert O.count_labels_outside_component(g.off, g.idx, labels) == 0


@pytest.mark.parametrize("n,hub", [(900, 0), (40_000, 0), (40_000, 3_001), (100_000, 90_001), (400_000, 9_000)])
def test_modularity_rows_and_communities(lpa, n, hub):
    """Q within 1e-10: sums of up to 2^21 fp64 terms carry a relative error below
    2^21 x 2^-53 = 2.4e-10 only if every rounding fell one way; both terms of Q
    are at most 1 and the roundings of a tree of partial sums (at most 2^9 terms
    in a row on either side) stay below 2^-44 = 6e-14 each."""
    import torch
    rng = np.random.default_rng(n)
    src, dst = rng.integers(0, n, 2 * n), rng.integers(0, n, 2 * n)
    if hub:
        src = np.concatenate([src, np.full(hub, 17)])
        dst = np.concatenate([dst, rng.integers(0, n, hub)])
    g = L.from_edges(n, src, dst, dedup=False, drop_self=False)
    labels = np.where(rng.random(n) < 0.5, 3, rng.integers(0, n, n)).astype(np.int32)
    for kind in ("unit", "quarter"):
        w = _weights(g, kind)
        ref = O.modularity(g.off, g.idx, w, labels)
        off, idx = torch.from_numpy(g.off).cuda(), torch.from_numpy(g.idx).cuda()
        wd = None if w is None else torch.from_numpy(w).cuda()
        lab = torch.from_numpy(labels).cuda()
        for flags in (0, lpa.LPA_REORDER_DEGREE):
            h = lpa.lpa_graph_create(g.n, g.nnz, off, idx, wd, lpa.LPA_DEVICE_PTRS | flags)
            try:
                assert abs(lpa.lpa_modularity(h, lab) - ref) <= 1e-10
            finally:
                lpa.lpa_graph_destroy(h)
        odd = torch.zeros(g.nnz + 1, dtype=torch.int32, device="cuda")
        odd[1:] = idx                                            # ids off the 16-byte boundary
        assert abs(lpa.lpa_modularity_noalloc(g.n, g.nnz, off, odd[1:], wd, lab) - ref) <= 1e-10
