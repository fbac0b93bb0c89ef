"""The majority kernels (lpa_sweep_majority.cu) on a graph that one label comes
to dominate: R-MAT 18, whose block bins hold more than the 4 M entries that the
kernels ask for.  The oracle's labels after each sweep tell which sweeps begin
with a label above the 5/8 of the entries that the search asks for: there the
kernels settle most rows, and leave those that the label does not decide.

Every weight kind, both tie-breaks, with and without marks.  Weights are multiples
of 1/4 with row sums below 2^22, so fp32 and integer sums are exact and labels and
counts must equal the oracle's.
"""
import numpy as np
import pytest

import lpa_inputs as L
import oracle as O
from async_bounds import assert_local_max_bound
from test_long_rows import weights

TOP = {"unit": None, "byte": 4, "word": 300, "quarter": 40}
SEARCH = 4 << 20            # entries that the block bins, and a frontier, must hold
SWEEPS = 7


@pytest.fixture(scope="module")
def rmat18():
    return L.rmat(18, 16, seed=3)


def _led_sweeps(g, w, nonstrict):
    """Per sweep 1..SWEEPS the oracle's labels and dN, and the sweeps (from 2 on)
    whose frontier, the neighbours of the vertices that changed, holds SEARCH
    entries while one label holds 0.66 of all (a sample of 4096 entries has a
    standard deviation of 0.0075): [(sweep, share)]."""
    deg = np.diff(g.off)
    row = np.repeat(np.arange(g.n), deg)
    labels, dN, led, prev = [], [], [], np.arange(g.n)
    for t in range(1, SWEEPS + 1):
        lab = O.lpa_sync(g.off, g.idx, w, 0.0, t, nonstrict=nonstrict)[0]
        moved = lab != prev
        near = np.zeros(g.n, dtype=bool)
        near[g.idx[moved[row]]] = True
        share = float(np.bincount(lab[g.idx]).max()) / g.nnz
        if share >= 0.66 and t < SWEEPS and int(deg[near & (deg > 4)].sum()) >= SEARCH:
            led.append((t + 1, share))
        labels.append(lab)
        dN.append(int(moved.sum()))
        prev = lab
    return labels, dN, led


def _weights(g, kind):
    return None if kind == "unit" else weights(g, kind, TOP[kind])


@pytest.mark.gpu
@pytest.mark.parametrize("nonstrict", [False, True], ids=["strict", "nonstrict"])
@pytest.mark.parametrize("kind", list(TOP))
def test_dominated_sweeps_match_the_oracle(rmat18, kind, nonstrict):
    import torch

    import paper_2312_08140_gb300 as lpa
    g = rmat18
    deg = np.diff(g.off)
    assert deg[deg > 128].sum() >= SEARCH
    w = _weights(g, kind)
    labels, dN, led = _led_sweeps(g, w, nonstrict)
    assert led, "no sweep of this case is dominated"
    assert any(share < 0.99 for _, share in led)              # some rows are not settled
    wd = None if w is None else torch.from_numpy(w).cuda()
    out = torch.empty(g.n, dtype=torch.int32, device="cuda")
    h = lpa.lpa_graph_create(g.n, g.nnz, torch.from_numpy(g.off).cuda(), torch.from_numpy(g.idx).cuda(), wd,
                             lpa.LPA_DEVICE_PTRS)
    try:
        for mode in (["sync+nonstrict"] if nonstrict else ["sync", "sync_full"]):
            for t in sorted({led[0][0], led[-1][0], SWEEPS}):
                info = lpa.lpa_run(h, mode, 0.0, t, out)
                got = out.cpu().numpy()
                assert list(info.changed[:t]) == dN[:t]
                assert np.array_equal(got, labels[t - 1]), (mode, t, int((got != labels[t - 1]).sum()))
        lpa.lpa_run_profiled(h, "sync+nonstrict" if nonstrict else "sync", 0.0, led[0][0], out)
        assert np.array_equal(out.cpu().numpy(), labels[led[0][0] - 1])
    finally:
        lpa.lpa_graph_destroy(h)


@pytest.mark.gpu
@pytest.mark.parametrize("kind", list(TOP))
def test_dominated_asynchronous_runs_end_at_local_maxima(rmat18, kind):
    """A settled row has the label that outweighs the rest of it: at a tolerance of
    1/1000 at most as many vertices are off their local argmax."""
    import torch

    import paper_2312_08140_gb300 as lpa
    g = rmat18
    gw = L.Graph(g.off, g.idx, _weights(g, kind))
    wd = None if gw.w is None else torch.from_numpy(gw.w).cuda()
    with lpa.Graph(torch.from_numpy(g.off).cuda(), torch.from_numpy(g.idx).cuda(), wd) as G:
        labels, info = G.run("async", 0.001, 40)
    labels = labels.cpu().numpy()
    assert info["exit_reason"] == 0
    assert O.count_labels_outside_component(g.off, g.idx, labels) == 0
    assert_local_max_bound(gw, labels, info, 0.001, f"async {kind}")
