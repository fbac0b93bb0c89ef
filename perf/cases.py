"""The label propagation work that programs built on this library do, as cases to time.

Each case is a dict of plain values.  Its graph comes from the seeded recipes
of this repository's workloads, drawn on the device with torch: R-MAT (the
web / social class), planted partitions (the community class, alone, batched
or served) and road-like grids.  A case names the graph, how its entries are
weighted, in which order the vertices are stored and what is done with it:

  "run"         one run on a graph handle that the program keeps (lpa_run);
  "default_run" Graph.run with its defaults: labels and the run's counts;
  "batch"       one run of many graphs packed into one handle (lpa_batch_run);
  "modularity"  Eq. 1 of a labelling on a handle (lpa_modularity);
  "oneshot"     host CSR in, labels out: create, run, copy back, destroy;
  "serve"       a burst of requests through the continuous-batching server.

Labels are whole numbers, so the synchronous modes (whose labels follow from
the graph alone) are compared exactly.  Asynchronous runs depend on the
schedule; they are listed on R-MAT graphs, where the hubs pull nearly every
vertex into one community under any schedule.
"""
import math
import time

import numpy as np
import torch

import paper_2312_08140_gb300 as lpa

TAU, CAP = 0.05, 20                 # the paper's tolerance and sweep cap
INSIDE = 0.8                        # share of a planted partition's edges inside blocks
RMAT_A, RMAT_B, RMAT_C = 0.57, 0.19, 0.19


def listed():
    return [
        # the smallest call: a 10,000-vertex planted partition (10 blocks, mean
        # degree 16), run with the defaults of the Python wrapper
        {"name": "planted10k_default", "do": "default_run", "graph": "planted", "n": 10_000, "blocks": 10,
         "degree": 16.0, "weights": "unit", "mode": "sync", "order": "caller"},
        # a web / social graph of scale 22, bit-exact mode
        {"name": "rmat22_sync", "do": "run", "graph": "rmat", "n": 1 << 22, "edge_factor": 16, "weights": "unit",
         "mode": "sync", "order": "caller"},
        # the same class in the paper's own asynchronous mode, at half the
        # paper-scale graph: the largest case
        {"name": "rmat26_async", "do": "run", "graph": "rmat", "n": 1 << 26, "edge_factor": 14, "weights": "unit",
         "mode": "async", "order": "caller"},
        # vertices stored by degree, the option for repeated runs on one graph
        {"name": "rmat23_async_degree", "do": "run", "graph": "rmat", "n": 1 << 23, "edge_factor": 16,
         "weights": "unit", "mode": "async", "order": "degree"},
        # a road network: degrees of at most a few, integer weights 1..8
        {"name": "grid4096_sync", "do": "run", "graph": "grid", "n": 4096 * 4096, "weights": "int8",
         "mode": "sync", "order": "caller"},
        # real-valued similarities as weights, an odd vertex count
        {"name": "rmat_float_sync", "do": "run", "graph": "rmat", "n": 700_001, "edge_factor": 11,
         "weights": "float", "mode": "sync", "order": "caller"},
        # the pseudo-random tie-break, which scans every vertex in every sweep
        {"name": "planted_nonstrict", "do": "run", "graph": "planted", "n": 300_007, "blocks": 64, "degree": 25.0,
         "weights": "unit", "mode": "sync+nonstrict", "order": "caller"},
        # many graphs in one launch: the batched workload's size distribution
        {"name": "batch256_sync", "do": "batch", "graphs": 256, "n_min": 100, "n_max": 200_000, "weights": "int4",
         "mode": "sync"},
        # many tiny graphs (ego networks): all of them fit the chip at once
        {"name": "batch64_small", "do": "batch", "graphs": 64, "n_min": 100, "n_max": 2_000, "weights": "unit",
         "mode": "sync"},
        # the quality of a labelling, computed after every run
        {"name": "modularity_rmat21", "do": "modularity", "graph": "rmat", "n": 1 << 21, "edge_factor": 16,
         "weights": "unit", "order": "caller"},
        # one graph once: host arrays in, labels back on the host
        {"name": "oneshot_planted200k", "do": "oneshot", "graph": "planted", "n": 200_000, "blocks": 40,
         "degree": 30.0, "weights": "int4", "mode": "sync", "order": "caller"},
        # sixteen requests arriving together at a server
        {"name": "serve_burst16", "do": "serve", "requests": 16, "n_min": 100, "n_max": 20_000,
         "weights": "int4", "mode": "sync"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _most_entries(case):
    """Entries that keep a drawn case below the cost of the largest listed one:
    the modes that scan every vertex in up to CAP sweeps take fewer."""
    most = 3.0e8 if case["weights"] == "unit" else 2.0e7 if case["weights"] == "float" else 1.0e8
    return most if case.get("mode", "sync") in ("sync", "async") else most / 5


def draw(rng):
    do = rng.choice(["run", "run", "run", "run", "default_run", "batch", "batch", "modularity", "oneshot", "serve"])
    if do == "serve":
        return {"do": do, "requests": rng.randint(1, 32), "n_min": 100, "n_max": _log_int(rng, 500, 50_000),
                "weights": rng.choice(["unit", "int4"]), "mode": "sync"}
    if do == "batch":
        case = {"do": do, "graphs": 2, "n_min": 100, "n_max": _log_int(rng, 500, 200_000),
                "weights": rng.choice(["unit", "int4", "int4"]),
                "mode": rng.choice(["sync", "sync", "sync_full", "sync+nonstrict"])}
        case["graphs"] = _log_int(rng, 2, min(256, max(2, int(_most_entries(case) * 2 / work(case)["flops"]))))
        return case
    graph = rng.choice(["rmat", "rmat", "planted", "grid"])
    case = {"do": do, "graph": graph}
    if graph == "rmat":
        big = do in ("run", "modularity")
        case["n"] = _log_int(rng, 2_000, 16_000_000 if big else 500_000)
        case["edge_factor"] = rng.randint(4, 20)
        case["weights"] = rng.choice(["unit", "unit", "unit", "int4", "int1000", "float"])
    elif graph == "planted":
        case["n"] = _log_int(rng, 500, 2_000_000 if do == "run" else 300_000)
        case["blocks"] = rng.randint(2, 64)
        case["degree"] = round(rng.uniform(4.0, 64.0), 2)
        case["weights"] = rng.choice(["unit", "unit", "int4", "int1000", "float"])
    else:
        case["n"] = _log_int(rng, 24, 4096 if do == "run" else 1024) ** 2
        case["weights"] = rng.choice(["unit", "int8", "int8"])
    case["order"] = rng.choice(["caller", "caller", "degree", "shuffle"]) if do == "run" else "caller"
    if do != "modularity":
        case["mode"] = rng.choice(["sync", "sync", "sync_full", "sync+nonstrict"])
        if do == "run" and graph == "rmat" and case["n"] > 1_000_000 and case["weights"] == "unit":
            case["mode"] = rng.choice(["sync", "async"])
    entries = work(case)["flops"]
    if entries > _most_entries(case):
        case["n"] = int(case["n"] * _most_entries(case) / entries)
        if graph == "grid":
            case["n"] = math.isqrt(case["n"]) ** 2
    return case


# ---- graphs ---------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _csr(n, u, v):
    """Symmetric CSR of the undirected edges (u, v): both directions, no
    self-loops, no duplicates, neighbours ascending."""
    keep = u != v
    u, v = u[keep], v[keep]
    keys = torch.cat([u * n + v, v * n + u])
    del u, v, keep
    keys = torch.sort(keys)[0]
    first = torch.ones(keys.shape[0], dtype=torch.bool, device="cuda")
    torch.ne(keys[1:], keys[:-1], out=first[1:])
    keys = keys[first]
    del first
    off = torch.searchsorted(keys, torch.arange(n + 1, device="cuda", dtype=torch.int64) * n)
    keys %= n
    return off, keys.to(torch.int32)


def _rmat_edges(n, edge_factor, gen):
    """edge_factor * n R-MAT draws; pairs with an end past n (a size that is
    not a power of two) are folded back into the range."""
    scale = max(1, (n - 1).bit_length())
    m = edge_factor * n
    u = torch.zeros(m, dtype=torch.int32, device="cuda")
    v = torch.zeros(m, dtype=torch.int32, device="cuda")
    for _ in range(scale):
        r = torch.rand(m, generator=gen, device="cuda")
        down = r >= RMAT_A + RMAT_B
        u.mul_(2).add_(down)
        v.mul_(2).add_(torch.where(down, r >= RMAT_A + RMAT_B + RMAT_C, r >= RMAT_A))
    return torch.where(u < n, u, u - n).long(), torch.where(v < n, v, v - n).long()


def _planted_edges(ns, blocks, degrees, gen):
    """Draws of planted partitions packed back to back: graph g has ns[g]
    vertices in blocks[g] equal blocks and ns[g] * degrees[g] / 2 draws."""
    ms = np.maximum(1, np.round(ns * degrees / 2.0)).astype(np.int64)
    at = np.concatenate([[0], np.cumsum(ms)])
    base = np.concatenate([[0], np.cumsum(ns)])
    m = int(at[-1])
    g = torch.searchsorted(torch.from_numpy(at).cuda(), torch.arange(m, device="cuda"), right=True) - 1
    n_e = torch.from_numpy(ns).cuda()[g]
    b_e = torch.from_numpy(blocks).cuda()[g]
    v0 = torch.from_numpy(base).cuda()[g]
    u = torch.minimum((torch.rand(m, generator=gen, device="cuda", dtype=torch.float64) * n_e).long(), n_e - 1)
    size = torch.div(n_e + b_e - 1, b_e, rounding_mode="floor")
    lo = torch.div(u, size, rounding_mode="floor") * size
    hi = torch.minimum(lo + size, n_e)
    r = torch.rand(m, generator=gen, device="cuda", dtype=torch.float64)
    inside = torch.rand(m, generator=gen, device="cuda") < INSIDE
    v_in = torch.minimum(lo + (r * (hi - lo)).long(), hi - 1)
    v_any = torch.minimum((r * n_e).long(), n_e - 1)
    return u + v0, torch.where(inside, v_in, v_any) + v0


def _grid_edges(side, gen):
    """4-neighbour lattice, 10% of the edges dropped, 0.1% shortcuts."""
    n = side * side
    p = torch.arange(n, device="cuda", dtype=torch.int64)
    right, below = p[p % side != side - 1], p[: n - side]
    u = torch.cat([right, below])
    v = torch.cat([right + 1, below + side])
    keep = torch.rand(u.shape[0], generator=gen, device="cuda") >= 0.1
    k = max(1, n // 1000)
    s = torch.randint(0, n, (2, k), generator=gen, device="cuda")
    return torch.cat([u[keep], s[0]]), torch.cat([v[keep], s[1]])


def _pair_weights(off, idx, kind, seed):
    """Symmetric weights: a hash of the vertex pair, as whole numbers 1..4,
    1..8 or 1..1000, or as real numbers in (0, 1]."""
    if kind == "unit":
        return None
    n = off.shape[0] - 1
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), off[1:] - off[:-1])
    col = idx.long()
    h = torch.minimum(row, col) * 0x9E3779B1 + torch.maximum(row, col) * 0x85EBCA77 + seed * 0x27D4EB2F
    h = h ^ (h >> 29)
    h = h * 0x165667B1
    h = (h ^ (h >> 31)) & 0xFFFFFF
    if kind == "float":
        return (h + 1).to(torch.float32) / float(1 << 24)
    return (h % {"int4": 4, "int8": 8, "int1000": 1000}[kind] + 1).to(torch.float32)


def _single(case, seed):
    """(off int64, idx int32, weights float32 or None) on the device."""
    n, gen = case["n"], _generator(seed)
    if case["graph"] == "rmat":
        u, v = _rmat_edges(n, case["edge_factor"], gen)
    elif case["graph"] == "planted":
        u, v = _planted_edges(np.array([n]), np.array([min(case["blocks"], n)]), np.array([case["degree"]]), gen)
    else:
        u, v = _grid_edges(math.isqrt(n), gen)
    off, idx = _csr(n, u, v)
    return off, idx, _pair_weights(off, idx, case["weights"], seed)


def _packed(case, count, seed):
    """Planted partitions of log-uniform sizes packed back to back: (vertex
    offsets, entry offsets, off, idx with local ids, weights).  The sizes
    belong to the case, the edges to the seed."""
    rng = np.random.default_rng(1000)
    ns = np.round(np.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"]), count))).astype(np.int64)
    blocks = np.minimum(rng.integers(2, 65, count), ns)
    degrees = rng.uniform(4.0, 64.0, count)
    u, v = _planted_edges(ns, blocks, degrees, _generator(seed))
    vtx = np.concatenate([[0], np.cumsum(ns)])
    off, idx = _csr(int(vtx[-1]), u, v)
    w = _pair_weights(off, idx, case["weights"], seed)
    start = torch.from_numpy(vtx).cuda()
    first = torch.repeat_interleave(start[:-1], off[start[1:]] - off[start[:-1]])
    return vtx, off[start].cpu().numpy(), off, (idx - first).to(torch.int32), w


def _some_labels(case, off, idx, seed):
    """A labelling such as a run ends with: for planted partitions the blocks
    with 5% of the vertices still on their own, for grids patches, for R-MAT
    the first neighbour's first neighbour (nearly every vertex ends with a hub)."""
    n = case["n"]
    own = torch.arange(n, device="cuda", dtype=torch.int64)
    if case["graph"] == "rmat":
        deg = off[1:] - off[:-1]
        f = torch.where(deg > 0, idx[torch.clamp(off[:-1], max=idx.shape[0] - 1)].long(), own)
        return f[f].to(torch.int32)
    size = -(-n // min(case["blocks"], n)) if case["graph"] == "planted" else 37
    lab = torch.div(own, size, rounding_mode="floor") * size
    alone = torch.rand(n, generator=_generator(seed + 1), device="cuda") < 0.05
    return torch.where(alone, own, lab).to(torch.int32)


# ---- cases ----------------------------------------------------------------
class _Handle:
    """A library handle that goes with its state."""

    def __init__(self, handle, destroy):
        self.handle, self.destroy = handle, destroy

    def __del__(self):
        self.destroy(self.handle)


_ORDERS = {"caller": 0, "degree": lpa.LPA_REORDER_DEGREE, "shuffle": lpa.LPA_REORDER_SHUFFLE}


def prepare(case, seed):
    do = case["do"]
    state = {"do": do, "mode": case.get("mode")}
    if do == "batch":
        vtx, edge, off, idx, w = _packed(case, case["graphs"], seed)
        state["G"] = case["graphs"]
        state["h"] = _Handle(lpa.lpa_batch_create(case["graphs"], vtx, edge, off, idx, w, lpa.LPA_DEVICE_PTRS),
                             lpa.lpa_batch_destroy)
        state["labels"] = torch.empty(int(vtx[-1]), dtype=torch.int32, device="cuda")
    elif do == "serve":
        vtx, edge, off, idx, w = _packed(case, case["requests"], seed)
        off, idx = off.cpu().numpy(), idx.cpu().numpy()
        w = None if w is None else w.cpu().numpy()
        reqs = []
        for a, b, e, f in zip(vtx[:-1], vtx[1:], edge[:-1], edge[1:]):
            reqs.append((int(b - a), int(f - e), off[a:b + 1] - e, idx[e:f].copy(), None if w is None else w[e:f].copy()))
        state["requests"] = reqs
        state["h"] = _Handle(lpa.lpa_serve_create(4 << 30, 1 << 21, 1 << 26, 64, case["mode"], TAU, CAP),
                             lpa.lpa_serve_destroy)
    else:
        off, idx, w = _single(case, seed)
        n, nnz = case["n"], int(idx.shape[0])
        if do == "oneshot":
            state["csr"] = [None if x is None else x.cpu().pin_memory() for x in (off, idx, w)]
            return state
        if do == "modularity":
            state["labels"] = _some_labels(case, off, idx, seed)
        if do == "default_run":
            state["graph"] = lpa.Graph(off, idx, w)
        else:
            state["h"] = _Handle(lpa.lpa_graph_create(n, nnz, off, idx, w, lpa.LPA_DEVICE_PTRS | _ORDERS[case["order"]]),
                                 lpa.lpa_graph_destroy)
        if do == "run":
            state["labels"] = torch.empty(n, dtype=torch.int32, device="cuda")
    return state


def run(state):
    do = state["do"]
    if do == "run":
        lpa.lpa_run(state["h"].handle, state["mode"], TAU, CAP, state["labels"], info=False)
        return state["labels"]
    if do == "default_run":
        labels, info = state["graph"].run(state["mode"])
        changed = np.zeros(CAP, dtype=np.int64)
        changed[:info["iterations"]] = info["changed"]
        return {"labels": labels, "iterations": info["iterations"], "changed": changed}
    if do == "batch":
        lpa.lpa_batch_run(state["h"].handle, state["G"], state["mode"], TAU, CAP, state["labels"], info=False)
        return state["labels"]
    if do == "modularity":
        return lpa.lpa_modularity(state["h"].handle, state["labels"])
    if do == "oneshot":
        with lpa.Graph(*state["csr"]) as g:
            labels, info = g.run(state["mode"])
            return {"labels": labels.cpu(), "iterations": info["iterations"]}
    server = state["h"].handle
    tickets = [lpa.lpa_serve_submit(server, n, nnz, off, idx, w) for n, nnz, off, idx, w in state["requests"]]
    left = len(tickets)
    while left:
        got = len(lpa.lpa_serve_poll(server))
        left -= got
        if left and not got:
            time.sleep(2e-5)
    out = []
    for t, r in zip(tickets, state["requests"]):
        out.append(lpa.lpa_serve_fetch(server, t, r[0])[0])
        lpa.lpa_serve_release(server, t)
    return np.concatenate(out)


def work(case):
    """The CSR read once and the labels (or Q) written once; one addition per
    entry.  Entry counts are the recipes' expected ones before duplicates go."""
    per_weight = {"unit": 0, "int4": 1, "int8": 1, "int1000": 4, "float": 4}[case["weights"]]
    if "graph" in case:
        n = case["n"]
        nnz = n * {"rmat": 2 * case.get("edge_factor", 0), "planted": case.get("degree", 0), "grid": 3.6}[case["graph"]]
    else:
        count = case.get("graphs", case.get("requests"))
        lo, hi = case["n_min"], case["n_max"]
        n = count * (hi - lo) / math.log(hi / lo)
        nnz = 34.0 * n
    return {"bytes": 8.0 * n + (4.0 + per_weight) * nnz + 4.0 * n, "flops": float(nnz)}


def exact(case, seed):
    """Modularity (Eq. 1) in 64 bits; labels are whole numbers."""
    if case["do"] != "modularity":
        return None
    off, idx, w = _single(case, seed)
    n = case["n"]
    lab = _some_labels(case, off, idx, seed).long()
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), off[1:] - off[:-1])
    w = torch.ones(idx.shape[0], dtype=torch.float64, device="cuda") if w is None else w.double()
    same = lab[row] == lab[idx.long()]
    total = w.sum()
    k = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, row, w)
    community = torch.bincount(lab, weights=k, minlength=n)
    q = (w * same).sum() / total - (community * community).sum() / (total * total)
    return float(q)
