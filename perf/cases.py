"""The library's work as its users have it done, as cases that can be timed.

Every case goes through the public binding (``paper_2009_12457_gb300``). The graphs are
the families that the repository's generators, tests and benchmark use -- R-MAT
(.57, .19, .19, .05), G(n, m) and capped Chung-Lu with degree exponent 2.1 -- drawn here
on the GPU so that inputs are quick to make. As there, a generated CSR keeps duplicate
entries and self-loops as drawn; removing them is the method's own first step.

Forms of a case (``form``):
  step     create a handle from a CSR, count, destroy: what a one-off count of a new graph costs
  recount  count again on a handle that holds its plan: what a resident graph costs per query
  batch    one union handle for many small graphs: create, count every graph, destroy
  handles  one bbtc_count_batch call over many resident handles: a batch of the server
  stream   count under a device budget, the blocks streamed from pinned host memory
"""
import math

import numpy as np
import torch

import paper_2009_12457_gb300 as bb

RMAT_A, RMAT_B, RMAT_C = 0.57, 0.19, 0.19
FRIENDSTER_N, FRIENDSTER_PAIRS = 65_608_366, 1_806_067_135


def listed():
    return [
        # a cold request of the server at its smallest scale: a host CSR, one create + count + destroy;
        # launches and host work are all there is
        {"name": "request_s10", "form": "step", "family": "rmat", "scale": 10, "pairs": 16 << 10,
         "symmetric": True, "host": True, "p": 0, "kernel": "auto"},
        # the README's call with no promise about the input: an edge list as drawn, each edge under one
        # endpoint only, rows unsorted, duplicates kept (the general preparation)
        {"name": "step_general_s20", "form": "step", "family": "rmat", "scale": 20, "pairs": 16 << 20,
         "symmetric": False, "one_sided": True, "host": False, "p": 0, "kernel": "auto"},
        # a social-network-shaped graph resident on the device, symmetric and sorted: the ordinary step
        {"name": "step_sym_s21", "form": "step", "family": "rmat", "scale": 21, "pairs": 16 << 21,
         "symmetric": True, "host": False, "p": 0, "kernel": "auto"},
        # the benchmark's default shape (Friendster-shaped Chung-Lu, p = 1) at a quarter of its size
        {"name": "step_chunglu_quarter", "form": "step", "family": "chunglu", "n": FRIENDSTER_N // 4,
         "pairs": FRIENDSTER_PAIRS // 4, "symmetric": True, "host": False, "p": 1, "kernel": "auto"},
        # a repeated query on a small resident graph (the parity configuration's size)
        {"name": "recount_s14", "form": "recount", "family": "rmat", "scale": 14, "pairs": 16 << 14,
         "p": 0, "kernel": "auto", "output": "total"},
        # the counting kernel on a large skewed graph with the paper's per-task counts at p = 4
        {"name": "recount_s22_tasks", "form": "recount", "family": "rmat", "scale": 22, "pairs": 16 << 22,
         "p": 4, "kernel": "auto", "output": "task"},
        # bbTC-Intersect (Alg. 5) chosen by the caller
        {"name": "recount_s18_intersect", "form": "recount", "family": "rmat", "scale": 18,
         "pairs": 16 << 18, "p": 4, "kernel": "intersect", "output": "total"},
        # triangles at every vertex (clustering coefficients), left on the device
        {"name": "vertex_s20", "form": "recount", "family": "rmat", "scale": 20, "pairs": 16 << 20,
         "p": 0, "kernel": "auto", "output": "vertex"},
        # the support of every edge (the input of k-truss), left on the device
        {"name": "edge_s19", "form": "recount", "family": "rmat", "scale": 19, "pairs": 16 << 19,
         "p": 0, "kernel": "auto", "output": "edge"},
        # many independent graphs at once, sizes as in the batched workload of the benchmark
        {"name": "batch_256", "form": "batch", "graphs": 256, "low": 1_000, "high": 2_000_000,
         "p": 1, "kernel": "auto"},
        # what a server's worker sends when requests of mixed sizes have queued up
        {"name": "handles_64", "form": "handles", "graphs": 64, "scale_low": 10, "scale_high": 18,
         "p": 0, "kernel": "auto"},
        # a graph counted under a device budget, its blocks kept in pinned host memory
        {"name": "stream_s20", "form": "stream", "family": "rmat", "scale": 20, "pairs": 16 << 20,
         "p": 8, "kernel": "auto", "budget": 192 << 20},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, lo, hi):
    """A family and sizes with lo to hi pairs."""
    family = rng.choice(["rmat", "rmat", "chunglu", "gnm"])
    pairs = _log_uniform(rng, lo, hi)
    if family == "rmat":
        scale = max(6, int(round(math.log2(pairs / rng.uniform(8, 32)))))
        return {"family": family, "scale": scale, "pairs": pairs}
    return {"family": family, "n": max(64, int(2 * pairs / rng.uniform(8, 64)) | 1), "pairs": pairs}


def draw(rng):
    form = rng.choice(["step", "step", "step", "recount", "recount", "recount", "batch", "handles", "stream"])
    kernel = rng.choice(["auto", "auto", "auto", "hashmap", "intersect"])
    p = rng.choice([0, 0, 1, 2, 4, 8, 16])
    if form == "batch":
        low = _log_uniform(rng, 200, 20_000)
        return {"form": form, "graphs": _log_uniform(rng, 2, 512), "low": low,
                "high": low * rng.randint(2, 60), "p": rng.choice([0, 1, 2]), "kernel": "auto"}
    if form == "handles":
        lo = rng.randint(8, 13)
        return {"form": form, "graphs": _log_uniform(rng, 2, 128), "scale_low": lo,
                "scale_high": lo + rng.randint(1, 4), "p": rng.choice([0, 0, 1, 4]), "kernel": "auto"}
    if form == "stream":
        g = _draw_graph(rng, 1 << 20, 24 << 20)
        # the in-edge and column blocks take about 20 bytes an edge: a budget near two thirds of that
        return {"form": form, **g, "p": rng.choice([8, 12, 16]), "kernel": "auto",
                "budget": g["pairs"] * 14 + (8 << 20)}
    if form == "step":
        symmetric = rng.random() < 0.6
        g = _draw_graph(rng, 2_000, (64 if symmetric else 24) << 20)
        return {"form": form, **g, "symmetric": symmetric, "one_sided": not symmetric and rng.random() < 0.5,
                "host": g["pairs"] < (1 << 18) and rng.random() < 0.5, "p": p,
                "kernel": kernel if kernel != "intersect" or g["pairs"] < (8 << 20) else "auto"}
    output = rng.choice(["total", "total", "task", "vertex", "edge"])
    g = _draw_graph(rng, 2_000, (64 if output in ("total", "task") and kernel != "intersect" else 16) << 20)
    return {"form": form, **g, "p": p or (4 if output == "task" else 0), "kernel": kernel, "output": output}


# ------------------------------------------------------------------ inputs

def _rmat_pairs(scale, pairs, gen, dev):
    src = torch.zeros(pairs, dtype=torch.int64, device=dev)
    dst = torch.zeros(pairs, dtype=torch.int64, device=dev)
    for _ in range(scale):
        r = torch.rand(pairs, device=dev, generator=gen)
        low = (r >= RMAT_A + RMAT_B)  # the lower half of the matrix
        right = ((r >= RMAT_A) & ~low) | (r >= RMAT_A + RMAT_B + RMAT_C)
        src = src * 2 + low
        dst = dst * 2 + right
    return 1 << scale, src, dst


def _gnm_pairs(n, pairs, gen, dev):
    return n, torch.randint(n, (pairs,), device=dev, generator=gen), \
        torch.randint(n, (pairs,), device=dev, generator=gen)


def _chunglu_pairs(n, pairs, gen, dev, exponent=2.1, cap=5000.0):
    base = torch.arange(1, n + 1, dtype=torch.float64, device=dev).pow(-1.0 / (exponent - 1.0))
    cap = min(cap, math.sqrt(2.0 * pairs))
    lo, hi = 0.0, float(2 * pairs)
    for _ in range(50):  # the scale for which the capped weights sum to 2 * pairs
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if float((base * mid).clamp_(max=cap).sum()) < 2.0 * pairs else (lo, mid)
    # whole-number weights: their running sums, hence the graph, are the same on every run
    cum = (base * hi).clamp_(max=cap).mul_(1 << 20).long().cumsum(0)
    total = int(cum[-1])
    ends = []
    for _ in range(2):
        parts = []
        for at in range(0, pairs, 1 << 26):
            r = torch.randint(total, (min(1 << 26, pairs - at),), device=dev, generator=gen)
            parts.append(torch.searchsorted(cum, r, right=True, out_int32=True))
        ends.append(torch.cat(parts))
    return n, ends[0], ends[1]


def _pairs(case, gen, dev):
    if case["family"] == "rmat":
        return _rmat_pairs(case["scale"], case["pairs"], gen, dev)
    if case["family"] == "gnm":
        return _gnm_pairs(case["n"], case["pairs"], gen, dev)
    return _chunglu_pairs(case["n"], case["pairs"], gen, dev)


def _rowptr(rows, n):
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=rows.device)
    torch.cumsum(torch.bincount(rows, minlength=n), 0, out=rowptr[1:])
    return rowptr


def _symmetric_csr(n, src, dst):
    """Every pair under both endpoints, rows ascending, duplicates and self-loops as drawn."""
    src, dst = src.long(), dst.long()
    key = torch.cat([src * n + dst, dst * n + src])
    del src, dst
    key = torch.sort(key).values
    rowptr = _rowptr(torch.div(key, n, rounding_mode="floor"), n)
    return n, rowptr, (key % n).int()


def _one_sided_csr(n, src, dst):
    """Every pair under its first endpoint only, in the order drawn."""
    rows, order = torch.sort(src.long(), stable=True)
    return n, _rowptr(rows, n), dst[order].int()


def _graph_csr(case, gen, dev):
    pairs = _pairs(case, gen, dev)
    return _one_sided_csr(*pairs) if case.get("one_sided") else _symmetric_csr(*pairs)


def _batch_csr(case, seed, gen, dev):
    """The union of case["graphs"] symmetric graphs: even ones G(n, m), odd ones R-MAT."""
    rng = np.random.default_rng(seed)
    ns, parts = [0], []
    for g in range(case["graphs"]):
        pairs = int(round(math.exp(rng.uniform(math.log(case["low"]), math.log(case["high"])))))
        if g % 2 == 0:
            n, src, dst = _gnm_pairs(max(2, int(2 * pairs / rng.uniform(8, 64))), pairs, gen, dev)
        else:
            scale = max(1, int(round(math.log2(pairs / rng.uniform(8, 32)))))
            n, src, dst = _rmat_pairs(scale, pairs, gen, dev)
        parts.append((src + ns[-1], dst + ns[-1]))
        ns.append(ns[-1] + n)
    voff = np.asarray(ns, dtype=np.int64)
    n, rowptr, colidx = _symmetric_csr(ns[-1], torch.cat([s for s, _ in parts]), torch.cat([d for _, d in parts]))
    first = torch.from_numpy(voff).to(dev)
    graph = torch.searchsorted(first, colidx.long(), right=True) - 1
    return voff, rowptr, (colidx - first[graph]).int()


def _handle_case(case, g):
    """Graph g of a case of many handles: scales in turn, edge factor 16."""
    span = case["scale_high"] - case["scale_low"] + 1
    scale = case["scale_low"] + g % span
    return {"family": "rmat", "scale": scale, "pairs": 16 << scale}


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev).manual_seed(seed)
    form, state = case["form"], {"case": case}
    if form == "batch":
        state["voff"], state["rowptr"], state["colidx"] = _batch_csr(case, seed, gen, dev)
    elif form == "handles":
        graphs = []
        for g in range(case["graphs"]):
            n, rowptr, colidx = _graph_csr(_handle_case(case, g), gen, dev)
            torch.cuda.synchronize()
            graphs.append(bb.Graph(n, rowptr, colidx, symmetric=True))
            bb.bbtc_graph_plan(graphs[-1].handle, bb.make_opts(p=case["p"], kernel=case["kernel"]))
        state["graphs"] = graphs
        state["opts"] = bb.make_opts(p=case["p"], kernel=case["kernel"])
    else:
        n, rowptr, colidx = _graph_csr(case, gen, dev)
        torch.cuda.synchronize()
        if form == "step":
            state["n"] = n
            if case["host"]:
                rowptr, colidx = rowptr.cpu().numpy(), colidx.cpu().numpy()
            state["rowptr"], state["colidx"] = rowptr, colidx
        else:
            graph = bb.Graph(n, rowptr, colidx, symmetric=True)
            state["graph"] = graph
            output = case.get("output", "total")
            opts = {"p": case["p"], "kernel": case["kernel"]}
            if output == "vertex":
                state["out"] = opts["per_vertex_out"] = torch.zeros(n, dtype=torch.int64, device=dev)
            elif output == "edge":
                # room for every pair drawn; the simple graph's edges fill the front of it
                state["out"] = opts["per_edge_out"] = torch.zeros(case["pairs"], dtype=torch.int32, device=dev)
            if form == "stream":
                opts["device_budget_bytes"] = case["budget"]
                state["opts"] = bb.make_opts(**opts)
                bb.bbtc_count(graph.handle, state["opts"])  # the plan's blocks move to the host once
            else:
                bb.bbtc_graph_plan(graph.handle, bb.make_opts(p=case["p"], kernel=case["kernel"]))
                state["opts"] = bb.make_opts(**opts)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()  # the library allocates beside torch
    return state


# -------------------------------------------------------------------- a pass

def run(state):
    case = state["case"]
    form = case["form"]
    if form == "step":
        with bb.Graph(state["n"], state["rowptr"], state["colidx"], symmetric=case["symmetric"]) as g:
            return {"total": g.count(p=case["p"], kernel=case["kernel"])}
    if form == "batch":
        with bb.BatchGraph(vertex_offsets=state["voff"], rowptr=state["rowptr"], colidx=state["colidx"],
                           symmetric=True) as g:
            out = g.count(p=case["p"], kernel=case["kernel"], per_graph=True)
            return {"total": out["total"], "graph": out["per_graph"].astype(np.int64)}
    if form == "handles":
        counts, _ = bb.bbtc_count_batch([g.handle for g in state["graphs"]], state["opts"])
        return {"graph": counts.astype(np.int64)}
    if case.get("output") == "task":
        out = state["graph"].count(p=case["p"], kernel=case["kernel"], per_task=True)
        return {"total": out["total"], "task": out["per_task"].astype(np.int64)}
    total = bb.bbtc_count(state["graph"].handle, state["opts"])
    return {"total": total, "each": state["out"]} if "out" in state else {"total": total}


def _sizes(case):
    """(vertices, pairs) of a case."""
    if case["form"] == "batch":
        mean = (case["high"] - case["low"]) / math.log(case["high"] / case["low"])
        return case["graphs"] * mean / 18, case["graphs"] * mean
    if case["form"] == "handles":
        graphs = [_handle_case(case, g) for g in range(case["graphs"])]
        return sum(1 << g["scale"] for g in graphs), sum(g["pairs"] for g in graphs)
    return (1 << case["scale"] if case["family"] == "rmat" else case["n"]), case["pairs"]


def work(case):
    """Bytes only: the input CSR read once (the oriented graph for a handle that is counted again; its
    blocks and in-edges under a budget) and the outputs written once. How many memberships are tested
    depends on the graph's degrees and on the algorithm, so no operations are stated."""
    n, pairs = _sizes(case)
    if case["form"] in ("step", "batch"):
        entries = pairs if case.get("one_sided") else 2 * pairs
        return {"bytes": 8.0 * (n + 1) + 4.0 * entries + 8.0 * case.get("graphs", 1), "flops": 0.0}
    if case["form"] == "stream":
        return {"bytes": 20.0 * pairs + 4.0 * n * (case["p"] + 1) / 2, "flops": 0.0}
    each = {"vertex": 8.0 * n, "edge": 4.0 * pairs}.get(case.get("output"), 8.0)
    return {"bytes": 8.0 * (n + 1) + 4.0 * pairs + each, "flops": 0.0}


# ----------------------------------------------------------- the exact values

EXACT_WEDGES = 600_000_000  # beyond this many open pairs the enumeration takes too long


def _oriented(n, rows, cols):
    """The simple graph of the entries, oriented from lower to higher (degree, id): rowptr and
    ascending rows by position, and the vertex at each position."""
    keep = rows != cols
    a, b = torch.minimum(rows, cols)[keep], torch.maximum(rows, cols)[keep]
    key = torch.unique(a * n + b)
    a, b = torch.div(key, n, rounding_mode="floor"), key % n
    deg = torch.bincount(a, minlength=n) + torch.bincount(b, minlength=n)
    perm = torch.sort(deg, stable=True).indices
    rank = torch.empty_like(perm)
    rank[perm] = torch.arange(n, device=perm.device)
    ra, rb = rank[a], rank[b]
    key = torch.sort(torch.minimum(ra, rb) * n + torch.maximum(ra, rb)).values
    u = torch.div(key, n, rounding_mode="floor")
    return _rowptr(u, n), u, key % n, key, perm


def _triangles(n, rowptr, u, v, key):
    """Chunks of (edge uv, edge uw, edge vw) positions, one row per triangle; None when too many."""
    m = key.numel()
    left = rowptr[u + 1] - torch.arange(m, device=u.device) - 1
    ends = torch.cumsum(left, 0)
    if m == 0 or int(ends[-1]) == 0:
        return []
    if int(ends[-1]) > EXACT_WEDGES:
        return None
    found, at = [], 0
    while at < m:
        base = int(ends[at - 1]) if at else 0
        to = max(at + 1, int(torch.searchsorted(ends, base + (1 << 25), right=True)))
        e = torch.repeat_interleave(torch.arange(at, to, device=u.device), left[at:to])
        if e.numel():
            f = e + 1 + torch.arange(e.numel(), device=u.device) - (ends[e] - left[e] - base)
            want = v[e] * n + v[f]
            g = torch.searchsorted(key, want).clamp_(max=m - 1)
            hit = key[g] == want
            found.append(torch.stack([e[hit], f[hit], g[hit]]))
        at = to
    return found


def _exact_one(n, rowptr_in, colidx):
    rows = torch.repeat_interleave(torch.arange(n, device=rowptr_in.device), rowptr_in.diff())
    rowptr, u, v, key, perm = _oriented(n, rows, colidx.long())
    return rowptr, u, v, perm, _triangles(n, rowptr, u, v, key)


def exact(case, seed):
    if case["form"] in ("batch", "handles"):
        n, pairs = _sizes(case)
        if pairs > 8_000_000:
            return None
    elif _sizes(case)[1] > 40_000_000:
        return None
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev).manual_seed(seed)
    if case["form"] == "handles":
        counts = []
        for g in range(case["graphs"]):
            found = _exact_one(*_graph_csr(_handle_case(case, g), gen, dev))[4]
            if found is None:
                return None
            counts.append(sum(t.shape[1] for t in found))
        return {"graph": np.asarray(counts, dtype=np.int64)}
    if case["form"] == "batch":
        voff, rowptr, colidx = _batch_csr(case, seed, gen, dev)
        first = torch.from_numpy(voff).to(dev)
        rows = torch.repeat_interleave(torch.arange(int(voff[-1]), device=dev), rowptr.diff())
        graph = torch.searchsorted(first, rows, right=True) - 1
        n, colidx = int(voff[-1]), colidx.long() + first[graph]
    else:
        n, rowptr, colidx = _graph_csr(case, gen, dev)
    rowptr, u, v, perm, found = _exact_one(n, rowptr, colidx)
    if found is None:
        return None
    total = sum(t.shape[1] for t in found)
    if case["form"] == "batch":
        counts = np.zeros(case["graphs"], dtype=np.int64)
        for t in found:
            g = torch.searchsorted(first, perm[u[t[0]]], right=True) - 1
            counts += torch.bincount(g, minlength=case["graphs"]).cpu().numpy()
        return {"total": total, "graph": counts}
    output = case.get("output", "total")
    if output == "vertex":
        each = torch.zeros(n, dtype=torch.int64, device=dev)
        for t in found:
            for x in (u[t[0]], v[t[0]], v[t[1]]):
                each += torch.bincount(perm[x], minlength=n)
        return {"total": total, "each": each}
    if output == "edge":
        each = torch.zeros(case["pairs"], dtype=torch.int64, device=dev)
        for t in found:
            for x in t:
                each += torch.bincount(x, minlength=each.numel())
        return {"total": total, "each": each.int()}
    if output == "task":
        p, m = case["p"], u.numel()
        target = torch.tensor([-(-i * m // p) for i in range(p)], device=dev)
        cuts = torch.searchsorted(rowptr, target)
        cuts[0] = 0
        index = {(i, j, k): 0 for i in range(p) for j in range(i, p) for k in range(j, p)}
        table = torch.zeros(p * p * p, dtype=torch.int64, device=dev)
        for x, (i, j, k) in enumerate(index):
            table[(i * p + j) * p + k] = x
        each = torch.zeros(len(index), dtype=torch.int64, device=dev)
        for t in found:
            i, j, k = (torch.searchsorted(cuts, x, right=True) - 1 for x in (u[t[0]], v[t[0]], v[t[1]]))
            each += torch.bincount(table[(i * p + j) * p + k], minlength=len(index))
        return {"total": total, "task": each.cpu().numpy()}
    return {"total": total}
