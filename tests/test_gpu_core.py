"""The dense core (bitmap rows of the top positions) against the oracle, at the
sizes where its layout changes: a graph that is all core, one vertex more than
that, a core cut at a group of columns, and parts that start inside a group."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2009_12457_gb300 as bb

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

GRAPHS = {
    "one_quad": lambda: graphgen.gnm(100, 2500, 3),                # all core, one quad of columns
    "quad_edge": lambda: graphgen.gnm(129, 4000, 4),               # one vertex in a second quad
    "two_groups": lambda: graphgen.gnm(4097, 150_000, 5),          # one vertex in a second group
    "all_core_most": lambda: graphgen.gnm(16384, 500_000, 6),      # the largest all-core graph
    "part_core": lambda: graphgen.rmat(15, 24, 7),                 # hubs in the core, lists below
    "core_edge": lambda: graphgen.chunglu(16385, 2.1, 2000.0, 1_000_000, 500_000, 8),
    "thin": lambda: graphgen.chunglu(16384, 2.1, 900.0, 60_000, 30_000, 9),  # few edges: a smaller core
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_core_counts_per_task(name):
    n, rp, ci = GRAPHS[name]()
    with bb.Graph(n, rp, ci, symmetric=True) as g:
        for p in (1, 3, 16, 40):
            ref = oracle.bbtc(n, rp, ci, p=p)
            out = g.count(p=p, per_task=True)
            assert out["total"] == ref["total"], p
            assert np.array_equal(out["per_task"], ref["per_task"]), p
            # the lists alone count the same
            assert g.count(p=p, kernel="intersect") == ref["total"], p


def test_core_of_a_batch_per_graph_and_of_handles():
    graphs = [graphgen.rmat(12, 16, 31), graphgen.gnm(300, 9000, 32), graphgen.rmat(15, 16, 33),
              graphgen.gnm(50, 40, 34), graphgen.gnm(9000, 200_000, 35)]
    want = np.array([oracle.bbtc(*g, p=1)["total"] for g in graphs], dtype=np.uint64)
    with bb.BatchGraph(graphs, symmetric=True) as u:
        for p in (1, 2, 5):
            out = u.count(p=p, per_graph=True)
            assert np.array_equal(out["per_graph"], want), p
            assert out["total"] == int(want.sum())
    hs = [bb.Graph(*g, symmetric=True) for g in graphs]
    try:
        for p in (0, 1, 4, 20):
            counts, stats = bb.bbtc_count_batch([h.handle for h in hs], bb.make_opts(p=p))
            assert not np.any(stats) and np.array_equal(counts, want), p
    finally:
        for h in hs:
            h.close()


def test_core_items_of_only_one_handle_of_a_batch():
    # a handle's core triangles are its own, also when no other handle has a core
    def complete(n):
        rp = np.arange(n + 1, dtype=np.int64) * (n - 1)
        ci = np.array([[v for v in range(n) if v != u] for u in range(n)], dtype=np.int32).ravel()
        return n, rp, ci

    edgeless = (7, np.zeros(8, dtype=np.int64), np.zeros(0, dtype=np.int32))
    two_edges = (3, np.array([0, 1, 3, 4], dtype=np.int64), np.array([1, 0, 2, 1], dtype=np.int32))
    sparse = graphgen.gnm(20_000, 60_000, 41)  # lists alone: no source has 64 core neighbours
    hubs = graphgen.rmat(15, 16, 33)
    for graphs in ([edgeless, complete(100)], [complete(100), edgeless],
                   [two_edges, edgeless, complete(65)], [sparse, hubs], [hubs, sparse, two_edges]):
        want = np.array([oracle.bbtc(*g, p=1)["total"] for g in graphs], dtype=np.uint64)
        hs = [bb.Graph(*g, symmetric=True) for g in graphs]
        try:
            handles = [h.handle for h in hs]
            for p in (0, 3):
                counts, stats = bb.bbtc_count_batch(handles, bb.make_opts(p=p))
                assert not np.any(stats) and np.array_equal(counts, want), p
                counts, stats = bb.bbtc_count_batch(handles[:1] + [None] + handles[1:],
                                                    bb.make_opts(p=p))
                assert stats[1] == 1 and not np.any(np.delete(stats, 1))
                assert np.array_equal(np.delete(counts, 1), want), p
        finally:
            for h in hs:
                h.close()


def test_a_core_with_more_items_than_its_list_holds():
    # the complete graph of 20,000 vertices has 1.33 M core items, the list room for 2^20:
    # the sources without room are counted by lists. Rows of every length, made on the device
    n = 20_000
    ids = torch.arange(n, dtype=torch.int32, device="cuda")
    ci = ids[None, :].expand(n, n)[ids[None, :] != ids[:, None]]
    rp = torch.arange(n + 1, dtype=torch.int64, device="cuda") * (n - 1)
    torch.cuda.synchronize()  # the library reads them on its own stream
    with bb.Graph(n, rp, ci, symmetric=True) as g:
        del ids, ci, rp
        assert g.count(p=1) == n * (n - 1) * (n - 2) // 6
        assert g.count(p=1, per_task=True)["per_task"].tolist() == [n * (n - 1) * (n - 2) // 6]
    torch.cuda.empty_cache()
