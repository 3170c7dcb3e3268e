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
