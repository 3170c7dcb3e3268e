"""The resident count (flat in-edges) against the oracle: short runs that share a
window, runs that cross windows and work items, lists too wide for a bitmap,
each lookup form, and attribution to few and to many parts."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2009_12457_gb300 as bb

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

GRAPHS = {
    "short_runs": lambda: graphgen.gnm(60_000, 150_000, 11),   # in-degrees of 0 to about 8
    "medium_runs": lambda: graphgen.gnm(20_000, 400_000, 12),  # about 20 in-edges a run
    "hubs": lambda: graphgen.rmat(16, 12, 13),
    "wide_lists": lambda: graphgen.chunglu(300_000, 2.1, 3000.0, 2_400_000, 1_200_000, 14),
}


@pytest.mark.parametrize("kernel", ["auto", "hashmap", "intersect"])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_flat_counts_per_task(name, kernel):
    n, rp, ci = GRAPHS[name]()
    prep = oracle.prepare(n, rp, ci)
    with bb.Graph(n, rp, ci, symmetric=True) as g:
        for p in (2, 4, 7):
            ref = oracle.bbtc(n, rp, ci, p=p, prep=prep)
            for chunk in (0, 1, 37):
                out = g.count(p=p, kernel=kernel, per_task=True, chunk=chunk)
                assert out["total"] == ref["total"], (p, chunk)
                assert np.array_equal(out["per_task"], ref["per_task"]), (p, chunk)
            assert g.count(p=p, kernel=kernel) == ref["total"], p


def test_total_and_task_by_task_counts_alternate_on_one_plan():
    n, rp, ci = graphgen.rmat(13, 16, 15)
    ref = oracle.bbtc(n, rp, ci, p=3, want_per_vertex=True)
    with bb.Graph(n, rp, ci) as g:
        for _ in range(2):
            assert g.count(p=3) == ref["total"]
            out = g.count(p=3, per_vertex=True, per_task=True)
            assert np.array_equal(out["per_vertex"], ref["per_vertex"])
            assert np.array_equal(out["per_task"], ref["per_task"])
        assert g.count(p=3, device_budget_bytes=64 << 20) == ref["total"]
        assert g.count(p=3) == ref["total"]


@pytest.mark.parametrize("kernel", ["auto", "intersect"])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_vertex_and_edge_outputs(name, kernel):
    n, rp, ci = GRAPHS[name]()
    prep = oracle.prepare(n, rp, ci)
    ref = oracle.bbtc(n, rp, ci, p=2, prep=prep, want_per_vertex=True)
    support = oracle.edge_support(n, prep["rowptr"], prep["colidx"])
    with bb.Graph(n, rp, ci, symmetric=True) as g:
        for chunk in (0, 5, 200_000):  # short items, and runs longer than a 16-bit counter holds
            out = g.count(p=2, kernel=kernel, per_vertex=True, chunk=chunk)
            assert out["total"] == ref["total"]
            assert np.array_equal(out["per_vertex"], ref["per_vertex"]), chunk
            out = g.count(p=2, kernel=kernel, per_edge=True, per_task=True, chunk=chunk)
            assert np.array_equal(out["per_edge"], support), chunk
            assert np.array_equal(out["per_task"], ref["per_task"])
        out = g.count(p=2, kernel=kernel, per_vertex=True, per_edge=True)
        assert out["total"] == ref["total"]
        assert np.array_equal(out["per_vertex"], ref["per_vertex"])
        assert np.array_equal(out["per_edge"], support)


def test_one_destination_with_more_in_edges_than_a_counter_holds():
    # 70,000 sources share the edge (a, b): support beyond 16 bits on one entry of one list
    k = 70_000
    src = np.concatenate([np.arange(k), np.arange(k), [k]])
    dst = np.concatenate([np.full(k, k), np.full(k, k + 1), [k + 1]])
    n, rp, ci = graphgen.pairs_to_csr(k + 2, src.astype(np.int32), dst.astype(np.int32))
    with bb.Graph(n, rp, ci, symmetric=True) as g:
        out = g.count(p=1, per_vertex=True, chunk=100_000)
        assert out["total"] == k
        assert int(out["per_vertex"][k]) == k and int(out["per_vertex"][k + 1]) == k
        sup = g.count(p=1, per_edge=True, chunk=100_000)["per_edge"]
        assert int(sup.max()) == k and int((sup == 1).sum()) == 2 * k


def test_work_items_of_every_kind_of_count():
    # without a core (INTERSECT) every in-edge is in a work item of `chunk` of them
    n, rp, ci = graphgen.rmat(14, 16, 15)
    with bb.Graph(n, rp, ci, symmetric=True) as g:
        m, chunk = g.info()["m"], 64
        items = -(-m // chunk)
        kw = dict(p=3, kernel="intersect", chunk=chunk)
        for more, want in (({"per_vertex": True}, items), ({}, items), ({"per_edge": True}, items),
                           ({"per_vertex": True, "per_task": True}, 2 * items),
                           ({"device_budget_bytes": 64 << 20}, items), ({}, items)):
            g.count(**kw, **more)
            assert g.timings()["work_items"] == want, more
        g.count(**kw, per_task_cycles=True)  # task by task: every task's in-edges
        assert g.timings()["work_items"] >= items
        g.count(p=3)
        assert g.timings()["work_items"] > 0
