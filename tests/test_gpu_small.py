"""Graphs prepared in one kernel (up to 1,024 vertices) against the oracle: every
input form, the sizes around its limits, and its error cases."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2009_12457_gb300 as bb

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def one_sided(n, src, dst):
    order = np.argsort(src, kind="stable")
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(src, minlength=n), out=rowptr[1:])
    return n, rowptr, dst[order].astype(np.int32)


@pytest.mark.parametrize("n,pairs", [(1, 3), (2, 5), (31, 60), (33, 400), (1000, 20_000),
                                     (1023, 900), (1024, 30_000), (1024, 65_536), (1024, 65_537),
                                     (1025, 30_000)])
def test_small_graph_matches_oracle(n, pairs):
    _, src, dst = graphgen.gnm_pairs(n, pairs, n + pairs)
    sym = graphgen.pairs_to_csr(n, src, dst)  # duplicates and self-loops as drawn
    ref = oracle.bbtc(*sym, p=3, want_per_vertex=True)
    for graph, symmetric in ((sym, True), (sym, False), (one_sided(n, src, dst), False)):
        with bb.Graph(*graph, symmetric=symmetric) as g:
            o = g.oriented()
            assert np.array_equal(o["rowptr"], ref["rowptr"])
            assert np.array_equal(o["colidx"], ref["colidx"])
            assert np.array_equal(o["perm"], ref["perm"])
            i = g.info()
            assert i["m"] == len(ref["colidx"])
            assert i["dplus_max"] == int(np.diff(ref["rowptr"]).max())
            out = g.count(p=3, per_task=True, per_vertex=True)
            assert out["total"] == ref["total"]
            assert np.array_equal(out["per_task"], ref["per_task"])
            assert np.array_equal(out["per_vertex"], ref["per_vertex"])


def test_small_graph_rejects_malformed_input():
    rp = np.array([0, 2, 4, 6], dtype=np.int64)
    ci = np.array([1, 2, 0, 2, 0, 1], dtype=np.int32)
    for bad_rp, bad_ci in (([0, 4, 2, 6], ci), ([1, 2, 4, 6], ci), (rp, [1, 2, 0, 3, 0, 1]),
                           (rp, [1, 2, 0, -1, 0, 1])):
        for symmetric in (False, True):
            with pytest.raises(bb.BbtcError) as e:
                bb.Graph(3, np.asarray(bad_rp, dtype=np.int64), np.asarray(bad_ci, dtype=np.int32),
                         symmetric=symmetric)
            assert e.value.status == 1


@pytest.mark.parametrize("n,pairs", [(1025, 40_000), (5000, 3), (70_000, 300_000)])
def test_general_input_with_duplicates(n, pairs):
    # beyond one CTA: distinct edges by hashing; every entry listed up to four times
    _, src, dst = graphgen.gnm_pairs(n, pairs, 3 * n + pairs)
    src, dst = np.concatenate([src, dst, src]), np.concatenate([dst, src, dst])
    graph = one_sided(n, src, dst)
    ref = oracle.bbtc(*graphgen.pairs_to_csr(n, src, dst), p=1)
    with bb.Graph(*graph) as g:
        o = g.oriented()
        assert np.array_equal(o["rowptr"], ref["rowptr"])
        assert np.array_equal(o["colidx"], ref["colidx"])
        assert np.array_equal(o["perm"], ref["perm"])
        assert g.count() == ref["total"]


def test_a_vertex_joined_to_all_others():
    # every key shares one endpoint, and every degree addition one counter
    n = 200_000
    rp = np.zeros(n + 1, dtype=np.int64)
    rp[1:] = n - 1
    with bb.Graph(n, rp, np.arange(1, n, dtype=np.int32)) as g:
        i = g.info()
        assert i["m"] == n - 1 and i["deg_max"] == n - 1 and i["dplus_max"] == 1
        assert g.count() == 0


def test_an_edge_listed_too_often_for_its_bucket():
    # its copies share one bucket of 2,048: the keys are sorted instead
    n = 3000
    _, src, dst = graphgen.gnm_pairs(n, 20_000, 77)
    src = np.concatenate([src, np.full(100_000, src[0])])
    dst = np.concatenate([dst, np.full(100_000, dst[0])])
    graph = one_sided(n, src, dst)
    ref = oracle.bbtc(*graphgen.pairs_to_csr(n, src, dst), p=1)
    with bb.Graph(*graph) as g:
        o = g.oriented()
        assert np.array_equal(o["rowptr"], ref["rowptr"])
        assert np.array_equal(o["colidx"], ref["colidx"])
        assert g.count() == ref["total"]


@pytest.mark.parametrize("row,value", [(1024, -1), (1024, -5), (1, -8), (2047, -(1 << 40)),
                                       (1500, 1 << 40)])
def test_interior_row_pointers_out_of_range_are_refused(row, value):
    # beyond one CTA; the error is known to the host only after the entries have been moved
    n, rp, ci = graphgen.gnm(2048, 30_000, 5)
    rp = rp.copy()
    rp[row] = value
    for symmetric in (True, False):
        with pytest.raises(bb.BbtcError) as e:
            bb.Graph(n, rp, ci, symmetric=symmetric)
        assert e.value.status == 1
    with bb.Graph(*graphgen.gnm(2048, 30_000, 5), symmetric=True) as g:  # all is well after
        assert g.count() == oracle.bbtc(*graphgen.gnm(2048, 30_000, 5), p=1)["total"]


def descending(graph):
    n, rp, ci = graph
    row = np.repeat(np.arange(n), np.diff(rp))
    return n, rp, ci[np.lexsort((-ci.astype(np.int64), row))]


@pytest.mark.parametrize("n,pairs", [(1100, 1500), (1100, 3000), (20_000, 300_000)])
@pytest.mark.parametrize("form", ["both", "repeated", "upward"])
def test_symmetric_input_with_unsorted_rows(n, pairs, form):
    # "repeated": one edge overflows its bucket; "upward": every edge under its lower
    # endpoint only, twice the keys that symmetric input gives (more than room, at 1,100
    # vertices, or more than the buckets hold)
    _, src, dst = graphgen.gnm_pairs(n, pairs, n + pairs)
    if form == "repeated":
        src, dst = np.append(src, np.full(50_000, 3)), np.append(dst, np.full(50_000, 5))
    sym = graphgen.pairs_to_csr(n, src.astype(np.int32), dst.astype(np.int32))
    ref = oracle.bbtc(*sym, p=1)
    if form == "upward":
        sym = one_sided(n, np.minimum(src, dst), np.maximum(src, dst))
    with bb.Graph(*descending(sym), symmetric=True) as g:
        o = g.oriented()
        assert np.array_equal(o["rowptr"], ref["rowptr"])
        assert np.array_equal(o["colidx"], ref["colidx"])
        assert np.array_equal(o["perm"], ref["perm"])
        assert g.count() == ref["total"]


def test_symmetric_batch_with_unsorted_rows():
    graphs = [graphgen.rmat(11, 12, 61), graphgen.gnm(3000, 9000, 62), graphgen.gnm(7, 4, 63)]
    want = [oracle.bbtc(*g, p=1)["total"] for g in graphs]
    with bb.BatchGraph([descending(g) for g in graphs], symmetric=True) as u:
        assert u.count(p=1, per_graph=True)["per_graph"].tolist() == want


@pytest.mark.parametrize("n,pairs", [(1500, 20_000), (20_000, 400_000), (300_000, 900_000)])
@pytest.mark.parametrize("form", ["upward", "less_one_up", "less_one_down", "less_half"])
def test_edges_listed_under_one_endpoint_though_said_to_be_symmetric(n, pairs, form):
    # rows sorted: the entries u < v are the edges, whatever the others say, and no
    # in-degree may be taken from a degree that misses some
    sym = graphgen.gnm(n, pairs, n)
    rp, ci = sym[1], sym[2]
    row, rng = np.repeat(np.arange(n), np.diff(rp)), np.random.default_rng(n)
    keep = np.ones(len(ci), dtype=bool)
    if form == "upward":
        keep = row <= ci
    elif form == "less_half":
        keep = (row <= ci) | (rng.random(len(ci)) < 0.5)
    else:
        u, v = (min, max) if form == "less_one_up" else (max, min)
        e = int(np.flatnonzero(row != ci)[len(ci) // 2])
        a, b = u(row[e], ci[e]), v(row[e], ci[e])
        keep = ~((row == a) & (ci == b))
    src, dst = row[keep], ci[keep]
    up = src < dst
    ref = oracle.bbtc(*graphgen.pairs_to_csr(n, src[up].astype(np.int32), dst[up].astype(np.int32)), p=1)
    with bb.Graph(*one_sided(n, src, dst), symmetric=True) as g:
        assert np.array_equal(g.oriented()["colidx"], ref["colidx"])
        for p in (1, 2):
            assert g.count(p=p) == ref["total"], p
