"""Kernels at the edges of their size and value ranges, against the oracle (every value a
whole number, compared exactly)."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import paper_1708_06127_gb300 as vc
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    vc.build()


def ring_graph(n, seed, wlo, whi):
    """A connected graph of exactly n vertices: a random one and a ring over it."""
    g = gg.er(n, min(10, (n - 1) / 2), seed)
    src = np.repeat(np.arange(n), np.diff(g.offsets))
    pairs = {(int(a), int(b)) for a, b in zip(src, g.adj) if a < b}
    pairs |= {(min(v, (v + 1) % n), max(v, (v + 1) % n)) for v in range(n) if n > 2 or v == 0}
    w = np.random.default_rng(seed).integers(wlo, whi + 1, len(pairs))
    return gg.from_edges(n, [(a, b, int(x)) for (a, b), x in zip(sorted(pairs), w)])


@pytest.mark.parametrize("wlo,whi", [(1, 1), (1, 9), (1 << 20, 1 << 30)])
@pytest.mark.parametrize("n", [2, 3, 31, 33, 512, 513, 2047, 8193, 16384, 16385])
def test_exact_round_sizes_and_weights(n, wlo, whi):
    """Rounds by a block: 32-bit values (bound x entries below 2^31), 64-bit values, and
    global-memory state above 16,384 vertices."""
    g = ring_graph(n, 7 + n, wlo, whi)
    h = oracle.as_csr64(g.offsets, g.adj, g.w)
    dmin = int(oracle.degrees(h).min())
    d = vc.viecut_graph_upload(h.offsets, h.adj, h.w)
    try:
        for lam in sorted({dmin, max(1, dmin // 3)}):
            got, ch = vc.viecut_step_noi_round(d, lam)
            ref, cnt = oracle.noi_round(h, lam)
            assert np.array_equal(got, ref), lam
            assert ch == (1 if cnt > 0 else 0)
    finally:
        vc.viecut_graph_free(d)


@pytest.mark.parametrize("wlo,whi", [(1, 1), (1, 9), (1 << 20, 1 << 30)])
@pytest.mark.parametrize("n", [2, 5, 33, 150, 151, 400, 512, 600])
def test_exact_step_whole(n, wlo, whi):
    """The whole exact step: first round on the lists, later ones on matrices in shared or
    global memory."""
    g = ring_graph(n, 90 + n, wlo, whi)
    cut, bits = vc.exact_min_cut(g.offsets, g.adj, g.w)
    ref = oracle.viecut(g.offsets, g.adj, g.w, seed=1, lp_iters=0, n0=g.n)
    assert cut == ref.cut and np.array_equal(bits, ref.side_bits)


def test_exact_step_parallel_entries():
    """Parallel entries are summed by the first round and by the matrix."""
    base = H.random_graph(60, 0.2, 4, wmax=3)
    edges = []
    for v in range(base.n):
        for e in range(base.offsets[v], base.offsets[v + 1]):
            if base.adj[e] > v:
                edges += [(v, int(base.adj[e]), int(base.w[e])), (v, int(base.adj[e]), 2)]
    g = gg.from_edges(base.n, edges)
    cut, bits = vc.exact_min_cut(g.offsets, g.adj, g.w)
    ref = oracle.viecut(g.offsets, g.adj, g.w, seed=1, lp_iters=0, n0=g.n)
    assert cut == ref.cut and np.array_equal(bits, ref.side_bits)


def test_exact_step_batch_classes():
    """A batch whose graphs fall into every size class of the sparse rounds and the dense
    step, light and heavy weights together."""
    graphs = [ring_graph(n, n, *w) for n in (2, 40, 512, 513, 2048, 2049, 4097, 8193, 17000)
              for w in ((1, 4), (1 << 20, 1 << 30))]
    with vc.Batch([(g.offsets, g.adj, g.w) for g in graphs], n0=1 << 40) as b:
        cuts, bits = b.run(3, 2)
    for g, cut, side in zip(graphs, cuts, bits):
        ref = oracle.viecut(g.offsets, g.adj, g.w, seed=3, lp_iters=2, n0=1 << 40)
        assert cut == ref.cut and np.array_equal(side, ref.side_bits), g.n


def check_contract(G, labels):
    """One contraction against the oracle's, element by element; returns the coarse graph."""
    labels = np.ascontiguousarray(labels, np.int32)
    d = vc.viecut_graph_upload(G.offsets, G.adj, G.w)
    out = None
    try:
        out, cid = vc.viecut_step_contract(d, labels)
        off, adj, w = vc.viecut_graph_download(out)
        ref, rcid = oracle.contract(G, labels)
        assert np.array_equal(cid, rcid)
        assert np.array_equal(off, ref.offsets)
        assert np.array_equal(adj, ref.adj)
        assert np.array_equal(w, ref.w)
        return ref
    finally:
        vc.viecut_graph_free(d)
        if out is not None:
            vc.viecut_graph_free(out)


@pytest.mark.parametrize("n,deg,clusters", [
    (2000, 300, 2), (2000, 300, 31), (2000, 300, 33), (2000, 300, 255), (2000, 300, 257),  # the table
    (40, 20, 5), (300, 3, 9),                      # of few pairs; one lane per list
    (40000, 4, 2), (70000, 4, 2), (70000, 4, 40),  # few sums: up to 65,536 pairs, above, 64 per sum
    (700, 300, 690)])                              # more sums than pairs would fill
def test_contract_to_few_clusters(n, deg, clusters):
    """The merge in a table and both sides of the line where it is taken; one vertex in ten
    with weights of 0, which leave an entry of weight 0."""
    g = gg.er(n, deg, 3 + clusters, 1, 100)
    G = oracle.as_csr64(g.offsets, g.adj, g.w)
    labels = np.random.default_rng(clusters).integers(0, clusters, n)
    check_contract(G, labels)
    src = np.repeat(np.arange(n), np.diff(g.offsets))
    check_contract(oracle.CsrGraph(G.offsets, G.adj, np.where((src % 10 == 0) | (G.adj % 10 == 0), 0, G.w)), labels)
