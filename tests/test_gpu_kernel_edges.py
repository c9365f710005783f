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
