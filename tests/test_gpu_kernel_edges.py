"""Kernels at the edges of their size and value ranges, against the oracle (every value a
whole number, compared exactly)."""
import heapq

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


def any_round(G, lam):
    """A round in whole numbers of any size (maximum-adjacency order, ties to the smallest id):
    every vertex's smallest joined id."""
    r, seen, parent = [0] * G.n, [False] * G.n, list(range(G.n))

    def find(x):
        while parent[x] != x:
            parent[x] = x = parent[parent[x]]
        return x

    off, adj, w = G.offsets.tolist(), G.adj.tolist(), G.w.tolist()
    heap = [(0, v) for v in range(G.n)]
    while heap:
        rx, x = heapq.heappop(heap)
        if seen[x] or -rx != r[x]:
            continue
        seen[x] = True
        for e in range(off[x], off[x + 1]):
            y = adj[e]
            if seen[y]:
                continue
            r[y] += w[e]
            heapq.heappush(heap, (-r[y], y))
            if r[y] >= lam:
                a, b = sorted((find(x), find(y)))
                parent[b] = a
    return [find(v) for v in range(G.n)]


@pytest.mark.parametrize("n", [2, 40, 513, 4000, 16384, 16390])
def test_exact_round_unchecked_weights(n):
    """A step takes any 64-bit weights: those below 0 count as 0, sums may pass 2^63, and every
    vertex is still taken exactly once."""
    g = ring_graph(n, 3 + n, 1, 9)
    G = oracle.as_csr64(g.offsets, g.adj, g.w)
    src = np.repeat(np.arange(n), np.diff(G.offsets))
    mixed = np.where((src * 7 + G.adj * 7) % 5 < 2, -G.w, G.w)
    huge = (1 << 60) * np.minimum(G.w, 7)
    for w, bounds in ((mixed, (1, 5, 20, 1 << 40)), (huge, (1, 1 << 60, (1 << 62) + 5, (1 << 63) - 1))):
        d = vc.viecut_graph_upload(G.offsets, G.adj, w)
        try:
            for lam in bounds:
                ref = any_round(oracle.CsrGraph(G.offsets, G.adj, np.maximum(w, 0)), lam)
                got, ch = vc.viecut_step_noi_round(d, lam)
                assert np.array_equal(got, ref), lam
                assert ch == int(any(ref[v] != v for v in range(n)))
        finally:
            vc.viecut_graph_free(d)


@pytest.mark.parametrize("n", [2, 40, 513, 4000, 16384, 16390])
def test_exact_round_negative_weights_large_bounds(n):
    """Few small weights, some below 0, under bounds near 2^63, at which two entries of the bound
    would already leave 64 bits."""
    g = ring_graph(n, 9 + n, 1, 9)
    G = oracle.as_csr64(g.offsets, g.adj, g.w)
    src = np.repeat(np.arange(n), np.diff(G.offsets))
    w = np.where((src * 7 + G.adj * 7) % 5 < 3, -G.w, G.w)
    d = vc.viecut_graph_upload(G.offsets, G.adj, w)
    try:
        for lam in (1 << 61, (1 << 62) + 5, (1 << 63) - 1):
            ref = any_round(oracle.CsrGraph(G.offsets, G.adj, np.maximum(w, 0)), lam)
            got, ch = vc.viecut_step_noi_round(d, lam)
            assert np.array_equal(got, ref), lam
            assert ch == int(any(ref[v] != v for v in range(n)))
    finally:
        vc.viecut_graph_free(d)


@pytest.mark.parametrize("n", [2, 40, 513, 3000, 16390])
def test_exact_round_zero_weights(n):
    """Entries of weight 0: they join their ends where the bound is below 1, and only there."""
    g = ring_graph(n, 5 + n, 1, 9)
    G = oracle.as_csr64(g.offsets, g.adj, g.w)
    src = np.repeat(np.arange(n), np.diff(G.offsets))
    for w in (np.where((src + G.adj) % 3 == 0, G.w, 0), np.zeros(G.nnz, np.int64)):
        Z = oracle.CsrGraph(G.offsets, G.adj, w)
        d = vc.viecut_graph_upload(Z.offsets, Z.adj, Z.w)
        try:
            for lam in (-3, 0, 1, 2, 12):
                got, ch = vc.viecut_step_noi_round(d, lam)
                ref, cnt = oracle.noi_round(Z, lam)
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


LENGTHS = (1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 257, 511, 512, 513, 1025, 2049, 4095, 4096,
           4097)


def lengths_graph(weights):
    """Vertices of exactly the list lengths at the edges of the kernels' classes, over 12,000
    leaves that form a ring."""
    rng = np.random.default_rng(len(weights))
    n, first = 12000 + len(LENGTHS), 12000
    pairs = [(v, (v + 1) % 12000) for v in range(12000)]
    for i, d in enumerate(LENGTHS):
        pairs += [(int(u), first + i) for u in rng.choice(12000, d, replace=False)]
    return gg.from_edges(n, [(a, b, int(x)) for (a, b), x in zip(pairs, rng.choice(weights, len(pairs)))])


@pytest.mark.parametrize("weights", [(1,), (1, 2, 9), (1 << 20, 1 << 30)])
def test_list_lengths(weights):
    """Label rounds (from the identity, from others' labels with few and with many distinct
    ones) and contractions by them; whole runs, which take input weights in 32 bits."""
    g = lengths_graph(weights)
    G = oracle.as_csr64(g.offsets, g.adj, g.w)
    key = oracle.level_key(4, 0)
    rng = np.random.default_rng(8)
    for start in (np.arange(G.n), rng.integers(0, 3, G.n), rng.permutation(G.n)):
        start = start.astype(np.int32)
        ref = oracle.lp_round(G, start, key)
        d = vc.viecut_graph_upload(G.offsets, G.adj, G.w)
        try:
            assert np.array_equal(vc.viecut_step_lp(d, start, key, 1)[0], ref)
        finally:
            vc.viecut_graph_free(d)
        check_contract(G, ref)
    for n0 in (10, 1000):
        ref = oracle.viecut(g.offsets, g.adj, g.w, seed=5, lp_iters=2, n0=n0)
        with vc.MinCut(g.offsets, g.adj, g.w, n0=n0) as mc:
            cut, bits = mc.run(5, 2)
            assert mc.trace() == ref.trace
        assert cut == ref.cut and np.array_equal(bits, ref.side_bits)


PAIRS = (2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 2047, 2048, 2049,
         4095, 4096, 4097, 5000)


@pytest.mark.parametrize("sparse", [True, False])
def test_contract_cluster_pairs(sparse):
    """Clusters of two vertices with exactly the pair counts at the edges of the merge's
    classes, half of the targets in both lists; the other clusters single vertices, under
    their own ids or another's."""
    rng = np.random.default_rng(2)
    leaves, edges = 9000, []
    for i, t in enumerate(PAIRS):
        us = rng.choice(leaves, t // 2 + t % 2, replace=False)
        a = leaves + 2 * i
        edges += [(int(u), a, int(rng.integers(1, 50))) for u in us]
        vs = np.concatenate([us[:t // 4], rng.choice(np.setdiff1d(np.arange(leaves), us), t // 2 - t // 4,
                                                     replace=False)])
        edges += [(int(u), a + 1, int(rng.integers(1, 50))) for u in vs]
    n = leaves + 2 * len(PAIRS)
    g = gg.from_edges(n, edges + [(v, (v + 1) % leaves, 3) for v in range(leaves)])
    G = oracle.as_csr64(g.offsets, g.adj, g.w)
    labels = np.arange(n) if sparse else np.roll(np.arange(n), 1)
    labels[leaves + 1::2] = labels[leaves::2]
    check_contract(G, labels)


@pytest.mark.parametrize("n", [16383, 16384, 16385, 32767, 32769])
def test_contract_vertex_counts(n):
    """Vertex counts at the edge of the one-block scan."""
    g = ring_graph(n, 5, 1, 9)
    G = oracle.as_csr64(g.offsets, g.adj, g.w)
    near = np.arange(n)
    near[1::400] = near[0::400][:len(near[1::400])]
    for labels in (near, np.random.default_rng(1).permutation(n) // 2, np.arange(n) // 3):
        check_contract(G, labels)


def test_contract_large_near_identity():
    """Graphs of more than 2^25 entries where few vertices merge: the lists next to a merged
    group are the only ones read (up to a sixteenth of the vertices), the others renumbered by
    the run (up to one in 512), also those of a hub and of vertices under another's id."""
    g = gg.er(700_000, 50, 3, 1, 100)
    G = oracle.as_csr64(g.offsets, g.adj, g.w)
    n = G.n
    assert G.nnz >= 1 << 25
    rng = np.random.default_rng(6)
    labels = np.arange(n)
    labels[rng.choice(n, 200, replace=False)] = 77
    hub = check_contract(G, labels)  # 77: a list of about 10,000 entries
    assert np.diff(hub.offsets).max() > 4096
    for gone in (hub.n // 512 - 8, hub.n // 512 + 8, hub.n // 16 + 8):
        labels = np.arange(hub.n)
        pick = rng.choice(hub.n, 2 * gone, replace=False)
        labels[pick[:gone]] = labels[pick[gone:]]
        labels[pick[0]] = int(np.diff(hub.offsets).argmax())
        check_contract(hub, labels)
    labels = np.arange(hub.n)
    a, b = rng.choice(hub.n, (2, 50), replace=False)
    labels[a], labels[b] = b, a
    check_contract(hub, labels)


def test_run_of_changed_lists_and_hubs():
    """A graph whose levels run many passes over the lists that the last one changed, with
    hubs of more than 4096 entries from merges, both ends of some pairs long."""
    g = gg.planted(4, 1 << 15, 24, 8, 3)
    ref = oracle.viecut(g.offsets, g.adj, g.w, seed=2, lp_iters=2, n0=1000)
    with vc.MinCut(g.offsets, g.adj, g.w, n0=1000) as mc:
        for _ in range(2):  # the second run finds every workspace in place
            cut, bits = mc.run(2, 2)
            assert mc.trace() == ref.trace
            assert cut == ref.cut and np.array_equal(bits, ref.side_bits)


@pytest.mark.parametrize("weighted", [False, True])
def test_converging_rounds_with_a_hub(weighted):
    """Rounds over the neighbours of changed vertices only, a hub among them."""
    base = gg.core_lcc(gg.rhg(1 << 16, 16, 12), 0)
    if weighted:
        base = gg.with_pair_weights(base, 4, 1, 9)
    src = np.repeat(np.arange(base.n), np.diff(base.offsets))
    hub = np.random.default_rng(3).choice(base.n, 6000, replace=False)
    one = np.ones(6000, np.int32)
    a = np.concatenate([src, hub, np.full(6000, base.n)])
    b = np.concatenate([base.adj, np.full(6000, base.n), hub])
    w = np.concatenate([base.w, one, one])
    order = np.lexsort((b, a))
    off = np.concatenate([[0], np.cumsum(np.bincount(a, minlength=base.n + 1))]).astype(np.int64)
    adj, w = b[order].astype(np.int32), w[order].astype(np.int32)
    ref = oracle.viecut(off, adj, w, seed=3, lp_iters=25, n0=500, converge=True)
    with vc.MinCut(off, adj, w, n0=500, lp_converge=True) as mc:
        cut, bits = mc.run(3, 25)
        assert mc.trace() == ref.trace
    assert cut == ref.cut and np.array_equal(bits, ref.side_bits)


def dropped(g, share, seed):
    """The graph without a random share of its entries, so that some edges are in one list only."""
    keep = np.random.default_rng(seed).random(len(g.adj)) >= share
    off = np.concatenate([[0], np.cumsum(keep)])[g.offsets].astype(np.int64)
    return off, g.adj[keep], g.w[keep]


def test_contract_large_not_symmetric():
    """More than 2^25 entries, some edges in one list only: a list next to a merged group cannot
    be found from the group's own."""
    G = oracle.as_csr64(*dropped(gg.er(700_000, 60, 3, 1, 100), 0.15, 1))
    assert G.nnz >= 1 << 25
    rng = np.random.default_rng(6)
    for gone in (200, G.n // 16 - 8):
        labels = np.arange(G.n)
        pick = rng.choice(G.n, 2 * gone, replace=False)
        labels[pick[:gone]] = labels[pick[gone:]]
        G = check_contract(G, labels)


def test_converging_rounds_not_symmetric():
    """Converging rounds where a vertex may follow one that does not list it."""
    off, adj, w = dropped(gg.core_lcc(gg.rhg(1 << 18, 24, 12), 0), 0.2, 2)
    ref = oracle.viecut(off, adj, w, seed=3, lp_iters=25, n0=500, pr_runs_max=0, converge=True)
    with vc.MinCut(off, adj, w, n0=500, pr_runs_max=0, lp_converge=True) as mc:
        cut, bits = mc.run(3, 25)
        assert mc.trace() == ref.trace
    assert cut == ref.cut and np.array_equal(bits, ref.side_bits)


@pytest.mark.parametrize("weighted", [False, True])
def test_converging_rounds_count_their_entries(weighted):
    """The statistics of a level whose later rounds visit the neighbours of changed vertices
    only: the entries those rounds read are counted, the others' are not."""
    g = gg.core_lcc(gg.rhg(1 << 16, 32, 5), 0)
    if weighted:
        g = gg.with_pair_weights(g, 4, 1, 9)
    G = oracle.as_csr64(g.offsets, g.adj, g.w)
    deg, src = np.diff(G.offsets), np.repeat(np.arange(G.n), np.diff(G.offsets))
    label, moved, few = np.arange(G.n, dtype=np.int32), None, False
    nnz, size, restricted = 0, 0, 0
    for r in range(25):
        entries = int(deg[np.unique(G.adj[moved[src]])].sum()) if few else G.nnz
        nnz += entries
        size += 8 * (G.n + 1) + entries * (4 + (4 if weighted else 0) + (4 if r else 0)) + 4 * G.n
        restricted += few
        after = oracle.lp_round(G, label, oracle.level_key(3, 0))
        moved, label = after != label, after
        if int(moved.sum()) * 10000 <= G.n:
            break
        few = few or int(moved.sum()) * 32 <= G.n
    assert restricted > 0
    with vc.MinCut(g.offsets, g.adj, g.w, n0=G.n - 1, lp_converge=True, timing=True) as mc:
        for _ in range(2):
            mc.run(3, 25)
            st = mc.stats()
            assert st["levels"] == 1 and st["lp_launches"] == r + 1
            assert st["lp_nnz"] == nnz and st["lp_bytes"] == size


@pytest.mark.parametrize("entries", [8192, 8193, 9000])
def test_partners_of_a_long_list_with_negative_weights(entries):
    """Weights below 0 (an upload takes any) count in a long list's degree as in a short one's."""
    ring = [(v, (v + 1) % entries, 90 if v in (6, 7) else 1) for v in range(entries)]
    star = [(v, entries, 100 if v == 7 else 1) for v in range(entries)]
    g = gg.from_edges(entries + 1, ring + star)
    src = np.repeat(np.arange(g.n), np.diff(g.offsets))
    hub = (src == entries) | (g.adj == entries)
    w = np.where(hub & ((src + g.adj) % 2 == 1) & (g.w == 1), -1, g.w)
    G = oracle.as_csr64(g.offsets, g.adj, w)
    d = vc.viecut_graph_upload(G.offsets, G.adj, G.w)
    try:
        ref, cnt = oracle.pr_pass_a(G, 1000)
        got, ch = vc.viecut_step_pr_a(d, 1000)
        assert ref[entries] == ref[7]  # by the hub's degree of about 100 alone: vertex 7's is 280
        assert np.array_equal(got, ref) and ch == (1 if cnt > 0 else 0)
    finally:
        vc.viecut_graph_free(d)


def check_pass_b(G, lam):
    d = vc.viecut_graph_upload(G.offsets, G.adj, G.w)
    try:
        got, ch = vc.viecut_step_pr_b(d, lam)
    finally:
        vc.viecut_graph_free(d)
    ref, cnt = oracle.pr_pass_b(G, lam)
    assert np.array_equal(got, ref) and ch == (1 if cnt > 0 else 0)
    return ref


@pytest.mark.parametrize("longer", [0, 1500])
def test_pass_b_long_pairs(longer):
    """Mutual partners whose shorter list is at the edge of what the grid's blocks share, one
    unit to either side of conditions 3 and 4 (each alone decisive; the longer list of some
    pairs first, of others second)."""
    lam, n0, rng = 10000, 20000, np.random.default_rng(5)
    blob = gg.er(n0, 56, 9)
    src = np.repeat(np.arange(n0), np.diff(blob.offsets))
    edges = [(int(a), int(b), 1) for a, b in zip(src, blob.adj) if a < b]
    pairs, at = [], n0

    def private(v, k, w, kw, avoid):  # neighbours of v alone and of w alone
        own = rng.choice(np.setdiff1d(np.arange(n0), avoid), k + kw, replace=False)
        edges.extend((int(u), v if i < k else w, 1) for i, u in enumerate(own))

    for size in (2047, 2048, 2049, 2050, 4097):  # entries of the shorter list
        for case in ("3", "not 3", "4", "not 4"):
            v, w = (at, at + 1) if len(pairs) % 2 else (at + 1, at)
            at += 2
            if case.endswith("3"):  # one common neighbour: degree = 2 (c + y) or one more
                p = size - 2
                c = p // 2 + 1
                y = p - c - (case != "3")
                u = int(rng.integers(n0))
                edges += [(u, v, y), (u, w, y), (v, w, c)]
                private(v, p, w, p, [u])
            else:  # 900 common neighbours of weight 10, c + 9000 = lam or one less
                u = rng.choice(n0, 900, replace=False)
                edges += [(int(x), v, 10) for x in u] + [(int(x), w, 10) for x in u]
                edges.append((v, w, lam - 9000 - (case != "4")))
                private(v, size - 901, w, size - 901 + longer, u)
            pairs.append((v, w, case))
    g = gg.from_edges(at, [(min(a, b), max(a, b), x) for a, b, x in edges])
    G = oracle.as_csr64(g.offsets, g.adj, g.w)
    assert G.nnz >= 1 << 20 and (np.diff(G.offsets)[n0:] > 2048).sum() >= 24
    ref = check_pass_b(G, lam)
    for v, w, case in pairs:
        assert (ref[v] == ref[w]) == (case in ("3", "4")), (v, w, case)


def test_run_of_passes_over_changed_lists():
    """Passes that test only the lists the last contractions changed, and find merges that those
    made: a and b are joined by an edge of the bound, then c and then d by two edges of half the
    bound each, one to either part of what was joined before, and pass B joins p and q once
    their common neighbour is one vertex.  A chain apart from the rest collapses a vertex a pass
    and ends the run with its last one."""
    n, lam, rng = 140_000, 10, np.random.default_rng(4)
    blob = gg.er(n, 36, 2)
    src = np.repeat(np.arange(n), np.diff(blob.offsets))
    weight = {(int(a), int(b)): 1 for a, b in zip(src, blob.adj) if a < b}
    pick = rng.permutation(np.flatnonzero(np.diff(blob.offsets) >= 26))[:20 * 6].reshape(20, 6)
    for a, b, c, d, p, q in pick.tolist():
        for x, y, wt in ((a, b, lam), (a, c, 5), (b, c, 5), (a, d, 5), (c, d, 5), (p, q, 6), (c, p, 4), (a, q, 4)):
            weight[min(x, y), max(x, y)] = wt
    for u in rng.choice(n, lam, replace=False):
        weight[int(u), n] = 1  # the vertex of smallest degree
    chain, e0 = 9, n + 1
    weight[e0, e0 + 1] = lam
    for k in range(2, chain):
        weight[e0 + k - 1, e0 + k] = 5
        for x in (e0, e0 + 1):
            weight[x, e0 + k] = weight.get((x, e0 + k), 0) + 3
    g = gg.from_edges(n + 1 + chain, [(a, b, wt) for (a, b), wt in sorted(weight.items())])
    ref = oracle.viecut(g.offsets, g.adj, g.w, seed=2, lp_iters=0, n0=1000)
    # a pass is restricted where the last one of its kind had the same bound and at most a quarter
    # of the lists changed since: at most those of the vertices merged so far and their neighbours
    widest = int(np.diff(g.offsets).max())
    size, seen, restricted = g.n, set(), {2: 0, 3: 0}
    assert [t[4] for t in ref.trace[2:]] == [lam] * (len(ref.trace) - 3) + [0]
    for kind, level, left, *_ in ref.trace[2:]:
        assert kind in (2, 3) and level == 0 and left >= 1 << 17
        restricted[kind] += kind in seen and 4 * 2 * (g.n - size) * (widest + 1) <= size
        seen.add(kind)
        size = left
    assert restricted[2] >= 2 and restricted[3] >= 1 and ref.cut == 0
    with vc.MinCut(g.offsets, g.adj, g.w, n0=1000) as mc:
        for _ in range(2):
            cut, bits = mc.run(2, 0)
            assert mc.trace() == ref.trace
            assert cut == ref.cut and np.array_equal(bits, ref.side_bits)


def test_contract_large_near_identity_unit():
    """As test_contract_large_near_identity on unit weights, then with several hubs among the
    merged vertices (their lists are shared by the grid's blocks)."""
    g = gg.er(700_000, 50, 8)
    G = oracle.as_csr64(g.offsets, g.adj, g.w)
    assert G.nnz >= 1 << 25
    rng = np.random.default_rng(9)
    labels = np.arange(G.n)
    pick = rng.choice(G.n, 2000, replace=False)
    labels[pick[:1000]] = labels[pick[1000:]]
    check_contract(G, labels)
    labels = np.arange(G.n)
    members = rng.choice(G.n, 1200, replace=False).reshape(6, 200)
    labels[members] = members[:, :1]
    hubs = check_contract(G, labels)
    wide = np.flatnonzero(np.diff(hubs.offsets) > 4096)
    assert len(wide) == 6
    labels = np.arange(hubs.n)
    labels[wide[:3]] = rng.choice(hubs.n, 3, replace=False)
    labels[wide[3]] = wide[4]
    check_contract(hubs, labels)


def test_exact_rounds_on_a_large_input():
    """Exact rounds on an input of more than 2^25 entries with 32-bit weights that join one pair
    of a regular circulant graph, so that nearly every list is renumbered by the run; the second
    round reads what the first one's contraction wrote.  A triangle apart from it collapses in
    two rounds and ends the run."""
    n, half = 40_000, 420
    step = np.concatenate([np.arange(1, half + 1), np.arange(n - half, n)])
    wt = (1 + np.minimum(step, n - step) % 7).astype(np.int32)
    adj = ((np.arange(n)[:, None] + step) % n).astype(np.int32)
    order = np.argsort(adj, axis=1)
    adj, w = np.take_along_axis(adj, order, 1).ravel(), wt[order].ravel()
    degree = int(wt.sum())
    side = degree // 2 + 1
    adj = np.concatenate([adj, np.array([n + 1, n + 2, n, n + 2, n, n + 1], np.int32)])
    w = np.concatenate([w, np.full(6, side, np.int32)])
    off = np.concatenate([np.arange(n + 1) * 2 * half, n * 2 * half + np.array([2, 4, 6])]).astype(np.int64)
    assert len(adj) >= 1 << 25
    ref = oracle.viecut(off, adj, w, seed=1, lp_iters=2, n0=n + 3)
    assert [t[0] for t in ref.trace] == [0, 4, 4] and ref.trace[2][3] >= 1 << 25
    assert [t[2] for t in ref.trace] == [n + 3, n + 1, n - 1] and ref.cut == 0
    with vc.MinCut(off, adj, w, n0=n + 3) as mc:
        cut, bits = mc.run(1, 2)
        assert mc.trace() == ref.trace
    assert cut == ref.cut and np.array_equal(bits, ref.side_bits)


def test_run_of_changed_lists_many_passes():
    """Degrees, partners and flags carried over many passes on a graph whose hubs grow from merges
    (planted blocks, 2^19 vertices)."""
    g = gg.planted(8, 1 << 16, 24, 8, 3)
    ref = oracle.viecut(g.offsets, g.adj, g.w, seed=2, lp_iters=2, n0=1000)
    assert sum(t[0] in (2, 3) and t[2] >= 1 << 17 for t in ref.trace) >= 8
    with vc.MinCut(g.offsets, g.adj, g.w, n0=1000) as mc:
        for _ in range(2):
            cut, bits = mc.run(2, 2)
            assert mc.trace() == ref.trace
            assert cut == ref.cut and np.array_equal(bits, ref.side_bits)
