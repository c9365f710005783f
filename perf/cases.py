"""Performance cases: minimum cuts of seeded synthetic graphs through the public entry points.

The graphs are drawn on the GPU from the seed alone, in the families this repository
tests and benchmarks: random hyperbolic graphs (exponent 5), Erdos-Renyi blocks with
bridges, clustered Erdos-Renyi graphs with weighted clusters, and the batch mix of them.  Every output is a whole number (the cut value and the side bitmap), so
there is nothing that a 64-bit evaluation would give more exactly (``exact``).
"""
import math

import numpy as np
import torch

import paper_1708_06127_gb300 as vc

N0 = 10000  # the library's default: at most this many vertices go to the exact step
DEVICE = "cuda" if torch.cuda.is_available() else "cpu"


def listed():
    return [
        # One tiny graph from host memory to a host result: the call a program makes per
        # small instance (a kernel of a branch and bound, a community of a network).  Its
        # whole run is the dense exact step; latency and launches count.
        {"name": "exact_500", "kind": "single", "family": "rhg", "n": 500, "deg": 16, "host": True},
        # A graph just below n0: the whole run is the exact step (the requests that a server
        # routes to its exact lanes, exact_min_cut on a mid-sized graph).
        {"name": "exact_8k", "kind": "single", "family": "rhg", "n": 8191, "deg": 32, "host": True},
        # The benchmark's small graph (n = 2^14, average degree 32, exponent 5): one level
        # of label propagation and the exact step, still bound by launches and host reads.
        {"name": "rhg_16k", "kind": "single", "family": "rhg", "n": 1 << 14, "deg": 32, "host": True},
        # A mid-sized weighted graph of ragged size (weights 1..10), resident on the device.
        {"name": "rhg_250k_weighted", "kind": "single", "family": "rhg", "n": 249989, "deg": 32, "wmax": 10},
        # The high-quality configuration (up to 25 rounds with the convergence stop, and the
        # correcting step) on a mid-sized graph.
        {"name": "rhg_300k_viecut25", "kind": "single", "family": "rhg", "n": 300007, "deg": 32, "lp_iters": 25,
         "converge": True, "correct": True},
        # The headline workload: n = 2^22, average degree 64, unit weights, on the device.
        {"name": "rhg_4m", "kind": "single", "family": "rhg", "n": 1 << 22, "deg": 64},
        # Dense weighted clusters (the clustered Erdos-Renyi family: density 10 %, two
        # clusters, heavy intra-cluster weights): lists of 1,600 entries.
        {"name": "clustered_16k", "kind": "single", "family": "clustered", "n": 16001, "density": 10.0, "k": 2},
        # The planted-cut workload at full size (8 blocks of 2^20 vertices, average degree
        # 48, 64 bridges, weights 1..100): weak clusters, many Padberg-Rinaldi passes.
        {"name": "planted_8x1m", "kind": "single", "family": "planted", "blocks": 8, "block_n": 1 << 20, "deg": 48},
        # The same family at a size where the passes are shorter and launches count more.
        {"name": "planted_8x60k", "kind": "single", "family": "planted", "blocks": 8, "block_n": 60013, "deg": 40},
        # End to end from page-locked host memory: load and run in one call.
        {"name": "solve_500k", "kind": "solve", "family": "rhg", "n": 500009, "deg": 64},
        # Many small weighted graphs in one call (the batch mix: n log-uniform 2^6..2^14, random
        # hyperbolic or Erdos-Renyi).
        {"name": "batch_1000", "kind": "batch", "count": 1000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["exact", "rhg", "rhg", "options", "clustered", "planted", "solve", "batch"])
    if kind == "exact":
        n = _log_int(rng, 64, N0)
        return {"kind": "single", "family": "rhg", "n": n, "deg": min(rng.randint(12, 64), (n - 1) // 3), "host": True}
    if kind == "rhg":
        deg = rng.randint(16, 64)
        n = _log_int(rng, N0 + 1, 1 << 22)
        return {"kind": "single", "family": "rhg", "n": n, "deg": deg, "wmax": rng.choice([1, 1, 10, 100]),
                "lp_iters": rng.choice([1, 2, 2, 3])}
    if kind == "options":
        return {"kind": "single", "family": "rhg", "n": _log_int(rng, N0 + 1, 600000), "deg": rng.randint(16, 64),
                "lp_iters": rng.choice([2, 25]), "converge": rng.random() < 0.5, "correct": rng.random() < 0.5,
                "lp_async": rng.choice([0, 0, 1, 2])}
    if kind == "clustered":
        return {"kind": "single", "family": "clustered", "n": _log_int(rng, N0 + 1, 24000),
                "density": round(rng.uniform(2.0, 10.0), 1), "k": rng.choice([2, 4, 8])}
    if kind == "planted":
        return {"kind": "single", "family": "planted", "blocks": rng.choice([4, 8]),
                "block_n": _log_int(rng, 4000, 400000), "deg": rng.randint(24, 48)}
    if kind == "solve":
        return {"kind": "solve", "family": "rhg", "n": _log_int(rng, 4096, 1 << 20), "deg": rng.randint(16, 64),
                "wmax": rng.choice([1, 1, 10])}
    return {"kind": "batch", "count": _log_int(rng, 32, 1200)}


# --------------------------------------------------------------------- graphs
def _uniform(g, count):
    return torch.rand(count, generator=g, device=DEVICE, dtype=torch.float64)


def _csr(n, a, b, g, wmax, weigh=None):
    """Sorted CSR of the undirected pairs (a, b) without repeats: offsets int64, ids and
    weights int32 (uniform in 1..wmax, or weigh(a, b, w))."""
    bits = max(1, (n - 1).bit_length())
    pair = torch.unique((torch.minimum(a, b) << bits) | torch.maximum(a, b))
    a, b = pair >> bits, pair & ((1 << bits) - 1)
    a, b = a[a != b], b[a != b]
    w = torch.randint(1, wmax + 1, a.shape, generator=g, device=DEVICE) if wmax > 1 else torch.ones_like(a)
    if weigh is not None:
        w = weigh(a, b, w)
    # sorted as (row, column, weight) packed into one integer
    wb = 24 if bits <= 19 else 8
    key = torch.sort(torch.cat([(a << bits | b) << wb | w, (b << bits | a) << wb | w]))[0]
    w, key = key & ((1 << wb) - 1), key >> wb
    off = torch.zeros(n + 1, dtype=torch.int64, device=DEVICE)
    torch.cumsum(torch.bincount(key >> bits, minlength=n), 0, out=off[1:])
    return off, (key & ((1 << bits) - 1)).to(torch.int32), w.to(torch.int32)


def _rhg_pairs(ns, degs, g):
    """Pairs of a disjoint union of threshold random hyperbolic graphs (power-law exponent
    5, alpha = 2), graph i of ns[i] vertices and about degs[i] neighbours each; the ids of
    a graph follow angular order.  Vertices are scanned against radial bands: band b's
    points within the angle at which its innermost radius still connects."""
    alpha = 2.0
    nt = torch.tensor(ns, dtype=torch.int64, device=DEVICE)
    n = int(sum(ns))
    gid = torch.repeat_interleave(torch.arange(len(ns), device=DEVICE), nt)
    xi = alpha / (alpha - 0.5)
    radius = torch.tensor([max(1.0, 2 * math.log(2 / math.pi * xi * xi * m / d)) for m, d in zip(ns, degs)],
                          dtype=torch.float64, device=DEVICE)
    big_r = radius[gid]
    r = torch.acosh(1 + _uniform(g, n) * (torch.cosh(alpha * big_r) - 1)) / alpha
    at = torch.sort(gid * 8.0 + _uniform(g, n) * (2 * math.pi))[0]  # graph, then angle
    theta = at - gid * 8.0
    ch, sh, cr = torch.cosh(r), torch.sinh(r), torch.cosh(big_r)
    # by distance from the rim: 0.25 wide up to 3 (nearly all points), then 1 wide to the centre
    edges = [0.25 * q for q in range(12)] + [3.0 + q for q in range(max(1, math.ceil(float(radius.max()) - 3.0)) + 1)]
    band = torch.searchsorted(torch.tensor(edges[1:-1], dtype=torch.float64, device=DEVICE), big_r - r, right=True)
    out_a, out_b = [], []
    ids = torch.arange(n, device=DEVICE)
    for q in range(len(edges) - 1):
        mem = ids[band == q]
        if mem.numel() == 0:
            continue
        mem_at = at[mem]
        inner = torch.clamp(big_r - edges[q + 1], min=0.0)
        den = sh * torch.sinh(inner)
        cosang = torch.where(den > 0, (ch * torch.cosh(inner) - cr) / torch.clamp(den, min=1e-300),
                             torch.full_like(den, -1.0))
        ang = torch.acos(torch.clamp(cosang, -1.0, 1.0)) + 1e-9
        end = gid * 8.0 + 7.0
        lo1 = torch.searchsorted(mem, ids, right=True)
        hi1 = torch.searchsorted(mem_at, torch.minimum(at + ang, end), right=True)
        lo2 = torch.searchsorted(mem_at, gid * 8.0 + torch.maximum(theta + 2 * math.pi - ang, theta + ang))
        hi2 = torch.searchsorted(mem_at, end)
        hi1 = torch.maximum(hi1, lo1)
        lo2 = torch.maximum(lo2, hi1)
        hi2 = torch.maximum(hi2, lo2)
        del den, cosang, ang, end
        for lo, hi in ((lo1, hi1), (lo2, hi2)):
            for c in range(0, n, 1 << 20):  # some ten million candidates at a time
                l, k = lo[c:c + (1 << 20)], (hi - lo)[c:c + (1 << 20)]
                v = torch.repeat_interleave(ids[c:c + (1 << 20)], k)
                if v.numel() == 0:
                    continue
                start = torch.cumsum(k, 0) - k
                u = mem[torch.arange(v.numel(), device=DEVICE) + torch.repeat_interleave(l - start, k)]
                near = ch[v] * ch[u] - sh[v] * sh[u] * torch.cos(theta[v] - theta[u]) <= cr[v]
                out_a.append(v[near])
                out_b.append(u[near])
    return n, torch.cat(out_a), torch.cat(out_b)


def _er_pairs(ns, degs, g):
    """Pairs of a disjoint union of Erdos-Renyi graphs with about degs[i] neighbours per vertex."""
    nt = torch.tensor(ns, dtype=torch.int64, device=DEVICE)
    mt = torch.tensor([int(m * d / 2) for m, d in zip(ns, degs)], dtype=torch.int64, device=DEVICE)
    base = torch.cumsum(nt, 0) - nt
    gid = torch.repeat_interleave(torch.arange(len(ns), device=DEVICE), mt)
    a = base[gid] + (_uniform(g, gid.numel()) * nt[gid]).long()
    b = base[gid] + (_uniform(g, gid.numel()) * nt[gid]).long()
    return a, b


def _graph(case, seed):
    """The case's graph on the device: offsets, ids, weights."""
    g = torch.Generator(device=DEVICE).manual_seed(seed)
    if case["family"] == "rhg":
        n, a, b = _rhg_pairs([case["n"]], [case["deg"]], g)
        return _csr(n, a, b, g, case.get("wmax", 1))
    if case["family"] == "planted":
        k, bn = case["blocks"], case["block_n"]
        a, b = _er_pairs([bn] * k, [case["deg"]] * k, g)
        block = torch.randint(0, k, (64,), generator=g, device=DEVICE)
        other = (block + torch.randint(1, k, (64,), generator=g, device=DEVICE)) % k
        ends = torch.randint(0, bn, (2, 64), generator=g, device=DEVICE)
        return _csr(k * bn, torch.cat([a, block * bn + ends[0]]), torch.cat([b, other * bn + ends[1]]), g, 100)
    n, k = case["n"], case["k"]
    a, b = _er_pairs([n], [case["density"] / 100 * (n - 1)], g)
    part = torch.arange(n, device=DEVICE) * k // n
    return _csr(n, a, b, g, 100, lambda x, y, w: torch.where(part[x] == part[y], w * n, w))


def _mix(ns, rhg, degs, g, wmax):
    """Host arrays of a list of graphs, random hyperbolic ones (rhg[i]) first, then
    Erdos-Renyi ones.  A vertex without a neighbour gets one (a cut of 0 ends a run at once)."""
    order = sorted(range(len(ns)), key=lambda i: not rhg[i])
    ns, degs, k = [ns[i] for i in order], [degs[i] for i in order], sum(rhg)
    n, a, b = 0, *(torch.zeros(0, dtype=torch.int64, device=DEVICE) for _ in range(2))
    if k:
        n, a, b = _rhg_pairs(ns[:k], degs[:k], g)
    if k < len(ns):
        x, y = _er_pairs(ns[k:], degs[k:], g)
        a, b = torch.cat([a, x + n]), torch.cat([b, y + n])
    n = sum(ns)
    used = torch.zeros(n, dtype=torch.bool, device=DEVICE)
    used[a[a != b]] = True
    used[b[a != b]] = True
    last = torch.zeros(n, dtype=torch.int64, device=DEVICE)
    last[torch.cumsum(torch.tensor(ns, device=DEVICE), 0) - 1] = 1
    lone = torch.nonzero(~used)[:, 0]
    off, adj, w = (x.cpu().numpy() for x in _csr(n, torch.cat([a, lone]), torch.cat([b, lone + 1 - 2 * last[lone]]),
                                                 g, wmax))
    out, v = [], 0
    for c in ns:
        e0, e1 = off[v], off[v + c]
        out.append((off[v:v + c + 1] - e0, adj[e0:e1] - np.int32(v), w[e0:e1]))
        v += c
    return out


def _batch_graphs(count, seed):
    """The batch mix: n = floor(2^U(6, 14)), random hyperbolic (average degree 16..64) or
    Erdos-Renyi (8..32), weights 1..10.  The sizes are those of the count, the graphs those of the seed."""
    rnd = np.random.RandomState(count)
    ns = [int(2.0 ** x) for x in rnd.uniform(6, 14, count)]
    rhg = [bool(x < 0.5) for x in rnd.uniform(size=count)]
    degs = [min((16 + 48 * x) if h else (8 + 24 * x), (m - 1) / 3) for x, h, m in zip(rnd.uniform(size=count), rhg, ns)]
    return _mix(ns, rhg, degs, torch.Generator(device=DEVICE).manual_seed(seed), 10)


# ---------------------------------------------------------------------- cases
def _pinned(x):
    return x.cpu().pin_memory().numpy() if torch.cuda.is_available() else x.numpy()


def prepare(case, seed):
    kind = case["kind"]
    state = {"kind": kind, "seed": seed & 0xffff, "lp_iters": case.get("lp_iters", 2)}
    if kind == "batch":
        graphs = _batch_graphs(case["count"], seed)
        state["batch"] = vc.Batch(graphs)
        state["k"] = len(graphs)
        state["bits"] = np.zeros(state["batch"].words, np.uint64)
    elif kind == "solve":
        state["graph"] = [_pinned(x) for x in _graph(case, seed)]
        # the handle that a loop over many graphs keeps, made here over one edge
        state["mc"] = vc.MinCut(np.array([0, 1, 2]), np.array([1, 0], np.int32), np.ones(2, np.int32))
    else:
        off, adj, w = _graph(case, seed)
        opts = {"correct": case.get("correct", False), "lp_converge": case.get("converge", False),
                "lp_async": case.get("lp_async", 0)}
        if case.get("host"):
            state["mc"] = vc.MinCut(*(x.cpu().numpy() for x in (off, adj, w)), **opts)
        else:
            torch.cuda.synchronize()  # the handle works on a stream of its own
            state["mc"] = vc.MinCut(off, adj, w, on_device=True, **opts)
            state["cut"] = torch.empty(1, dtype=torch.int64, device=DEVICE)
            state["bits"] = torch.empty((off.numel() + 62) // 64, dtype=torch.int64, device=DEVICE)
        state["host"] = bool(case.get("host"))
    return state


def run(state):
    seed, lp_iters = state["seed"], state["lp_iters"]
    if state["kind"] == "batch":
        cuts = vc.viecut_batch_run(state["batch"].b, state["k"], seed, lp_iters, state["bits"])
        return {"cut": cuts, "side": state["bits"].view(np.int64)}
    if state["kind"] == "solve":
        cut, bits = state["mc"].solve(*state["graph"], seed=seed, lp_iters=lp_iters)
        return {"cut": cut, "side": bits.view(np.int64)}
    if state["host"]:
        cut, bits = state["mc"].run(seed=seed, lp_iters=lp_iters)
        return {"cut": cut, "side": bits.view(np.int64)}
    vc.viecut_run_device(state["mc"].h, seed, lp_iters, state["cut"], state["bits"])
    return {"cut": state["cut"], "side": state["bits"]}


def work(case):
    """Bytes of one pass: the offsets, ids and (where they are not all 1) weights of the input
    read once, the cut and the bitmap written once; the sums are one addition per entry."""
    if case["kind"] == "batch":
        # E[n] of floor(2^U(6, 14)), average degree 40 (hyperbolic) or 20 (Erdos-Renyi)
        n = case["count"] * (2 ** 14 - 2 ** 6) / (8 * math.log(2))
        m, w = 30 * n, 4
    else:
        n = case["blocks"] * case["block_n"] if case["family"] == "planted" else case["n"]
        m = n * case["deg"] if case["family"] != "clustered" else n * case["density"] / 100 * (n - 1)
        weighted = case["family"] != "rhg" or case.get("wmax", 1) > 1 or case["kind"] == "solve"
        w = 4 if weighted else 0
    return {"bytes": 8 * (n + 1) + m * (4 + w) + n / 8 + 8, "flops": m}


def exact(case, seed):
    """Every output is a whole number: compared as it is."""
    return None
