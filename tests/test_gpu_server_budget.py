"""A server's admission budget covers what a request takes on the device."""
import gc

import numpy as np
import pytest

import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [4, 6])
def test_budget_covers_a_sparse_request(k):
    """A forest of paths of k vertices, run without label propagation: arrays of a vertex's size
    outweigh those of an entry's.  A budget just below what the run takes refuses the request."""
    import torch

    import paper_1708_06127_gb300 as vc
    n = (1 << 21) // k * k
    v = np.arange(n)
    degree = 2 - (v % k == 0) - (v % k == k - 1)
    off = np.concatenate([[0], np.cumsum(degree)]).astype(np.int64)
    src = np.repeat(v, degree)
    second = np.arange(len(src)) - off[src] == 1
    adj = np.where(second | (src % k == 0), src + 1, src - 1).astype(np.int32)
    w = np.ones(len(adj), np.int32)
    small = gg.core_lcc(gg.rhg(1 << 14, 32, 5), 0)
    for n0 in (10000, 1000):  # what a process allocates once
        with vc.MinCut(small.offsets, small.adj, small.w, n0=n0) as mc:
            mc.run(1, 0)
    gc.collect()
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    with vc.MinCut(off, adj, w, n0=1000) as mc:
        cut, _ = mc.run(1, 0)
        assert cut == 0
        taken = before - torch.cuda.mem_get_info()[0]
    assert taken > 0
    with vc.Server(hbm_budget_bytes=taken - 1, n0=1000, lp_iters=0, solo_lanes=1, max_slots=4) as srv:
        with pytest.raises(vc.ViecutError) as e:
            srv.submit(off, adj, w, seed=1)
        assert e.value.code == vc.VIECUT_EINVAL and "budget" in str(e.value)
