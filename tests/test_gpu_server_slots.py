"""A server's unused slots: their per-slot records start defined, whatever the device memory
held before, so kernels that visit every slot leave them alone."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fill", [0xFF, 0x08])
def test_unused_slots_on_reused_memory(fill):
    import torch

    import paper_1708_06127_gb300 as vc
    # device memory that held other data goes back to the driver just before the start
    old = [torch.full((1 << k,), fill, dtype=torch.uint8, device="cuda") for k in range(12, 27)]
    torch.cuda.synchronize()
    del old
    torch.cuda.empty_cache()
    graphs = [gg.core_lcc(gg.rhg(n, 16, 5 + n), 0, True) for n in (100, 700, 1500)]
    with vc.Server(max_slots=512, n0=200, solo_min_n=0) as srv:
        tickets = [srv.submit(g.offsets, g.adj, g.w, seed=3) for g in graphs]
        for g, t in zip(graphs, tickets):
            cut, bits, _ = srv.wait(t, timeout=60.0)
            ref = oracle.viecut(g.offsets, g.adj, g.w, seed=3, lp_iters=2, n0=200)
            assert cut == ref.cut
            assert np.array_equal(bits, ref.side_bits)
