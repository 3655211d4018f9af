"""Exact ranges with the context's own keys and with keys in the workspace (more blocks), at the edges
of tiles and kernels, called repeatedly: the keys of one call have to be cleared for the next."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2302_08545_b200 import workloads as W

pytestmark = pytest.mark.gpu
T = W.TABLES[(4, 30)]


@pytest.mark.parametrize("k,d,n", [(3, 4096 * 8, 2), (3, 4097 * 8, 2), (12, 100_001, 2), (14, 40_000, 1), (15, 100_000, 2), (16, 65_536 * 70, 1),
                                   (17, 300_000, 2), (20, (1 << 20) + 3, 2)])
def test_exact_ranges(k, d, n):
    import torch
    from paper_2302_08545_b200 import runner
    w = W.Workload("plain", n=n, d=d, log2_block=k, bits=4, granularity=30, table=T, data_seed=k)
    ctx = runner.context_for(w, exact_range=True)
    r = runner.Round(ctx, n, d)
    c = O.Config(bits=4, granularity=30, table=T, t_p=w.t_p, log2_block=k, seed=w.seed)
    for call in range(3):
        W.fill_torch(w, r.grads, seed_offset=call)
        if call == 1:
            r.grads[0][d - 1] = float("inf")
        r.prepare_minmax(call)
        torch.cuda.synchronize()
        s = r.scales.cpu().numpy()
        nb = r.sz.nblocks
        last = nb - 1 if call == 1 else nb
        if call == 1:
            assert ctx.status() & 1 and s[nb - 1] == 0 and s[2 * nb - 1] == 0
            r.grads[0][d - 1] = 0.0
        lo, hi = O.ranges(np.stack([t.cpu().numpy() for t in r.grads]), c, call)
        assert np.array_equal(s[:last].view(np.uint32), lo[:last].view(np.uint32))
        assert np.array_equal(s[nb: nb + last].view(np.uint32), hi[:last].view(np.uint32))
