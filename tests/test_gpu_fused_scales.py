"""Scales and compress in one launch at every block size that has it, from its smallest number of
blocks on (called repeatedly: the counters have to be zero again)."""
import pytest

from paper_2302_08545_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,nblk,n,bits", [(17, 16, 5, 8), (17, 130, 2, 4), (18, 20, 3, 3), (19, 9, 4, 1),
                                           (18, 131, 1, 4), (17, 16, 1, 4), (18, 1, 1, 4), (18, 14, 3, 2),
                                           (19, 2, 1, 8), (19, 6, 4, 4), (20, 2, 1, 1), (20, 4, 4, 4)])
def test_one_launch_equals_the_two_calls(k, nblk, n, bits):
    import torch
    from paper_2302_08545_b200 import runner
    g = {1: 1, 2: 3, 3: 12, 4: 30, 8: 255}[bits]
    table = {3: (0, 2, 4, 5, 6, 7, 9, 12)}.get(bits) or W.TABLES[(bits, g)]
    d = nblk * (1 << k) - 777
    w = W.Workload("plain", n=n, d=d, log2_block=k, bits=bits, granularity=g, table=tuple(table), data_seed=k)
    ctx = runner.context_for(w)
    r = runner.Round(ctx, n, d)
    assert r.sz.fused_scales == 1
    for call in range(2):
        W.fill_torch(w, r.grads, seed_offset=call)
        r.grads[0][: 1 << k] = 0.0
        if n > 1:
            r.grads[n - 1][5] = 1e-30
        r.prepare_compress(call)
        torch.cuda.synchronize()
        assert ctx.status() & ~2 == 0
        s, p = r.scales.clone(), [t.clone() for t in r.packed]
        r.prepare()
        ulp = (s.view(torch.int32) - r.scales.view(torch.int32)).abs().max().item()
        assert ulp <= 1
        r.scales.copy_(s)
        r.compress(call)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(p, r.packed))
