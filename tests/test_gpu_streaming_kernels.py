"""The streaming kernels at the edges of their splits: 3-bit sums (any table, 8- and 16-bit), sums to an
address that is only 16-byte aligned, residuals added in one launch and, where one gradient takes
several, in order."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2302_08545_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,g,table,n,d,k,acc", [
    (3, 7, tuple(range(8)), 3, 128, 7, 0), (3, 14, (0, 2, 4, 6, 8, 10, 12, 14), 18, 5000, 7, 0),
    (3, 14, (0, 2, 4, 6, 8, 10, 12, 14), 19, 40_000, 10, 0), (3, 200, (0, 1, 50, 99, 128, 160, 199, 200), 5, 9000, 12, 0),
    (3, 255, (0, 1, 50, 99, 128, 160, 199, 255), 2, 1000, 8, 16), (3, 9, (0, 1, 2, 3, 5, 7, 8, 9), 4, 200, 5, 0),
    (4, 30, W.TABLES[(4, 30)], 8, 100_000, 12, 0), (4, 30, W.TABLES[(4, 30)], 17, 100_000, 12, 0),
    (2, 3, (0, 1, 2, 3), 9, 100_000, 12, 0), (1, 4, (0, 4), 9, 100_000, 12, 0), (8, 255, tuple(range(256)), 9, 50_000, 12, 0),
])
@pytest.mark.parametrize("shift", [0, 16])
def test_sums(bits, g, table, n, d, k, acc, shift):
    import torch
    from paper_2302_08545_b200 import runner
    w = W.Workload("plain", n=n, d=d, log2_block=k, bits=bits, granularity=g, table=tuple(table), data_seed=1)
    ctx = runner.context_for(w, acc_bits=acc)
    sz = ctx.sizes(d, n)
    rng = np.random.default_rng(d + bits)
    packed = rng.integers(0, 256, (n, sz.packed_bytes), dtype=np.uint8)
    dev = [torch.from_numpy(p).cuda() for p in packed]
    room = torch.zeros(sz.sum_bytes + 64, dtype=torch.uint8, device="cuda")
    total = room[shift: shift + sz.sum_bytes]
    ctx.aggregate(dev, d, total)
    torch.cuda.synchronize()
    c = O.Config(bits=bits, granularity=g, table=tuple(table), t_p=w.t_p, log2_block=k, seed=w.seed)
    ref = O.aggregate(packed, sz.d_pad, c, sz.acc_bits)
    assert np.array_equal(total.cpu().numpy().view(ref.dtype), ref)
    assert not room[:shift].any() and not room[shift + sz.sum_bytes:].any()


@pytest.mark.parametrize("d,n", [(1, 2), (3, 1), (4095, 3), (4096 * 4 + 5, 2), (300_001, 5)])
def test_residuals_are_added(d, n):
    import torch
    from paper_2302_08545_b200 import runner
    w = W.Workload("plain", n=n, d=d, log2_block=10, bits=4, granularity=30, table=W.TABLES[(4, 30)], data_seed=1)
    ctx = runner.context_for(w)
    x = [torch.randn(d, device="cuda") for _ in range(n)]
    e = [torch.randn(d, device="cuda") for _ in range(n)]
    ref = [a + b for a, b in zip(x, e)]
    y = [a.clone() for a in x]
    ctx.accumulate_error(y, e, d)
    assert all(torch.equal(a, b) for a, b in zip(y, ref))
    one = x[0].clone()
    ctx.accumulate_error([one] * n, e, d)
    acc = x[0].clone()
    for r in e:
        acc = acc + r
    assert torch.equal(one, acc)
