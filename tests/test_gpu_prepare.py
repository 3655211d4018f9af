"""thc_prepare at the edges of its split: blocks below and above a slab, a CTA's tile and a chunk, more
blocks than there are counters, many workers, ragged ends; called twice, because the counters of
the first call have to be zero again for the second."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2302_08545_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,d,n,dtype", [
    (3, 4097, 2, "f32"), (3, 4095, 3, "bf16"), (6, 70_001, 33, "f32"), (7, 4096, 2, "f32"), (8, 9000, 64, "bf16"),
    (9, 12_289, 2, "f32"), (10, 50_000, 3, "bf16"), (11, 4096 * 3, 5, "f32"), (11, 6000, 2, "bf16"), (12, 8193, 9, "f32"),
    (12, 100_000, 2, "bf16"), (13, 8193, 3, "f32"), (13, 4100 << 13, 1, "bf16"), (14, 16_385, 17, "f32"),
    (17, 300_001, 2, "bf16"), (22, (1 << 22) + 5, 2, "f32"),
])
def test_scales_at_the_edges(k, d, n, dtype):
    import torch
    from paper_2302_08545_b200 import runner
    w = W.Workload("cfg4_x" if dtype == "bf16" else "plain", n=n, d=d, log2_block=k, bits=4, granularity=30,
                   table=W.TABLES[(4, 30)], in_dtype=dtype, data_seed=k + d % 89)
    c = O.Config(bits=4, granularity=30, table=tuple(w.table), t_p=w.t_p, log2_block=k, seed=w.seed)
    ctx = runner.context_for(w)
    r = runner.Round(ctx, n, d, dtype)
    for call in range(2):
        W.fill_torch(w, r.grads, seed_offset=call)
        if call == 1:
            r.grads[n - 1][d - 1] = float("nan")
        r.prepare()
        torch.cuda.synchronize()
        got = r.scales.cpu().numpy()
        if call == 1:
            assert got[-1] == 0.0 and ctx.status() & 1
            r.grads[n - 1][d - 1] = 0.0
        ref = O.scales(np.stack([t.float().cpu().numpy() for t in r.grads]), c)
        if call == 1:
            got, ref = got[:-1], ref[:-1]
        ulp = np.abs(got.view(np.int32).astype(np.int64) - ref.view(np.int32).astype(np.int64))
        assert ulp.size == 0 or ulp.max() <= 1
