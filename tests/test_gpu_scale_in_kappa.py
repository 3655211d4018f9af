"""Compress of 2^20 blocks, whose 1/sqrt(B) is a power of two, leaves out the scaling of every coordinate where
the clamp bound is of ordinary size: the indices without the rotated output (that path) and with it
(the other one) equal each other and the oracle's, also for bounds far outside the ordinary sizes.
Blocks of 2^22 scale every coordinate in both calls."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2302_08545_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,dtype", [(20, "f32"), (20, "bf16"), (22, "f32"), (22, "bf16")])
@pytest.mark.parametrize("size", [1.0, 1e-17, 1e-21, 1e-36, 1e25, 1e33])
def test_indices_with_and_without_scaling(k, dtype, size):
    import torch
    from paper_2302_08545_b200 import runner
    d = (1 << k) - 3
    w = W.Workload("cfg4_x" if dtype == "bf16" else "plain", n=1, d=d, log2_block=k, bits=4, granularity=30,
                   table=W.TABLES[(4, 30)], in_dtype=dtype, data_seed=k)
    c = O.Config(bits=4, granularity=30, table=tuple(w.table), t_p=w.t_p, log2_block=k, seed=w.seed)
    ctx = runner.context_for(w)
    r = runner.Round(ctx, 1, d, dtype, want_rotated=True)
    x = torch.randn(d, device="cuda") * size
    r.grads[0].copy_(x.to(r.grads[0].dtype))
    r.prepare()
    r.compress(2)
    with_rotated = r.packed[0].clone()
    r.rotated = None
    r.packed[0].zero_()
    r.compress(2)
    torch.cuda.synchronize()
    assert torch.equal(r.packed[0], with_rotated)
    ref = O.thc_round(np.stack([r.grads[0].float().cpu().numpy()]), c, 2, scl=r.scales.cpu().numpy())
    assert np.array_equal(r.packed[0].cpu().numpy(), ref["packed"][0])
