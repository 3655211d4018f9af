"""Blocks held in shared memory (thc_block.cu) at the edges of their tiles: one coordinate more or
less than a tile, several tiles per CTA, clusters (2^15 .. 2^17) and the sizes from which 2^16 and 2^17
blocks take the two-pass pipeline, for fp32 and bf16 gradients: every step against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2302_08545_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,d,n,dtype,bits", [
    (3, 8193, 2, "f32", 4), (5, 16_384 - 31, 2, "bf16", 3), (9, 8191, 3, "f32", 2), (11, 8192 * 3 + 1, 2, "bf16", 4),
    (12, 5_000_001, 2, "f32", 4), (13, 8192, 1, "f32", 8), (13, 5_000_000, 2, "bf16", 1), (14, 16_385, 2, "f32", 4),
    (14, 5_100_003, 2, "f32", 4), (15, 32_769, 3, "bf16", 4), (15, 10_000_019, 1, "f32", 2), (16, 65_535, 2, "f32", 4),
    (16, 1 << 22, 1, "f32", 4), (16, (1 << 22) + 1, 1, "f32", 4), (16, 65_537, 20, "bf16", 4),
    (17, 5 * (1 << 17) - 3, 3, "f32", 4), (17, 8 * (1 << 17) - 3, 2, "bf16", 4),
])
def test_edges_of_tiles_and_clusters(k, d, n, dtype, bits):
    import torch
    from paper_2302_08545_b200 import runner
    g = {1: 5, 2: 3, 3: 12, 4: 30, 8: 255}[bits]
    table = {1: (0, 5), 3: (0, 2, 4, 5, 6, 7, 9, 12)}.get(bits) or W.TABLES[(bits, g)]
    w = W.Workload("cfg4_x" if dtype == "bf16" else "plain", n=n, d=d, log2_block=k, bits=bits, granularity=g,
                   table=tuple(table), in_dtype=dtype, data_seed=k)
    c = O.Config(bits=bits, granularity=g, table=tuple(table), t_p=w.t_p, log2_block=k, seed=w.seed)
    ctx = runner.context_for(w)
    r = runner.Round(ctx, n, d, dtype)
    W.fill_torch(w, r.grads)
    r.run(5)
    tail = torch.zeros_like(r.out)
    ctx.aggregate_decompress(r.packed, d, 5, r.scales, tail, r.workspace)
    ef = [torch.zeros(d, dtype=torch.float32, device=r.device) for _ in range(n)]
    if dtype == "f32":
        ctx.error_feedback(r.grads, r.packed, d, 5, r.scales, ef, r.workspace)
    torch.cuda.synchronize()
    assert ctx.status() == 0
    x = np.stack([t.float().cpu().numpy() for t in r.grads])
    scl = r.scales.cpu().numpy()
    ref = O.thc_round(x, c, 5, scl=scl)
    assert np.array_equal(np.stack([p.cpu().numpy() for p in r.packed]), ref["packed"])
    assert np.array_equal(r.sum_numpy(), ref["sum"])
    assert np.array_equal(r.out.cpu().numpy().view(np.uint32), ref["out"].view(np.uint32))
    assert torch.equal(tail.view(torch.int32), r.out.view(torch.int32))
    if dtype == "f32":
        z = O.unpack(r.packed[n - 1].cpu().numpy(), r.sz.d_pad, bits)
        e = O.error_feedback(x[n - 1], z, scl, c, 5)
        assert np.array_equal(ef[n - 1].cpu().numpy().view(np.uint32), e.view(np.uint32))


@pytest.mark.parametrize("k,d", [(12, 9 * 592 * 8192 + 5), (14, 8 * 296 * 16_384 + 1), (15, 9 * 148 * 32_768 + 3)])
def test_tasks_claimed_from_the_counter(k, d):
    """So many tasks per CTA that every mode claims them; each call of the round needs the counter at zero again."""
    test_edges_of_tiles_and_clusters(k, d, 1, "f32", 4)


def _claimed(tile_log2, n, per_cta=8):
    """A vector of which n have more than per_cta tiles for each CTA that the GPU can hold: they are claimed."""
    import torch
    ctas = torch.cuda.get_device_properties(0).multi_processor_count * (4 if tile_log2 == 13 else 2)
    return (per_cta * ctas // n + 1 << tile_log2) + 5


@pytest.mark.parametrize("k,n", [(12, 3), (15, 2)])
def test_tasks_of_several_workers_claimed_from_the_counter(k, n):
    """Error feedback too: a claimed task is a tile and a worker."""
    test_edges_of_tiles_and_clusters(k, _claimed(13, n) if k == 12 else _claimed(14, n, 20), n, "f32", 4)


def test_exact_range_with_claimed_tasks():
    """The last CTA clears the counter of the claimed tasks and finishes the ranges: twice, against the extremes of
    the rotated coordinates that the call hands out, and compress and error feedback on these ranges."""
    import torch
    from paper_2302_08545_b200 import runner
    k, d = 14, _claimed(14, 1)
    w = W.Workload("plain", n=1, d=d, log2_block=k, bits=4, granularity=30, table=W.TABLES[(4, 30)], data_seed=1)
    ctx = runner.context_for(w, exact_range=True)
    r = runner.Round(ctx, 1, d, want_rotated=True)
    nb = r.sz.nblocks
    assert nb <= 4096                                   # finished in the same launch
    for call in range(2):
        W.fill_torch(w, r.grads, seed_offset=call)
        r.scales.fill_(-7.0)
        r.rotated[0].fill_(float("nan"))
        r.prepare_minmax(call)
        torch.cuda.synchronize()
        assert ctx.status() == 0
        blocks = r.rotated[0].view(nb, 1 << k)
        assert torch.equal(r.scales[:nb], blocks.amin(1)) and torch.equal(r.scales[nb:], blocks.amax(1))
        r.compress(call)
        one = r.packed[0].clone()
        r.quantize_rotated(call)
        assert torch.equal(one, r.packed[0])
    x = r.grads[0].cpu().numpy()
    c = O.Config(bits=4, granularity=30, table=tuple(w.table), t_p=w.t_p, log2_block=k, seed=w.seed)
    lo, hi = O.ranges(x[None], c, 1)
    got = r.scales.cpu().numpy()
    assert np.array_equal(got[:nb].view(np.uint32), lo.view(np.uint32))
    assert np.array_equal(got[nb:].view(np.uint32), hi.view(np.uint32))


def test_skipped_tasks_leave_no_tile_out():
    """The hook for the pipeline's waits has no effect on blocks that claim their tiles from the same counter."""
    import torch
    from paper_2302_08545_b200 import runner
    d = _claimed(13, 1)
    w = W.Workload("plain", n=1, d=d, log2_block=12, bits=4, granularity=30, table=W.TABLES[(4, 30)], data_seed=1)
    ctx = runner.context_for(w)
    r = runner.Round(ctx, 1, d)
    W.fill_torch(w, r.grads)
    r.prepare()
    r.compress(3)
    want = r.packed[0].clone()
    r.packed[0].fill_(0xAA)
    ctx.debug_skip_tasks(3)
    r.compress(3)
    torch.cuda.synchronize()
    assert ctx.status() == 0
    assert torch.equal(r.packed[0], want)
