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


@pytest.mark.parametrize("k,d,n,dtype,bits", [
    (8, 8193, 3, "f32", 4), (8, 255, 1, "f32", 1), (9, 16_384 + 511, 8, "bf16", 3), (10, 3000, 5, "f32", 2),
    (11, 8192 * 5 - 2048, 2, "bf16", 8), (12, 8 * 8192 + 4097, 6, "f32", 4), (12, 20_000_003, 1, "f32", 4),
    (12, 2_500_000, 8, "f32", 4), (13, 8191, 7, "f32", 8), (13, 1_000_001, 4, "bf16", 4), (14, 16_385, 8, "f32", 3),
    (14, 5_000_000, 3, "f32", 4), (14, 4_000_001, 1, "bf16", 1),
])
def test_blocks_in_shared_memory_one_launch_equals_the_two_calls(k, d, n, dtype, bits):
    """One tile, ragged last tiles, several tasks per cluster and claimed ones, every number of workers it takes: the
    scales within one ulp of thc_prepare's (fp64 sums in another order), the indices those of compress on them.  A
    block of zeros, one with an infinity and one with a NaN in the last worker's gradient, and a tiny value."""
    import torch
    from paper_2302_08545_b200 import runner
    g = {1: 5, 2: 3, 3: 12, 4: 30, 8: 255}[bits]
    table = {1: (0, 5), 3: (0, 2, 4, 5, 6, 7, 9, 12)}.get(bits) or W.TABLES[(bits, g)]
    w = W.Workload("cfg4_x" if dtype == "bf16" else "plain", n=n, d=d, log2_block=k, bits=bits, granularity=g,
                   table=tuple(table), in_dtype=dtype, data_seed=k)
    ctx = runner.context_for(w)
    r = runner.Round(ctx, n, d, dtype)
    assert r.sz.fused_scales == 1
    nblk = r.sz.nblocks
    for call in range(3):
        W.fill_torch(w, r.grads, seed_offset=call)
        r.grads[0][0] = 1e-30
        if nblk > 4 and call:
            for t in r.grads:
                t[1 << k: 2 << k] = 0.0
            r.grads[n - 1][(2 << k) + 7] = float("inf")
            r.grads[n - 1][(3 << k) + (1 << k) - 1] = float("nan")
        r.prepare_compress(call)
        torch.cuda.synchronize()
        flags = ctx.status()
        s, p = r.scales.clone(), [t.clone() for t in r.packed]
        r.scales.fill_(-1.0)
        for t in r.packed:
            t.fill_(0xAA)
        r.prepare()
        torch.cuda.synchronize()
        assert flags == ctx.status()
        assert torch.isfinite(s).all()
        assert (s.view(torch.int32) - r.scales.view(torch.int32)).abs().max().item() <= 1
        r.scales.copy_(s)
        r.compress(call)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(p, r.packed))


@pytest.mark.parametrize("k,n,dtype,bits", [(14, 1, "f32", 4), (14, 4, "f32", 2), (11, 2, "bf16", 3), (8, 8, "f32", 4)])
def test_blocks_in_shared_memory_with_claimed_clusters(k, n, dtype, bits):
    """More than eight (tiles of 2^13: six) tasks for each cluster that the GPU can hold."""
    import torch
    ctas = torch.cuda.get_device_properties(0).multi_processor_count * (2 if k == 14 else 4)
    tile_log2, per_cluster = (14, 8) if k == 14 else (13, 6)
    d = (per_cluster * ctas // n + 1 << tile_log2) + 5
    test_blocks_in_shared_memory_one_launch_equals_the_two_calls(k, d, n, dtype, bits)


@pytest.mark.parametrize("k,d,n,dtype", [(8, 8192 * 3 + 77, 3, "f32"), (12, 100_003, 2, "bf16"), (14, 50_000, 5, "f32")])
def test_blocks_in_shared_memory_rotated_and_worker_base(k, d, n, dtype):
    """The rotated coordinates, and the random numbers of workers that do not begin at 0."""
    import torch
    from paper_2302_08545_b200 import runner
    w = W.Workload("plain", n=n, d=d, log2_block=k, bits=4, granularity=30, table=W.TABLES[(4, 30)], in_dtype=dtype, data_seed=k)
    ctx = runner.context_for(w)
    r = runner.Round(ctx, n, d, dtype, want_rotated=True)
    assert r.sz.fused_scales == 1
    W.fill_torch(w, r.grads)
    got = []
    for base in (5, 0):
        for t in r.rotated:
            t.fill_(float("nan"))
        ctx.prepare_compress(r.grads, d, 2, r.scales, r.packed, r.workspace, rotated=r.rotated, worker_base=base)
        p, rot = [t.clone() for t in r.packed], [t.clone() for t in r.rotated]
        for t in r.packed:
            t.fill_(0xAA)
        ctx.compress(r.grads, d, 2, r.scales, r.packed, r.workspace, rotated=r.rotated, worker_base=base)
        torch.cuda.synchronize()
        assert ctx.status() == 0
        assert all(torch.equal(a, b) for a, b in zip(p, r.packed))
        assert all(torch.equal(a.view(torch.int32), b.view(torch.int32)) for a, b in zip(rot, r.rotated))
        got.append(p[0])
    assert not torch.equal(got[0], got[1])
