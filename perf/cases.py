"""The work a user of this library has it do, as cases that can be timed and compared.

A case is one pass through the public entry points on buffers that the program keeps between
steps, as a training loop does: `prepare` makes the context, the buffers and seeded gradients,
`run` is one pass, and its outputs are the buffers that the pass wrote.  Four kinds of pass:

  round     n workers' gradients on one GPU through the whole round: scales + compress,
            aggregate, decompress (runner.Round.run, the step that bench.py times)
  feedback  the same with error feedback: scales + compress, the residuals of all workers, these
            added to the next gradients, and the aggregated estimate in one call
  rank      what one rank's GPU does in the data-parallel round: its own scales and indices, the
            sums of its block range over all ranks' indices, the estimate of the whole vector
            (the collectives between these steps are not part of it)
  range     the exact-range form (Algorithm 1's preliminary stage): range of the rotated
            coordinates, quantisation of these, aggregate, decompress

Sizes, index widths, tables and value distributions are those of the benchmark configurations
(workloads.py), the d x b x n sweep, the granularity study and the tests.
"""
import math

import torch

from paper_2302_08545_b200 import data_parallel, runner, tables, workloads

# (bits, granularity) pairs in use: the sweep's, the prototype's table and the study's 3-bit one.
GRANULARITY = {1: 1, 2: 3, 3: 14, 4: 30, 8: 255}

# A workload's name selects its value distribution in workloads.fill_torch.
DISTRIBUTION = {"outliers": "cfg1", "segments": "cfg2", "laplace": "cfg3", "student": "cfg4", "normal": "plain"}


def _case(kind, n, d, k, bits, dtype="f32", values="normal", **more):
    return dict(more, kind=kind, n=n, d=d, log2_block=k, bits=bits, dtype=dtype, values=values)


def listed():
    return [
        # the smallest calls: a bias or normalisation layer's gradient, a few blocks of 2^8
        _case("round", 2, 3_000, 8, 4, name="small_layer"),
        # benchmark configuration 1: one 2^16 block per worker, bound by latency
        _case("round", 4, 65_536, 16, 4, values="outliers", name="cfg1_one_block"),
        # a bucket of small layers in small blocks (the whole block fits one SM)
        _case("round", 8, 3_000_001, 12, 4, name="small_blocks"),
        # benchmark configuration 2: ResNet-50 sized vectors in 4 MB partitions, bench.py's default
        _case("round", 8, 25_557_032, 20, 4, values="segments", name="cfg2_resnet50"),
        # benchmark configuration 3: VGG-16 sized vectors, two bits
        _case("round", 8, 138_357_544, 20, 2, values="laplace", name="cfg3_vgg16_b2"),
        # benchmark configuration 4, the largest: GPT-2-medium sized bf16 vectors in 2^22 blocks
        _case("round", 16, 355_000_000, 22, 4, dtype="bf16", values="student", name="cfg4_gpt2m_bf16"),
        # a point of the d x b x n sweep: many workers, 16-bit sums
        _case("round", 32, 1 << 22, 20, 4, name="sweep_32_workers"),
        # a point of the granularity study: ten workers, three bits
        _case("round", 10, 1 << 22, 20, 3, name="study_b3"),
        # training with error feedback, a ragged vector in 2^18 blocks
        _case("feedback", 4, 7_000_003, 18, 4, values="laplace", name="feedback"),
        # one rank of an eight-rank job on configuration 2's vector
        _case("rank", 8, 25_557_032, 20, 4, values="segments", name="rank_of_8"),
        # one rank of a two-rank job on a bf16 bucket, one bit
        _case("rank", 2, 1_500_007, 17, 1, dtype="bf16", values="student", name="rank_of_2_bf16_b1"),
        # uniform quantisation on the exact range, eight bits
        _case("range", 4, (1 << 22) + 99, 16, 8, name="exact_range_b8"),
    ]


def draw(rng):
    """A case of the same ranges: 1 to 32 workers, a thousand coordinates to a few hundred
    million (at most 2^31 over all workers), blocks of 2^8 .. 2^22 not much longer than the
    vector, every index width and both input types where the entry points take them."""
    kind = rng.choice(["round", "round", "round", "feedback", "rank", "range"])
    n = max(1, min(20 if kind == "feedback" else 32, round(2 ** rng.uniform(0.0, 5.0))))
    workers = 1 if kind == "rank" else n
    d = int(2 ** rng.uniform(10.0, min(28.0, 31.0 - math.log2(workers)))) + rng.randrange(0, 97)
    k = rng.choice([k for k in (8, 10, 12, 13, 14, 15, 16, 17, 18, 19, 20, 20, 20, 21, 22) if (1 << k) <= 2 * d])
    bits = rng.choice([1, 2, 3, 4, 4, 4, 8])
    dtype = rng.choice(["f32", "f32", "bf16"]) if kind in ("round", "rank") else "f32"
    values = "student" if dtype == "bf16" else rng.choice(["outliers", "laplace", "normal"])
    return _case(kind, n, d, k, bits, dtype=dtype, values=values)


def _workload(case):
    bits, g = case["bits"], GRANULARITY[case["bits"]]
    if bits == 3:
        table, t_p = tables.optimal_table(bits, g, 1 / 1024)[0], tables.t_p(1 / 1024)
    else:
        table, t_p = workloads.TABLES[(bits, g)], workloads.T_P["1/32"]
    return workloads.Workload(DISTRIBUTION[case["values"]], n=case["n"], d=case["d"], log2_block=case["log2_block"],
                              bits=bits, granularity=g, table=tuple(table), t_p=t_p, in_dtype=case["dtype"],
                              data_seed=1000)


def prepare(case, seed):
    w = _workload(case)
    kind = case["kind"]
    ctx = runner.context_for(w, exact_range=kind == "range")
    state = {"kind": kind, "ctx": ctx, "w": w, "rnd": seed % 1000}
    if kind == "rank":
        dev = torch.device("cuda", torch.cuda.current_device())
        gen = torch.Generator(device=dev)
        gen.manual_seed(seed)
        grad = torch.empty(w.d, dtype=torch.bfloat16 if w.in_dtype == "bf16" else torch.float32, device=dev)
        workloads.fill_torch(w, [grad], seed_offset=seed * 64)
        ops = data_parallel.CudaOps(ctx, w.d, dev)
        first, count = data_parallel.block_ranges(w.nblocks, w.n)[0]
        coords = count * w.block
        # what the collectives would have delivered: every rank's indices of the own range, and
        # the sums of all ranges
        recv = torch.randint(0, 256, (w.n * coords * w.bits // 8,), generator=gen, device=dev, dtype=torch.uint8)
        most = w.n * w.granularity
        sums = torch.randint(0, most + 1, (w.d_pad,), generator=gen, device=dev, dtype=torch.int32)
        if w.acc_bits == 8:
            total = sums.to(torch.uint8)
        elif w.acc_bits == 16:
            total = sums.to(torch.int16).view(torch.uint8)
        else:
            total = sums.view(torch.uint8)
        state.update(ops=ops, grad=grad, slices=list(recv.split(coords * w.bits // 8)), coords=coords, total=total)
        return state
    r = runner.Round(ctx, w.n, w.d, w.in_dtype, want_rotated=kind == "range")
    workloads.fill_torch(w, r.grads, seed_offset=seed * 64)
    state["round"] = r
    if kind == "feedback":
        state["ef"] = [torch.zeros_like(g) for g in r.grads]
        state["next"] = [torch.zeros_like(g) for g in r.grads]
    return state


def run(state):
    kind, rnd = state["kind"], state["rnd"]
    if kind == "rank":
        ops, w = state["ops"], state["w"]
        scales = ops.local_scales(state["grad"])
        packed = ops.compress(state["grad"], rnd, scales, 0)
        part = ops.aggregate(state["slices"], state["coords"])
        out = ops.decompress(state["total"], w.n, rnd, scales)
        return {"scales": scales, "packed": packed, "part": part, "out": out}
    r = state["round"]
    if kind == "round":
        r.run(rnd, fused=True)
        return {"scales": r.scales, "packed": r.packed, "total": r.total, "out": r.out}
    if kind == "range":
        r.prepare_minmax(rnd)
        r.quantize_rotated(rnd)
        r.aggregate()
        r.decompress(rnd)
        return {"scales": r.scales, "packed": r.packed, "total": r.total, "out": r.out}
    ctx = state["ctx"]
    r.prepare_compress(rnd)
    ctx.error_feedback(r.grads, r.packed, r.d, rnd, r.scales, state["ef"], r.workspace)
    ctx.accumulate_error(state["next"], state["ef"], r.d)
    r.aggregate_decompress(rnd)
    return {"scales": r.scales, "packed": r.packed, "ef": state["ef"], "next": state["next"], "out": r.out}


def work(case):
    w = _workload(case)
    kind, n, d, dp, k = case["kind"], w.n, w.d, w.d_pad, w.log2_block
    s_in = 2 if w.in_dtype == "bf16" else 4
    scales = 4 * w.nblocks * (2 if kind == "range" else 1)
    packed, total = dp * w.bits // 8, dp * w.acc_bits // 8
    # per coordinate: k additions of the transform; about 20 for sign, scaling, the random bits,
    # the quantiser and packing; about 6 for estimate, sign and scaling on the way back
    forward, back = k + 20, k + 6
    if kind == "rank":
        coords = data_parallel.block_ranges(w.nblocks, n)[0][1] * w.block
        return {"bytes": s_in * d + scales + packed + n * coords * w.bits // 8 + coords * w.acc_bits // 8 + total + 4 * d,
                "flops": dp * forward + n * coords + dp * back}
    if kind == "round":
        return {"bytes": n * (s_in * d + packed) + scales + total + 4 * d, "flops": n * dp * forward + n * dp + dp * back}
    if kind == "range":
        # the rotated coordinates are an intermediate result
        return {"bytes": n * (s_in * d + packed) + scales + total + 4 * d, "flops": n * dp * forward + n * dp + dp * back}
    # gradients in, indices out, residuals out, the next gradients read and written, estimate out
    return {"bytes": n * (4 * d + packed + 4 * d + 8 * d) + scales + 4 * d,
            "flops": n * dp * (forward + back) + n * d + n * dp + dp * back}


def tolerance(case):
    # fp32 butterflies and an fp32 estimate; indices and sums are whole numbers, where a scale
    # that rounds the other way may move a coordinate that lies on a rounding threshold
    return {"rel": 1e-5, "differ": 1e-6}
