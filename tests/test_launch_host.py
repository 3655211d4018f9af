"""Host code of the launching calls on a fake CUDA runtime (tests/fake_cudart.c): which kernel a call launches,
with what grid and shared memory.  Runs without a GPU, in child processes; no kernel is executed."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# What a child process has at hand: contexts, buffers that are only addresses, and the log of launches.
PRELUDE = """
import ctypes, sys
sys.path.insert(0, {root!r})
from paper_2302_08545_b200 import thc, workloads as W
fake = ctypes.CDLL(None)
fake.fake_log.restype = ctypes.c_char_p

class Space:
    nbytes = 1 << 40
    def data_ptr(self):
        return 1 << 32

ws = Space()
buf = [(i + 1) << 20 for i in range(64)]

def context(k, **kw):
    return thc.Context(**dict(dict(bits=4, granularity=30, table=W.TABLES[(4, 30)], t_p=2.0, log2_block=k, seed=1), **kw))

def log():
    # [kind, kernel, numbers...] per line since the last call
    rows = [line.split() for line in fake.fake_log().decode().splitlines()]
    return [row[:2] + [int(v) for v in row[2:]] for row in rows]

def kernels():
    return ["block" if "block_kernel" in r[1] else "pipeline" if "pipeline_kernel" in r[1] else r[1]
            for r in log() if r[0] == "launch"]

def transforms(c, d, n=2):
    x = buf[:n]
    calls = [lambda: c.compress(x, d, 0, buf[0], x, ws, stream=0), lambda: c.decompress(buf[0], n, d, 0, buf[1], buf[2], ws, stream=0),
             lambda: c.aggregate_decompress(x, d, 0, buf[0], buf[1], ws, stream=0)]
    return calls + [lambda: c.error_feedback(x, x, d, 0, buf[0], x, ws, stream=0)]

"""


@pytest.fixture(scope="module")
def child(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fake") / "fake_cudart.so")
    subprocess.run([os.environ.get("CC", "gcc"), "-O1", "-fPIC", "-shared", "-I/usr/local/cuda/include", "-o", so,
                    os.path.join(ROOT, "tests", "fake_cudart.c")], check=True)

    def run(code):
        res = subprocess.run([sys.executable, "-c", PRELUDE.format(root=ROOT) + code], capture_output=True, text=True,
                             env=dict(os.environ, LD_PRELOAD=so), timeout=300)
        assert res.returncode == 0, res.stderr[-3000:]
        return res.stdout
    return run


@pytest.mark.parametrize("k", [3, 12, 13, 14])
def test_skipped_tasks_never_send_a_small_block_to_the_pipeline(child, k):
    child(f"""
k = {k}
c = context(k)
m = context(k, range_mode=1)
for call in transforms(c, 1 << 15) + [lambda: m.prepare_minmax(buf[:2], 1 << 15, 0, buf[0], ws, stream=0)]:
    for ctx in (c, m):
        ctx.debug_skip_tasks(1)
    call()
    assert kernels() == ["block"], k
""")


@pytest.mark.parametrize("k", [3, 12, 14])
def test_skipped_tasks_leave_the_counter_of_claimed_tiles_alone(child, k):
    """Launches with many tiles claim them from a counter of the context: all of them, from the first on."""
    child(f"""
k = {k}
fake.fake_device_block.restype = ctypes.c_void_p
size = ctypes.c_size_t()
for mode in (0, 1):
    c = context(k, range_mode=mode)
    block = lambda: ctypes.string_at(fake.fake_device_block(ctypes.byref(size)), size.value)
    before = block()
    assert before[128:132] == bytes(4)
    c.debug_skip_tasks(3)
    for d in (5, 1 << 25):
        c.compress(buf[:3], d, 0, buf[0], buf[:3], ws, stream=0)
    assert [r[6] for r in log() if r[0] == "launch"] == [0, 1]
    assert block() == before
c = context(20)
c.debug_skip_tasks(3)
assert block()[128:132] == bytes([3, 0, 0, 0])
""")


@pytest.mark.parametrize("k", [15, 16, 17])
def test_skipped_tasks_take_the_pipeline_once(child, k):
    child(f"""
k = {k}
c = context(k)
m = context(k, range_mode=1)
for ctx, call in [(c, f) for f in transforms(c, 3 << k)] + [(m, lambda: m.prepare_minmax(buf[:2], 3 << k, 0, buf[0], ws, stream=0))]:
    call()
    assert kernels() == ["block"]
    ctx.debug_skip_tasks(1)
    call()
    call()
    assert kernels() == ["pipeline", "block"]
""")


def test_shared_memory_limit_is_set_once_per_kernel_and_never_lowered(child):
    """More kernels than any process of the other tests uses, each with launches of several sizes (tables of
    different granularity), largest first: a limit that is set again for a smaller launch would let another
    thread's larger one fail."""
    out = child("""
limit, sets, largest = {}, {}, {}
for size in (255, 60, 255):
    for k in (3, 9, 14, 15, 16, 17, 20, 22):
        for bits in (1, 2, 3, 4, 8):
            levels = 1 << bits
            for g in {size, levels - 1}:
                table = list(range(levels - 1)) + [g]
                if g < levels - 1:
                    continue
                for dtype in (0, 1):
                    for acc in (0, 32):
                        c = context(k, bits=bits, granularity=g, table=table, in_dtype=dtype, acc_bits=acc)
                        for call in transforms(c, 1 << max(k, 15))[:4 - dtype]:
                            call()
                        for row in log():
                            if row[0] == "attr":
                                sets[row[1]] = sets.get(row[1], 0) + 1
                                limit[row[1]] = row[2]
                            elif row[4] > 48 << 10:
                                largest[row[1]] = max(row[4], largest.get(row[1], 0))
                                assert limit[row[1]] >= row[4], row
assert len(limit) > 180, len(limit)
print(len(limit), max(sets.values()))
assert max(sets.values()) == 1
assert all(limit[f] >= largest[f] for f in largest)
""")
    assert out.split()[1] == "1"


@pytest.mark.parametrize("k,g,ctas", [
    (3, 30, 592), (12, 30, 592), (12, 166, 592), (12, 167, 444), (12, 255, 444), (3, 255, 296), (14, 255, 296), (15, 255, 296),
    (16, 166, 8 * 71), (16, 255, 8 * 48),
])
def test_grid_of_the_block_kernel_is_what_the_gpu_holds(child, k, g, ctas):
    """The CTAs walk over the tasks in a fixed stride: one that has to wait for another to end doubles the time."""
    child(f"""
k, g, ctas = {k}, {g}, {ctas}
c = context(k, granularity=g, table=W.TABLES[(4, 30)][:15] + (g,), workers=1)
d = 64 << 16 if k == 16 else 1 << 26
for _ in range(2):
    c.compress(buf[:1], d, 0, buf[0], buf[:1], ws, stream=0)
    assert [r[2] for r in log() if r[0] == "launch"] == [min(ctas, 8 * 64) if k == 16 else ctas]
    c.decompress(buf[0], 1, d, 0, buf[1], buf[2], ws, stream=0)     # no table
    assert [r[2] for r in log() if r[0] == "launch"] == [8 * 64 if k == 16 else 296 if k in (14, 15) else 592]
    c.compress(buf[:1], 5, 0, buf[0], buf[:1], ws, stream=0)
    assert [r[2] for r in log() if r[0] == "launch"] == [8 if k == 16 else 2 if k == 15 else 1]                                  # one tile or cluster
""")


@pytest.mark.parametrize("k,last", [(16, 64), (17, 15)])
def test_largest_number_of_blocks_held_in_clusters(child, k, last):
    """Up to `last` blocks over all workers are held in clusters, more take the pipeline; scales + compress is one
    launch only where compress takes the pipeline."""
    child(f"""
k, last = {k}, {last}
c = context(k)
for blocks in (1, last, last + 1):
    for n in (1, blocks):
        d = blocks // n << k
        x = buf[:1] * n
        want = ["block" if blocks <= last else "pipeline"]
        if n <= 64:
            c.compress(x, d, 0, buf[0], x, ws, stream=0)
            assert kernels() == want, (blocks, n)
            c.error_feedback(x, x, d, 0, buf[0], x, ws, stream=0)
            assert kernels() == want, (blocks, n)
            fused = c.sizes(d, n).fused_scales
            assert not fused or want == ["pipeline"]
            c.prepare_compress(x, d, 0, buf[0], x, ws, stream=0)
            assert len(kernels()) == 2 - fused
        if n == 1:
            c.decompress(buf[0], 1, d, 0, buf[1], buf[2], ws, stream=0)
            assert kernels() == want, blocks
""")


@pytest.mark.parametrize("k,n,dtype,small,large", [
    (7, 2, 0, 2, 2), (8, 1, 0, 1, 1), (8, 8, 1, 1, 1), (8, 9, 0, 2, 2), (12, 5, 1, 1, 1), (13, 3, 1, 1, 2), (13, 8, 0, 1, 1),
    (14, 6, 0, 1, 1), (14, 7, 0, 1, 2), (14, 1, 1, 1, 2), (14, 9, 1, 2, 2), (15, 2, 0, 2, 2),
])
def test_scales_and_compress_of_blocks_in_shared_memory(child, k, n, dtype, small, large):
    """One launch, in clusters of one CTA per worker, exactly where thc_sizes says so; what the two calls refuse is
    refused there too, before anything is launched."""
    child(f"""
k, n, dtype, small, large = {k}, {n}, {dtype}, {small}, {large}
c = context(k, in_dtype=dtype)
x = buf[:n]
for d, launches in ((5, small), (1 << 15, small), (20_000_003, large)):
    c.prepare_compress(x, d, 0, buf[0], x, ws, stream=0)
    rows = [r for r in log() if r[0] == "launch"]
    assert len(rows) == launches and c.sizes(d, n).fused_scales == (launches == 1)
    if launches == 1:
        assert "block_kernel" in rows[0][1] and rows[0][5] == n and rows[0][2] % n == 0
class Short(Space):
    nbytes = c.sizes(5, n).workspace_bytes - 1
m = context(k, range_mode=1)
for ctx, grads, scales, packed, space in [(c, [8] * n, buf[0], x, ws), (c, x, buf[0], [0] * n, ws), (c, x, 0, x, ws), (c, x, buf[0], x, Short()),
                                          (m, x, buf[0], x, ws)]:
    try:
        ctx.prepare_compress(grads, 5, 0, scales, packed, space, stream=0)
        assert False
    except thc.ThcError:
        pass
    assert small == 2 or log() == []
    log()
""")


@pytest.mark.parametrize("k,d,n,launches", [
    (12, 1 << 24, 32, 1), (14, 1 << 20, 16, 1), (14, 1 << 20, 17, 2), (15, 1 << 20, 17, 2), (16, 1 << 20, 32, 1), (16, 1 << 24, 13, 2),
    (17, 1 << 20, 2, 2), (17, 1 << 23, 12, 1), (20, 1 << 22, 12, 1), (20, 1 << 22, 13, 2),
])
def test_one_call_tail_is_two_launches_where_these_are_faster(child, k, d, n, launches):
    """With the sums wanted; without them it is one launch for 4-bit indices."""
    child(f"""
c = context({k}, workers=32)
for total, want in ((buf[2], {launches}), (None, 1)):
    c.aggregate_decompress(buf[:{n}], {d}, 0, buf[0], buf[1], ws, total=total, stream=0)
    assert len(kernels()) == want
""")


@pytest.mark.parametrize("k,d,n,launches", [
    (14, 1 << 24, 24, 1), (14, 1 << 24, 25, 2), (14, 1 << 22, 32, 1), (15, 1 << 22, 32, 1), (15, 1 << 24, 17, 1), (15, 1 << 24, 32, 2),
    (17, 9 << 17, 2, 2), (17, 10 << 17, 13, 1), (17, 10 << 17, 14, 2), (18, 1 << 25, 14, 1), (18, 1 << 25, 15, 2),
    (22, 1 << 24, 13, 2), (22, 1 << 25, 18, 1), (22, 1 << 25, 19, 2),
])
def test_one_call_tail_by_the_number_of_tiles(child, k, d, n, launches):
    child(f"""
c = context({k}, workers=32)
c.aggregate_decompress(buf[:{n}], {d}, 0, buf[0], buf[1], ws, total=buf[2], stream=0)
assert len(kernels()) == {launches}
""")


@pytest.mark.parametrize("k,bits,d,n", [(17, 4, 1 << 20, 2), (20, 4, 1 << 22, 13), (20, 2, 1 << 22, 2), (15, 4, 1 << 20, 17)])
def test_one_call_tail_refuses_before_it_launches(child, k, bits, d, n):
    """Where it runs the two calls too: a missing, misaligned or short workspace leaves the caller's sums alone."""
    child(f"""
g = {{2: 3, 4: 30}}[{bits}]
c = context({k}, bits={bits}, granularity=g, table=W.TABLES[({bits}, g)], workers=32)
def space(nbytes, address=1 << 32):
    s = Space()
    s.nbytes, s.data_ptr = nbytes, lambda: address
    return s
sz = c.sizes({d}, 1)
enough = sz.workspace_bytes
log()
for total in (buf[2], None):
    for ws in (space(0, 0), space(enough, 8), space(255)):
        try:
            c.aggregate_decompress(buf[:{n}], {d}, 0, buf[0], buf[1], ws, total=total, stream=0)
            assert False
        except thc.ThcError:
            pass
        assert log() == []
    c.aggregate_decompress(buf[:{n}], {d}, 0, buf[0], buf[1], space(enough), total=total, stream=0)
    assert len(kernels()) == (2 if total or {bits} == 2 else 1)
""")


@pytest.mark.parametrize("k,n,mode,tasks_to_a_cta,claims", [
    (12, 1, "compress", 5, 0), (12, 3, "compress", 5.1, 1), (14, 1, "compress", 8, 0), (14, 2, "compress", 8.1, 1),
    (12, 3, "error_feedback", 8, 0), (12, 3, "error_feedback", 8.1, 1), (14, 1, "prepare_minmax", 8, 0), (14, 1, "prepare_minmax", 8.1, 1),
    (12, 1, "decompress", 8, 0), (12, 1, "decompress", 8.1, 1), (15, 2, "compress", 10, 0), (15, 1, "compress", 10.1, 1),
    (15, 1, "prepare_minmax", 10, 0), (15, 1, "prepare_minmax", 10.1, 1),
    (15, 2, "error_feedback", 20, 0), (15, 2, "error_feedback", 20.1, 1), (15, 1, "decompress", 20.1, 1),
    (11, 2, "prepare_compress", 6.1, 1), (12, 1, "prepare_compress", 6, 0), (14, 4, "prepare_compress", 8.1, 1), (8, 8, "prepare_compress", 6.1, 1),
])
def test_which_launches_claim_their_tasks(child, k, n, mode, tasks_to_a_cta, claims):
    child(f"""
k, n, mode = {k}, {n}, "{mode}"
tile = 13 if k <= 13 else max(k, 14)                                # of a CTA, or of a cluster
ctas = 592 if k <= 13 else 296 if k == 14 else 148
c = context(k, workers=n, range_mode=int(mode == "prepare_minmax"))
x = buf[:n]
d = int({tasks_to_a_cta} * ctas / n) << tile
assert d * n >> tile == int({tasks_to_a_cta} * ctas / n) * n
dict(compress=lambda: c.compress(x, d, 0, buf[0], x, ws, stream=0),
     prepare_compress=lambda: c.prepare_compress(x, d, 0, buf[0], x, ws, stream=0),
     prepare_minmax=lambda: c.prepare_minmax(x, d, 0, buf[0], ws, stream=0),
     decompress=lambda: c.decompress(buf[0], n, d, 0, buf[1], buf[2], ws, stream=0),
     error_feedback=lambda: c.error_feedback(x, x, d, 0, buf[0], x, ws, stream=0))[mode]()
rows = [r for r in log() if r[0] == "launch" and "block_kernel" in r[1]]
assert len(rows) == 1 and rows[0][6] == {claims}, rows
""")
