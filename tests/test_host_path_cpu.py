"""The host side of the entry points on the CPU: the library's own objects
linked with a CUDA runtime that runs nothing (fake_cudart.cpp) and writes down
each launch -- kernel, device, stream, grid, first parameter bytes."""
import ctypes
import os
import subprocess

import pytest

from paper_2607_02630_gb300 import aesoffload as A
from paper_2607_02630_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))
P = 0x7F00_0000_0000  # a payload address (nothing reads it)


class Launch(ctypes.Structure):
    _fields_ = [("device", ctypes.c_int), ("grid", ctypes.c_int), ("block", ctypes.c_int),
                ("programmatic", ctypes.c_int), ("stream", ctypes.c_uint64), ("args", ctypes.c_uint64 * 10),
                ("name", ctypes.c_char * 128)]

    def raw(self, n=80):
        b = bytes(self.args)
        if b"BatchParams" in self.name:
            b = b[:12] + bytes(4) + b[16:]  # padding behind the request count
        return b[:n]


class Host:
    def __init__(self, lib):
        self.lib = lib

    def ctx(self, bits=128):
        h = ctypes.c_void_p()
        assert self.lib.aes_ctx_create(ctypes.byref(h), bytes(32), bits) == A.AES_OK
        return h

    def descs(self, reqs):
        arr = (A.Desc * len(reqs))()
        for d, (ctx, low, src, dst, n) in zip(arr, reqs):
            d.ctx, d.inp, d.out, d.len = ctx, src, dst, n
            d.iv[15] = low
        return arr

    def launches(self):
        out = []
        for i in range(self.lib.fake_launches()):
            out.append(Launch())
            self.lib.fake_launch(i, ctypes.byref(out[-1]))
        return out

    def during(self, f, *args):
        """(status, launches) of one call."""
        self.lib.fake_reset()
        return f(*args), self.launches()


@pytest.fixture(scope="module")
def built(tmp_path_factory):
    B.build()
    nvcc = B._nvcc()
    cuda_inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    so = str(tmp_path_factory.mktemp("fake") / "libaes_fake.so")
    objs = [os.path.join(B.BUILD, n + ".o") for n in ("capi", "batch", "batch_noalloc", "ctr", "tables", "tune")]
    r = subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-Wl,-Bsymbolic", "-I", cuda_inc,
                        os.path.join(HERE, "fake_cudart.cpp")] + objs + ["-o", so], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return so


@pytest.fixture()
def host(built):
    lib = ctypes.CDLL(built)
    vp, sz, ci = ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int
    lib.aes_ctx_create.argtypes = [vp, ctypes.c_char_p, ci]
    lib.aes_ctr.argtypes = [vp, ctypes.c_char_p, vp, vp, sz, vp]
    lib.aes_ctr_ex.argtypes = [vp, ctypes.c_char_p, vp, vp, sz, vp, vp]
    lib.aes_ctr_batch_ex.argtypes = [vp, ci, vp, vp]
    lib.aes_ctr_batch_noalloc.argtypes = [vp, ci, vp]
    lib.aes_batch_plan_create.argtypes = [vp, vp, ci, vp]
    lib.aes_batch_plan_launch.argtypes = [vp, vp]
    lib.aes_batch_plan_destroy.argtypes = [vp]
    lib.aes_batch_plan_bytes.argtypes = [vp]
    lib.aes_batch_plan_bytes.restype = ctypes.c_int64
    lib.aes_tuned_shape.argtypes = [sz, ci, vp]
    lib.fake_launch.argtypes = [ci, vp]
    lib.fake_stream.restype = vp
    lib.fake_other_kernel.argtypes = [vp]
    for f in (lib.fake_news, lib.fake_queries, lib.fake_lookups):
        f.restype = ctypes.c_long
    lib.fake_set_segment.argtypes = [sz]
    lib.fake_cost.argtypes = [ci, ctypes.c_float, ctypes.c_float]
    lib.fake_set_segment(1 << 40)
    lib.fake_set_device(0)
    lib.fake_reset()
    return Host(lib)


@pytest.mark.parametrize("low", [0, 1, 31, 32, 255])
@pytest.mark.parametrize("below", [1, 8, 15])
def test_length_whose_end_wraps_is_no_work(host, low, below):
    """A length within 15 bytes of 2^64 (a negative one passed through an
    unsigned argument) is no whole number of blocks: the calls accept it and
    encrypt nothing, alone and beside a request that has work."""
    n = (1 << 64) - below
    ctx = host.ctx()
    iv = bytes(15) + bytes([low])
    assert host.during(host.lib.aes_ctr, ctx, iv, P, P, n, None) == (A.AES_OK, [])
    for variant, threads in ((1, 512), (2, 128)):
        shape = A.LaunchShape(variant, threads, 1, 0)
        assert host.during(host.lib.aes_ctr_ex, ctx, iv, P, P, n, None, ctypes.byref(shape)) == (A.AES_OK, [])
    assert host.during(host.lib.aes_ctr, ctx, iv, P + 8, P, n, None) == (A.AES_EALIGN, [])
    one = host.descs([(ctx, low, P, P, n)])
    two = host.descs([(ctx, low, P, P, n), (ctx, low, P, P, 100)])
    want = host.during(host.lib.aes_ctr_batch_ex, host.descs([(ctx, low, P, P, 100)]), 1, None, None)[1]
    for variant in (1, 2):
        opts = A.BatchOpts(variant, 0, 0, 0, 0, 0)
        assert host.during(host.lib.aes_ctr_batch_ex, one, 1, None, ctypes.byref(opts)) == (A.AES_OK, [])
        plan = ctypes.c_void_p()
        assert host.lib.aes_batch_plan_create(ctypes.byref(plan), one, 1, ctypes.byref(opts)) == A.AES_OK
        assert host.during(host.lib.aes_batch_plan_launch, plan, None) == (A.AES_OK, [])
        host.lib.aes_batch_plan_destroy(plan)
    for call in (lambda d: host.lib.aes_ctr_batch_ex(d, 2, None, None),
                 lambda d: host.lib.aes_ctr_batch_noalloc(d, 2, None)):
        rc, got = host.during(call, two)
        assert rc == A.AES_OK and [(l.grid, l.raw()) for l in got] == [(l.grid, l.raw()) for l in want]


def _opts(variant=0, tile_blocks=0):
    return ctypes.byref(A.BatchOpts(variant, 0, tile_blocks, 0, 0, 0))


@pytest.mark.parametrize("variant,tile_blocks,limit", [(0, 0, 2048), (1, 256, 256), (1, 7936, 7936), (2, 0, 2048),
                                                       (2, 1024, 1024)])
def test_batches_of_more_than_2_32_tiles_are_refused(host, variant, tile_blocks, limit):
    """A batch or plan of more than 2^32 - 1 tiles is AES_ETOOBIG, in one
    request, over several, and where the count itself would wrap; a request
    that is bad for another reason keeps its own status.  The built-in shape
    counts tiles of 2048 blocks."""
    ctx = host.ctx()
    most = (2 ** 32 - 1) * limit * 16  # bytes, a whole number of tiles
    half = (2 ** 31) * limit * 16
    ok = [[most], [half, most - half], [limit * 16] * 5 + [most - 5 * limit * 16]]
    bad = [[most + 16], [most, 1], [half, half], [1 << 62] * 9, [(1 << 64) - 16] * 3]
    for lens in ok + bad:
        want = A.AES_OK if lens in ok else A.AES_ETOOBIG
        d = host.descs([(ctx, 0, P, P, n) for n in lens])
        rc, got = host.during(host.lib.aes_ctr_batch_ex, d, len(lens), None, _opts(variant, tile_blocks))
        assert rc == want and len(got) == (1 if lens in ok else 0)
        plan = ctypes.c_void_p()
        assert host.lib.aes_batch_plan_create(ctypes.byref(plan), d, len(lens), _opts(variant, tile_blocks)) == want
        assert bool(plan.value) == (want == A.AES_OK)
        host.lib.aes_batch_plan_destroy(plan)
    d = host.descs([(ctx, 0, P, P, 1 << 62), (ctx, 0, P + 8, P, 16)])
    assert host.lib.aes_ctr_batch_ex(d, 2, None, _opts(variant, tile_blocks)) == A.AES_EALIGN


@pytest.mark.parametrize("variant", [1, 2])
def test_plan_stays_on_its_device_and_in_order(host, variant):
    """A plan runs on the device it was created on, whatever device is
    current when it is launched (initialised or not by then) and whichever
    device's stream it is launched into: behind that stream's earlier work,
    before its later work, and behind the plan's last launch."""
    lib = host.lib
    ctx = host.ctx()
    plan = ctypes.c_void_p()
    d = host.descs([(ctx, 7, P, P, 9 << 20)])
    assert lib.aes_batch_plan_create(ctypes.byref(plan), d, 1, _opts(variant)) == A.AES_OK
    streams = [None, lib.fake_stream(0), lib.fake_stream(1), lib.fake_stream(1), lib.fake_stream(0)]
    rc, first = host.during(lib.aes_batch_plan_launch, plan, None)
    assert rc == A.AES_OK and len(first) == 1
    first = first[0]
    lib.fake_reset()
    try:
        last = None
        for current, ready in ((0, True), (1, False), (1, True)):
            lib.fake_set_device(current)
            if ready and current:
                host.ctx()
            for s in streams + streams[::-1]:
                i = lib.fake_launches()
                lib.fake_other_kernel(s)
                assert lib.aes_batch_plan_launch(plan, s) == A.AES_OK
                assert lib.fake_device() == current
                lib.fake_other_kernel(s)
                before, got, after = host.launches()[i:]
                assert (got.name, got.grid, got.raw(40), got.device) == (first.name, first.grid, first.raw(40), 0)
                assert lib.fake_behind(i + 1, i) and lib.fake_behind(i + 2, i + 1)
                assert last is None or lib.fake_behind(i + 1, last)
                last = i + 1
    finally:
        lib.fake_set_device(0)
        lib.aes_batch_plan_destroy(plan)


def test_plan_launches_on_one_stream_stay_overlapped(host):
    """Launches of a plan in a row on one stream wait for no event: each may
    start while the one before drains."""
    ctx = host.ctx()
    plan = ctypes.c_void_p()
    assert host.lib.aes_batch_plan_create(ctypes.byref(plan), host.descs([(ctx, 0, P, P, 5000)]), 1, None) == A.AES_OK
    s = host.lib.fake_stream(0)
    for _ in range(3):
        rc, got = host.during(host.lib.aes_batch_plan_launch, plan, s)
        assert rc == A.AES_OK and [(l.programmatic, l.stream) for l in got] == [(1, s)]
    host.lib.aes_batch_plan_destroy(plan)


@pytest.mark.parametrize("n", [1, 64, 65, 500, 501, 777, 1024])
@pytest.mark.parametrize("empty", [0, 3])
def test_noalloc_allocates_nothing(host, n, empty):
    """aes_ctr_batch_noalloc takes nothing from the host's heap either, at any
    request count, makes the launches the one-shot batch makes, and makes none
    if its last request is bad."""
    ctxs = [host.ctx(b) for b in (128, 192, 256)]
    reqs = [(ctxs[i % 3], i & 255, P + (i << 20), P + (i << 20), 0 if empty and i % empty == 0 else 700 + 37 * i)
            for i in range(n)]
    d = host.descs(reqs)
    host.lib.fake_reset()
    news = host.lib.fake_news()
    assert host.lib.aes_ctr_batch_noalloc(d, n, None) == A.AES_OK
    assert host.lib.fake_news() == news
    got = host.launches()
    rc, want = host.during(host.lib.aes_ctr_batch_ex, d, n, None, None)
    assert rc == A.AES_OK and [(l.name, l.grid, l.raw()) for l in got] == [(l.name, l.grid, l.raw()) for l in want]
    work = sum(1 for r in reqs if r[4])
    assert len(got) == -(-work // 500)
    bad = host.descs(reqs[:-1] + [(ctxs[0], 0, P + 8, P, 16)])
    assert host.during(host.lib.aes_ctr_batch_noalloc, bad, n, None) == (A.AES_EALIGN, [])


@pytest.mark.parametrize("low", [0, 31, 255])
@pytest.mark.parametrize("bits", [128, 256])
def test_short_calls_leave_sms_to_others(host, bits, low):
    """A single call takes one CTA per 4 KiB (8 chunks) it touches, so that
    calls on many streams or beside the resident server do not each fill the
    tables of every SM; a CTA of fewer than 8 warps takes a chunk per warp."""
    ctx = host.ctx(bits)
    iv = bytes(15) + bytes([low])
    for n in (1, 16, 4096, 4097, 16384, 61453, 65536, 262144, 600_000, 1 << 20, 8 << 20):
        rc, got = host.during(host.lib.aes_ctr, ctx, iv, P, P, n, None)
        assert rc == A.AES_OK and len(got) == 1
        chunks = (((low + (n + 15) // 16 - 1) >> 5) - (low >> 5)) + 1
        assert got[0].grid == min(152, -(-chunks // 8))
        for threads in (32, 96, 256, 1024):
            shape = A.LaunchShape(1, threads, 1, 0)
            rc, got = host.during(host.lib.aes_ctr_ex, ctx, iv, P, P, n, None, ctypes.byref(shape))
            assert rc == A.AES_OK and got[0].grid == min(152, -(-chunks // min(8, threads // 32)))
        rc, got = host.during(host.lib.aes_ctr, ctx, iv, P, P, n, None)
        if low == 0:
            s = A.LaunchShape()
            assert host.lib.aes_tuned_shape(n, bits, ctypes.byref(s)) == A.AES_OK and s.ctas == got[0].grid


@pytest.mark.parametrize("n,nbytes", [(1, 100), (8, 512), (8, 5000), (64, 6000), (600, 700), (3, 1 << 20), (1100, 64)])
def test_small_batches_leave_sms_to_others(host, n, nbytes):
    """A batch of short requests takes one T-table CTA per 8 chunks it
    touches, as single calls do; a grid that the caller names is kept while
    every CTA has a chunk."""
    ctx = host.ctx()
    d = host.descs([(ctx, 0, P, P, nbytes)] * n)
    chunks = (nbytes + 511) // 512 * n
    plan = ctypes.c_void_p()
    assert host.lib.aes_batch_plan_create(ctypes.byref(plan), d, n, None) == A.AES_OK
    rc, got = host.during(host.lib.aes_batch_plan_launch, plan, None)
    assert rc == A.AES_OK and [l.grid for l in got] == [min(152, -(-chunks // 8))]
    host.lib.aes_batch_plan_destroy(plan)
    rc, got = host.during(host.lib.aes_ctr_batch_ex, d, n, None, None)
    per_launch = [-(-(n * (k + 1) // len(got) - n * k // len(got)) * chunks // n // 8) for k in range(len(got))]
    assert rc == A.AES_OK and [l.grid for l in got] == [min(152, g) for g in per_launch]
    rc, got = host.during(host.lib.aes_ctr_batch_ex, d, min(n, 64), None, ctypes.byref(A.BatchOpts(1, 512, 256, 40, 0, 1)))
    assert rc == A.AES_OK and got[0].grid == min(40, chunks // n * min(n, 64))


def test_whole_line_counters_take_turns(host):
    """A plan that claims from the whole line (T-tables from 2^18 chunks on,
    the bitsliced kernel always) hands each launch the counter that the one
    before cleared; smaller T-table plans have none."""
    ctx = host.ctx()
    for variant, n, whole in ((1, (1 << 27) - 512, False), (1, 1 << 27, True), (2, 5000, True), (1, 5000, False)):
        d = host.descs([(ctx, 0, P, P, n)])
        plan = ctypes.c_void_p()
        assert host.lib.aes_batch_plan_create(ctypes.byref(plan), d, 1, _opts(variant)) == A.AES_OK
        host.lib.fake_reset()
        for _ in range(3):
            assert host.lib.aes_batch_plan_launch(plan, None) == A.AES_OK
        pairs = [tuple(l.args[8:10]) for l in host.launches()]  # claimed, cleared
        if whole:
            a, b = pairs[0]
            assert a and b and a != b and pairs == [(a, b), (b, a), (a, b)]
        else:
            assert pairs == [(0, 0)] * 3
        host.lib.aes_batch_plan_destroy(plan)


@pytest.mark.parametrize("n", [40, 1000])
@pytest.mark.parametrize("segment", [1 << 40, 64 << 20, 20 << 20, 6 << 20, 4 << 20, 2 << 20])
@pytest.mark.parametrize("stride", [1, 7])
def test_payload_checks_pay_for_themselves(host, n, segment, stride):
    """What a batch spends on its payload pointers, in pointer queries with a
    lookup of an allocation's bounds counted as 12 (about 1 and 0.09 us): next
    to nothing where the payloads share an allocation, and never much more
    than the two queries a request that need no bounds, however the payloads
    are spread over allocations."""
    host.lib.fake_set_segment(segment)
    ctx = host.ctx()
    reqs = []
    for i in range(n):
        at = P + (i * stride % n) * (4 << 20)
        reqs.append((ctx, 0, at, at + (2 << 20), 2000))
    d = host.descs(reqs)
    for call in (lambda: host.lib.aes_ctr_batch_ex(d, n, None, None), lambda: host.lib.aes_ctr_batch_noalloc(d, n, None)):
        host.lib.fake_reset()
        assert call() == A.AES_OK
        cost = host.lib.fake_queries() + 12 * host.lib.fake_lookups()
        assert cost <= 2 * n + 60
        if segment >= n * (4 << 20):
            assert cost <= 60


def test_tuned_tiles_reach_the_built_in_run(host):
    """The tuner's largest tile (4096 blocks) is cut as the built-in shape's:
    T-table tiles of more than half a run are whole runs of 7936 blocks, which
    leave no short run behind; smaller ones and the bitsliced kernel's stay."""
    ctx = host.ctx()
    d = host.descs([(ctx, 0, P, P, 64 << 20)])

    def tile(variant, tile_blocks):
        rc, got = host.during(host.lib.aes_ctr_batch_ex, d, 1, None, _opts(variant, tile_blocks))
        assert rc == A.AES_OK
        return got[0].args[3]

    run = tile(0, 0)
    assert [tile(1, t) for t in (4096, 7936, 8192)] == [run] * 3
    assert tile(1, 16384) == 2 * run
    assert [tile(1, t) * 31 for t in (256, 1024, 2048, 3840)] == [run, 4 * run, 8 * run, 15 * run]
    assert tile(2, 4096) == 2 * tile(2, 2048) == 4 * tile(2, 1024)


def test_single_call_tuner_times_calls_in_a_row(host):
    """aes_autotune times each candidate as calls in a row, whose set-up
    overlaps, and keeps the built-in shape where no other is faster by more
    than the launches of one shape differ."""
    def tuned(n):
        s = A.LaunchShape()
        assert host.lib.aes_tuned_shape(n, 256, ctypes.byref(s)) == A.AES_OK
        return s.variant, s.threads

    def costs(**us):  # CTA size -> (us of a launch after an event, of one in a row)
        host.lib.fake_clear_costs()
        for k, (first, next_) in us.items():
            host.lib.fake_cost(int(k[1:]), first, next_)

    sizes = (4096, 1 << 20, 4 << 20, 64 << 20)
    costs(t128=(90, 90), t256=(5, 6), t512=(10, 4), t768=(9, 6), t1024=(9, 6))
    assert host.lib.aes_autotune(None) == A.AES_OK
    assert [tuned(n) for n in sizes] == [(1, 512)] * 4
    costs(t128=(90, 90), t256=(9.9, 4.97), t512=(10, 5), t768=(9.9, 4.96), t1024=(9.95, 4.99))
    assert host.lib.aes_autotune(None) == A.AES_OK
    assert [tuned(n) for n in sizes] == [(1, 512)] * 4
    costs(t128=(90, 90), t256=(9, 5), t512=(10, 5), t768=(9, 3), t1024=(9, 3.5))
    assert host.lib.aes_autotune(None) == A.AES_OK
    assert [tuned(n) for n in sizes] == [(1, 768)] * 4
    costs(t128=(90, 90), t256=(9, 5), t512=(10, 3), t768=(9, 4), t1024=(9, 4))
    assert host.lib.aes_autotune(None) == A.AES_OK
    assert [tuned(n) for n in sizes] == [(1, 512)] * 4
    host.lib.fake_clear_costs()
