"""Batched varlen AES-CTR (one persistent launch, work-stealing tiles) and its
CUDA-graph plans, bit-exact against the CPU oracle request by request."""
import numpy as np
import pytest

import oracle
from paper_2607_02630_gb300 import workloads as W

from gpu_util import iv_plus, iv_with_low, set_batch_shape, to_dev, to_host

pytestmark = pytest.mark.gpu


def make_requests(torch, aes, g, lengths, bits_list, kinds=None):
    """Requests packed into one device arena at 256-byte aligned offsets."""
    pad = [(n + 255) // 256 * 256 + 256 for n in lengths]
    offs = np.concatenate([[0], np.cumsum(pad)[:-1]]).astype(np.int64)
    total = int(sum(pad))
    payload = W.random_bytes(g, total)
    src = to_dev(torch, payload)
    dst = to_dev(torch, np.zeros(0, np.uint8), pad=total)
    reqs, meta = [], []
    for i, (n, bits) in enumerate(zip(lengths, bits_list)):
        key = W.random_bytes(g, bits // 8)
        iv = iv_with_low(g, kinds[i] if kinds else "random")
        ctx = aes.Context(key.tobytes(), bits)
        o = int(offs[i])
        reqs.append((ctx, iv.tobytes(), src.data_ptr() + o, dst.data_ptr() + o, int(n)))
        meta.append((key, bits, iv, o, int(n)))
    return reqs, meta, payload, src, dst


def check_all(torch, meta, payload, dst, ncpu):
    torch.cuda.synchronize()
    out = to_host(dst)
    for key, bits, iv, o, n in meta:
        want = oracle.ctr_mt(key, bits, iv, payload[o: o + n], ncpu)
        np.testing.assert_array_equal(out[o: o + n], want, err_msg=f"request at {o} len {n}")
        assert (out[o + n: o + n + 16] == 0xA5).all(), "bytes past len were written"


def mixed_lengths(g, k):
    fixed = [0, 1, 15, 16, 17, 31, 33, 4095, 4096, 4097]
    rand = [int(x) for x in np.exp(g.uniform(np.log(1024), np.log(3 << 20), k - len(fixed)))]
    return fixed + rand


# Every shape the batch autotuner can pick (variant, CTA size, blocks per lane
# in flight, tile size), plus odd CTA sizes and the defaults.
SHAPES = [(1, th, tb, nb) for tb in (1024, 2048, 4096) for th in (256, 512, 1024) for nb in (1, 2, 4)] + \
    [(2, 128, tb, 0) for tb in (1024, 2048, 4096)] + \
    [(1, 1024, 8192, 2), (1, 256, 512, 1), (1, 544, 1024, 2), (2, 128, 256, 0), (0, 0, 2048, 0), (0, 0, 0, 0)]


@pytest.mark.parametrize("variant,threads,tile_blocks,nb", SHAPES,
                         ids=[f"v{v}_t{th}_tile{tb}_nb{nb}" for v, th, tb, nb in SHAPES])
def test_mixed_batch_matches_oracle(cuda, aes, ncpu, variant, threads, tile_blocks, nb):
    g = W.rng(40 + tile_blocks + threads + nb)
    lengths = mixed_lengths(g, 48)
    bits = [(128, 192, 256)[i % 3] for i in range(len(lengths))]
    kinds = [("random", "low32", "low64", "wrap128")[i % 4] for i in range(len(lengths))]
    reqs, meta, payload, src, dst = make_requests(cuda, aes, g, lengths, bits, kinds)
    aes.batch(reqs, variant=variant, tile_blocks=tile_blocks, threads=threads, blocks_per_thread=nb)
    check_all(cuda, meta, payload, dst, ncpu)


def test_batch_autotune_picks_a_shape_that_stays_exact(cuda, aes, ncpu, tmp_path):
    """aes_batch_autotune times every candidate shape on the caller's own
    requests (overwriting their outputs with the correct ciphertext), makes
    the fastest the device's batch shape, and batches that then use it (plans
    and one-shot calls) still give the oracle's bytes."""
    g = W.rng(47)
    lengths = mixed_lengths(g, 40)
    bits = [(128, 256)[i % 2] for i in range(len(lengths))]
    reqs, meta, payload, src, dst = make_requests(cuda, aes, g, lengths, bits)
    d = aes.batch_tuned_shape()
    default = (d["variant"], d["threads"], d["tile_blocks"], d["blocks_per_thread"])
    try:
        best = aes.batch_autotune(reqs)
        assert best == aes.batch_tuned_shape()
        assert best["variant"] in (1, 2) and best["tile_blocks"] in (1024, 2048, 4096)
        check_all(cuda, meta, payload, dst, ncpu)  # the candidates' own launches
        dst.fill_(0xA5)
        plan = aes.BatchPlan(reqs)
        plan.launch()
        check_all(cuda, meta, payload, dst, ncpu)
        plan.close()
        dst.fill_(0xA5)
        aes.batch(reqs)
        check_all(cuda, meta, payload, dst, ncpu)
    finally:
        set_batch_shape(cuda, aes, tmp_path / "shape.json", default)  # for the tests that follow


@pytest.mark.parametrize("seed", [1, 7, 12345])
def test_scrambled_tile_order_gives_same_result(cuda, aes, ncpu, seed):
    g = W.rng(50)
    lengths = mixed_lengths(g, 40)
    bits = [128 if i % 2 else 256 for i in range(len(lengths))]
    reqs, meta, payload, src, dst = make_requests(cuda, aes, g, lengths, bits)
    aes.batch(reqs, tile_blocks=1024, tile_order_seed=seed)
    check_all(cuda, meta, payload, dst, ncpu)


def test_batch_equals_per_request_calls(cuda, aes):
    g = W.rng(51)
    lengths = mixed_lengths(g, 32)
    bits = [128 if i % 2 else 256 for i in range(len(lengths))]
    reqs, meta, payload, src, dst = make_requests(cuda, aes, g, lengths, bits)
    aes.batch(reqs)
    cuda.cuda.synchronize()
    batched = to_host(dst).copy()
    dst.fill_(0xA5)
    for r in reqs:
        aes.ctr(*r)
    cuda.cuda.synchronize()
    np.testing.assert_array_equal(to_host(dst), batched)


def test_plan_graph_replays(cuda, aes, ncpu):
    g = W.rng(52)
    lengths = mixed_lengths(g, 24)
    bits = [(128, 256)[i % 2] for i in range(len(lengths))]
    reqs, meta, payload, src, dst = make_requests(cuda, aes, g, lengths, bits)
    plan = aes.BatchPlan(reqs)
    assert plan.nbytes == sum(lengths)
    plan.launch()
    check_all(cuda, meta, payload, dst, ncpu)
    # same layout, new payload bytes: the replay encrypts the new contents
    payload2 = W.random_bytes(g, payload.size)
    src.copy_(cuda.from_numpy(payload2))
    dst.fill_(0xA5)
    plan.launch()
    plan.launch()  # idempotent: out depends only on in
    check_all(cuda, meta, payload2, dst, ncpu)
    plan.close()


def test_batch_argument_errors(cuda, aes):
    ctx = aes.Context(bytes(16), 128)
    buf = cuda.zeros(1 << 16, dtype=cuda.uint8, device="cuda")
    p = buf.data_ptr()
    ok = (ctx, bytes(16), p, p + 4096, 1024)
    assert aes.batch_status([ok]) == aes.AES_OK
    assert aes.batch_status([ok, (ctx, bytes(16), p + 8, p + 8192, 64)]) == aes.AES_EALIGN
    assert aes.batch_status([ok, (ctx, bytes(16), p, p + 16, 64)]) == aes.AES_EOVERLAP
    assert aes.batch_status([ok], tile_blocks=100) == aes.AES_EINVAL
    assert aes.batch_status([ok], threads=1000) == aes.AES_EINVAL
    assert aes.batch_status([(ctx, bytes(16), 0, 0, 0)]) == aes.AES_OK  # all empty
    cuda.cuda.synchronize()


def test_full_size_batch_workload_matches_oracle(cuda, aes, ncpu):
    """The 4096-request workload at full size (~3.7 GB), launched as the
    benchmark launches it (a graph plan with the device's batch shape), and
    every byte of every request compared with the oracle (about 80 s of
    oracle time on 16 host cores), as is every byte past each request up to
    the next 256-byte boundary (untouched)."""
    import concurrent.futures as cf

    w = W.batch_varlen(seed=W.SEED_BASE + 3)
    src = to_dev(cuda, w.payload)
    dst = cuda.full((w.arena_bytes,), 0xA5, dtype=cuda.uint8, device="cuda")
    ctxs = [aes.Context(w.key_of(i).tobytes(), int(w.bits[i])) for i in range(w.n)]
    reqs = [(ctxs[i], w.ivs[i].tobytes(), src.data_ptr() + int(w.offsets[i]),
             dst.data_ptr() + int(w.offsets[i]), int(w.lengths[i])) for i in range(w.n)]
    plan = aes.BatchPlan(reqs)
    assert plan.nbytes == w.total_bytes
    plan.launch()
    cuda.cuda.synchronize()
    plan.close()
    out = to_host(dst)
    del src, dst

    def check(i):
        o, n = int(w.offsets[i]), int(w.lengths[i])
        want = oracle.ctr_mt(w.key_of(i), int(w.bits[i]), w.ivs[i], w.payload[o: o + n],
                             ncpu if n >= (8 << 20) // 4 else 1)
        if not np.array_equal(out[o: o + n], want):
            bad = int(np.flatnonzero(out[o: o + n] != want)[0])
            return f"request {i} (len {n}) differs from byte {bad}"
        pad_end = (o + n + 255) // 256 * 256
        if not (out[o + n: pad_end] == 0xA5).all():
            return f"request {i}: bytes past len were written"
        return None

    # large requests use every core each; the many small ones run side by side
    order = sorted(range(w.n), key=lambda i: -int(w.lengths[i]))
    big = [i for i in order if w.lengths[i] >= (8 << 20) // 4]
    small = [i for i in order if w.lengths[i] < (8 << 20) // 4]
    errors = [e for e in map(check, big) if e]
    with cf.ThreadPoolExecutor(ncpu) as ex:
        errors += [e for e in ex.map(check, small) if e]
    assert not errors, errors[:5]
    cuda.cuda.empty_cache()


def test_batch_pinned_host_buffers(cuda, aes, ncpu):
    """Batch requests whose payloads live in pinned host memory (the kernel
    reads and writes them over NVLink-C2C through their device aliases), mixed
    with device-resident ones in the same launch."""
    g = W.rng(48)
    lengths = [1, 17, 4096 + 5, 1 << 20, (1 << 20) + 9, 3 << 16]
    pad = [(n + 255) // 256 * 256 + 256 for n in lengths]
    offs = np.concatenate([[0], np.cumsum(pad)[:-1]]).astype(np.int64)
    total = int(sum(pad))
    payload = W.random_bytes(g, total)
    hsrc = cuda.from_numpy(payload.copy()).pin_memory()
    hdst = cuda.full((total,), 0xA5, dtype=cuda.uint8).pin_memory()
    dsrc = to_dev(cuda, payload)
    ddst = to_dev(cuda, np.zeros(0, np.uint8), pad=total)
    reqs, meta = [], []
    for i, n in enumerate(lengths):
        bits = (128, 256)[i % 2]
        key = W.random_bytes(g, bits // 8)
        iv = iv_with_low(g, ("random", "low32")[i % 2])
        ctx = aes.Context(key.tobytes(), bits)
        o = int(offs[i])
        src, dst = (hsrc, hdst) if i % 3 != 2 else (dsrc, ddst)
        reqs.append((ctx, iv.tobytes(), src.data_ptr() + o, dst.data_ptr() + o, n))
        meta.append((key, bits, iv, o, n, i % 3 != 2))
    aes.batch(reqs)
    cuda.cuda.synchronize()
    hout, dout = hdst.numpy(), to_host(ddst)
    for key, bits, iv, o, n, on_host in meta:
        out = hout if on_host else dout
        want = oracle.ctr_mt(key, bits, iv, payload[o: o + n], ncpu)
        np.testing.assert_array_equal(out[o: o + n], want, err_msg=f"request at {o} len {n}")
        assert (out[o + n: o + n + 16] == 0xA5).all(), "bytes past len were written"


def test_in_place_batch_matches_oracle(cuda, aes, ncpu):
    """Every other request of the batch encrypts in place (in == out); the
    rest write to a second buffer.  All match the oracle."""
    g = W.rng(52)
    lengths = mixed_lengths(g, 24)
    bits = [(128, 256)[i % 2] for i in range(len(lengths))]
    reqs, meta, payload, src, dst = make_requests(cuda, aes, g, lengths, bits)
    reqs = [(c, iv, i_, i_ if k % 2 == 0 else o_, n) for k, (c, iv, i_, o_, n) in enumerate(reqs)]
    aes.batch(reqs, tile_blocks=1024)
    cuda.cuda.synchronize()
    out_src, out_dst = to_host(src), to_host(dst)
    for k, (key, b, iv, o, n) in enumerate(meta):
        got = out_src[o: o + n] if k % 2 == 0 else out_dst[o: o + n]
        np.testing.assert_array_equal(got, oracle.ctr_mt(key, b, iv, payload[o: o + n], ncpu),
                                      err_msg=f"request {k} len {n}")


@pytest.mark.parametrize("bits", [128, 256])
def test_batch_every_length_0_to_64(cuda, aes, ncpu, bits):
    """One batch of 65 requests, of every length from 0 to 64 bytes (each
    tail u = 1..15 of a partial final block several times over)."""
    g = W.rng(53 + bits)
    lengths = list(range(65))
    reqs, meta, payload, src, dst = make_requests(cuda, aes, g, lengths, [bits] * len(lengths))
    aes.batch(reqs, tile_blocks=1024)
    check_all(cuda, meta, payload, dst, ncpu)


@pytest.mark.parametrize("n", [1, 31, 33, 500, 501, 3000])
@pytest.mark.parametrize("ctas,tile_blocks,seed,threads", [(0, 0, 0, 0), (1, 256, 0, 0), (3, 256, 9, 0), (0, 512, 5, 1024),
                                                           (2, 0, 0, 96)])
def test_cost_line_edges(cuda, aes, ncpu, n, ctas, tile_blocks, seed, threads):
    """The split of a batch into equal pieces of cost and tiles of it: many
    requests of around a chunk (empty ones among them, also first and last),
    one of several CTA pieces, all key sizes, IV low bytes on both sides of a
    chunk edge, a carry into counter byte 10 inside a run, and request counts
    around the search's 32 and past one piece's worth."""
    g = W.rng(5400 + n + ctas + tile_blocks + seed)
    sizes = [0, 1, 15, 16, 496, 511, 512, 513, 528, 4096, 8000]
    lengths = [int(sizes[i]) for i in g.integers(0, len(sizes), n)]
    if n == 1:
        lengths = [300_000 + 7]
    elif n > 500:
        lengths[0] = lengths[-1] = 0
        lengths[n // 2] = (1 << 20) + 3
    bits = [(128, 192, 256)[int(x)] for x in g.integers(0, 3, n)]
    reqs, meta, payload, src, dst = make_requests(cuda, aes, g, lengths, bits)
    lows = [0x00, 0x1F, 0x20, 0xFF]
    for i, (ctx, iv, s, d, k) in enumerate(reqs):
        b = bytearray(iv)
        b[15] = lows[i % 4]
        if i % 3 == 0:
            b[11:15] = b"\xff\xff\xff\xff" if i % 2 else b"\xff\xff\xff\xfc"
        reqs[i] = (ctx, bytes(b), s, d, k)
        meta[i] = (meta[i][0], meta[i][1], np.frombuffer(bytes(b), np.uint8), meta[i][3], k)
    aes.batch(reqs, ctas=ctas, tile_blocks=tile_blocks, tile_order_seed=seed, threads=threads)
    check_all(cuda, meta, payload, dst, 1)


@pytest.mark.parametrize("n", [3, 64, 65, 1100])
def test_batch_calls_under_capture(cuda, aes, ncpu, n):
    """One-shot batches captured into a CUDA graph (their requests travel in
    kernel parameters, several launches of them past 500): nothing runs during
    the capture, and every replay encrypts what the buffers then hold.  A
    plan's launch is refused while its stream is being captured."""
    g = W.rng(5600 + n)
    lengths = [int(x) for x in g.integers(0, 3000, n)]
    bits = [(128, 192, 256)[i % 3] for i in range(n)]
    for call in (aes.batch_status, aes.batch_noalloc_status):
        if call is aes.batch_noalloc_status and n > 1024:
            continue
        reqs, meta, payload, src, dst = make_requests(cuda, aes, g, lengths, bits)
        plan = aes.BatchPlan(reqs)
        s = cuda.cuda.Stream()
        cuda.cuda.synchronize()
        graph = cuda.cuda.CUDAGraph()
        with cuda.cuda.graph(graph, stream=s, capture_error_mode="thread_local"):
            assert call(reqs, stream=s) == aes.AES_OK
            assert aes.lib().aes_batch_plan_launch(plan.handle, s.cuda_stream) == aes.AES_ECUDA
        plan.close()
        assert (dst == 0xA5).all()
        graph.replay()
        check_all(cuda, meta, payload, dst, 1)
        payload2 = W.random_bytes(g, payload.size)
        src.copy_(cuda.from_numpy(payload2))
        dst.fill_(0xA5)
        graph.replay()
        check_all(cuda, meta, payload2, dst, 1)
        del graph


@pytest.mark.parametrize("n", [2, 70, 600])
def test_batch_checks_every_payload_pointer(cuda, aes, n):
    """A batch whose payloads share allocations still refuses the one request
    whose pointer the GPU cannot address, wherever it stands in the batch, and
    accepts pinned host memory among device memory."""
    ctx = aes.Context(bytes(16), 128)
    buf = cuda.zeros(n * 512, dtype=cuda.uint8, device="cuda")
    pinned = cuda.zeros(4096, dtype=cuda.uint8).pin_memory()
    pageable = np.zeros(8192, np.uint8)
    bad = (pageable.ctypes.data + 15) & ~15
    p = buf.data_ptr()
    reqs = [(ctx, bytes(16), p + 512 * i, p + 512 * i + 256, 200) for i in range(n)]
    for at in sorted({0, 1, n - 1}):
        for src, dst, want in ((bad, p + 256, aes.AES_EPTR), (p, bad, aes.AES_EPTR), (bad, bad, aes.AES_EPTR),
                               (256, p + 256, aes.AES_EPTR), (0, p + 256, aes.AES_EINVAL),
                               (pinned.data_ptr(), pinned.data_ptr() + 1024, aes.AES_OK)):
            q = list(reqs)
            q[at] = (ctx, bytes(16), src, dst, 200)
            assert aes.batch_status(q) == want
            assert aes.batch_noalloc_status(q) == want
    cuda.cuda.synchronize()


def test_plan_launches_are_ordered_across_streams(cuda, aes, ncpu):
    """Launches of one plan on different streams run one after the other: a
    plan that encrypts in place, launched an even number of times from two
    streams that wait for nothing, gives its input back."""
    g = W.rng(5700)
    lengths = [(24 << 20) + 7, 4096, 17, (3 << 20) + 16, 900_000]
    bits = [(128, 256, 192)[i % 3] for i in range(len(lengths))]
    reqs, meta, payload, src, dst = make_requests(cuda, aes, g, lengths, bits)
    plan = aes.BatchPlan([(c, iv, s, s, k) for c, iv, s, d, k in reqs])
    streams = [cuda.cuda.Stream(), cuda.cuda.Stream()]
    cuda.cuda.synchronize()
    for i in range(40):
        plan.launch(streams[i & 1])
    cuda.cuda.synchronize()
    np.testing.assert_array_equal(to_host(src), payload)
    plan.launch(streams[0])
    plan.launch(streams[1])
    plan.launch(streams[1])
    cuda.cuda.synchronize()
    out = to_host(src)
    for key, b, iv, o, k in meta:
        np.testing.assert_array_equal(out[o: o + k], oracle.ctr_mt(key, b, iv, payload[o: o + k], ncpu))
    plan.close()


def test_claims_from_the_whole_line(cuda, aes, ncpu):
    """Plans and one-shot tables of 2^18 chunks and more, whose warps claim
    from the whole batch through one counter in device memory, launched
    several times (two counters take turns): device and pinned payloads, keys
    in registers and in shared memory, seeded tile orders, the bitsliced
    kernel; short, empty and tailed requests among long ones, all key sizes."""
    g = W.rng(5800)
    n = 1100
    lengths = [int(x) for x in np.exp(g.uniform(np.log(64), np.log(1 << 20), n))]
    lengths[0] = lengths[-1] = lengths[500] = 0
    lengths[7] = (9 << 20) + 5
    lengths[900] = max((1 << 27) + 4096 - sum(lengths), 16)
    bits = [(128, 192, 256)[int(x)] for x in g.integers(0, 3, n)]
    kinds = [("random", "low32", "low64", "wrap128")[i % 4] for i in range(n)]
    reqs, meta, payload, src, dst = make_requests(cuda, aes, g, lengths, bits, kinds)
    cuda.cuda.synchronize()
    hsrc, hdst = src.cpu().pin_memory(), dst.cpu().pin_memory()
    h = [(c, iv, hsrc.data_ptr() + o, hdst.data_ptr() + o, k) for (c, iv, _, _, k), (_, _, _, o, _) in zip(reqs, meta)]
    want = np.full(payload.size, 0xA5, np.uint8)
    for key, b, iv, o, k in meta:
        want[o: o + k] = oracle.ctr_mt(key, b, iv, payload[o: o + k], ncpu if k > 1 << 16 else 1)
    for pinned in (False, True):
        r, out = (h, hdst) if pinned else (reqs, dst)
        for opts in ({}, {"threads": 1024}, {"tile_order_seed": 3}, {"tile_order_seed": 8, "tile_blocks": 256},
                     {"variant": 2}, {"variant": 2, "tile_order_seed": 5}):
            plan = aes.BatchPlan(r, **opts)
            for launch in (plan.launch, plan.launch, lambda: aes.batch(r, **opts), plan.launch):
                out.fill_(0xA5)
                cuda.cuda.synchronize()
                launch()
                cuda.cuda.synchronize()
                assert np.array_equal(out.cpu().numpy(), want), (pinned, opts)
            plan.launch()  # in a row, on two streams
            plan.launch(cuda.cuda.Stream())
            plan.launch()
            cuda.cuda.synchronize()
            assert np.array_equal(out.cpu().numpy(), want), (pinned, opts)
            plan.close()


@pytest.mark.parametrize("n", [6, 70, 600, 1100])
@pytest.mark.parametrize("threads", [0, 1024])
def test_pinned_payloads_in_every_kernel(cuda, aes, ncpu, n, threads, tmp_path):
    """Pinned payloads (chunk pairs in address order) through every kernel
    that takes them: requests in parameters (up to 64, up to 500, several
    launches) and in a device table, keys in registers and in shared memory;
    all key sizes, IV low bytes on both sides of a chunk edge, tails, odd
    chunk counts (a half-empty last pair), a device payload among them."""
    g = W.rng(5900 + n + threads)
    sizes = [1, 16, 511, 512, 513, 1024 + 16, 1536, 1536 + 7, 4096 + 5, 40_000 + 3]
    lengths = [int(sizes[i % len(sizes)]) for i in range(n)]
    lengths[n // 2] = 300_000 + 9
    bits = [(128, 192, 256)[int(x)] for x in g.integers(0, 3, n)]
    reqs, meta, payload, src, dst = make_requests(cuda, aes, g, lengths, bits)
    cuda.cuda.synchronize()
    hsrc, hdst = src.cpu().pin_memory(), dst.cpu().pin_memory()
    lows = [0x00, 0x1F, 0x20, 0xE1, 0xFF]
    want = np.full(payload.size, 0xA5, np.uint8)
    r = []
    for i, ((c, iv, s, d, k), (key, b, _, o, _)) in enumerate(zip(reqs, meta)):
        iv = iv[:15] + bytes([lows[i % 5]])
        want[o: o + k] = oracle.ctr(key, b, np.frombuffer(iv, np.uint8), payload[o: o + k])
        r.append((c, iv, s, d, k) if i == 1 else (c, iv, hsrc.data_ptr() + o, hdst.data_ptr() + o, k))
    o, k = meta[1][3], meta[1][4]

    def check(call):
        hdst.fill_(0xA5)
        dst.fill_(0xA5)
        cuda.cuda.synchronize()
        call()
        cuda.cuda.synchronize()
        out = hdst.numpy().copy()
        out[o: o + k] = to_host(dst)[o: o + k]
        np.testing.assert_array_equal(out, want)

    check(lambda: aes.batch(r, threads=threads))
    plan = aes.BatchPlan(r, threads=threads)
    check(plan.launch)
    plan.close()
    if n <= 1024:
        d = aes.batch_tuned_shape()
        default = (d["variant"], d["threads"], d["tile_blocks"], d["blocks_per_thread"])
        try:
            if threads:
                set_batch_shape(cuda, aes, tmp_path / "shape.json", (1, threads, 2048, 1))
            check(lambda: aes.batch_noalloc_status(r))
        finally:
            set_batch_shape(cuda, aes, tmp_path / "shape.json", default)
