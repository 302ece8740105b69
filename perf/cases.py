"""The library's work as its users have it done, as cases that can be timed.

``listed()`` names the cases, ``draw()`` makes more from the same ranges,
``prepare()`` holds what a program has in hand before a call (payloads, keys,
plans, a running server), ``run()`` makes one pass through the public entry
points and returns its outputs, and ``work()`` counts the bytes a pass cannot
do without.  Outputs are ciphertext bytes: exactly one answer is right.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_02630_gb300 import aesoffload as aes
from paper_2607_02630_gb300 import workloads as W

KIB, MIB = 1 << 10, 1 << 20


def listed():
    return [
        # A small page of a response, encrypted on the stream that made it: the
        # lower end of the offload's size range, where the launch is the cost.
        {"name": "call_4k", "kind": "call", "nbytes": 4 * KIB, "bits": 128},
        # A medium payload of no round size under the longer key.
        {"name": "call_60k_tail", "kind": "call", "nbytes": 61453, "bits": 256},
        # The offload most of the measurements are about: 1 MiB, made and
        # waited for on the server's own thread (the blocking offload call).
        {"name": "sync_1m", "kind": "sync", "nbytes": MIB, "bits": 128},
        # The upper end of the per-request range, with a tail.
        {"name": "call_8m_tail", "kind": "call", "nbytes": 8 * MIB + 9, "bits": 256},
        # The largest size of the single-buffer sweep (a file, a shard).
        {"name": "call_256m", "kind": "call", "nbytes": 256 * MIB, "bits": 128},
        # A payload that stays in pinned host memory on both sides, read and
        # written by the kernel over the host link.
        {"name": "host_16m", "kind": "host", "nbytes": 16 * MIB, "bits": 128},
        # What a busy server collects in one poll: short requests, each with
        # its own key, length and IV, encrypted by one call.
        {"name": "batch_64_small", "kind": "batch", "n": 64, "lo": KIB, "hi": 16 * KIB, "mix": 11},
        # The same over the whole request range, sizes known only at the call.
        {"name": "batch_512", "kind": "batch", "n": 512, "lo": KIB, "hi": 8 * MIB, "mix": 12},
        # The benchmark's batch: 4096 requests prepared once as a plan and
        # launched for every new payload.
        {"name": "plan_4096", "kind": "plan", "n": 4096, "lo": KIB, "hi": 8 * MIB, "mix": 3},
        # The batched call of a process that may not allocate.
        {"name": "noalloc_256", "kind": "noalloc", "n": 256, "lo": 4 * KIB, "hi": MIB, "mix": 13},
        # The resident server under a burst of its own request mix (70 % 1 MiB,
        # 10 % 8 MiB, 20 % 4-64 KiB).
        {"name": "served_mix_256", "kind": "served", "n": 256, "fixed": 0, "mix": 14},
        # The resident server with one 1 MiB request in flight: its latency.
        {"name": "served_one_1m", "kind": "served", "n": 1, "fixed": MIB, "mix": 15},
    ]


def _size(rng, lo, hi):
    """Log-uniform on [lo, hi]; half of the sizes are whole 16-byte blocks."""
    n = int(math.exp(rng.uniform(math.log(lo), math.log(hi))))
    return max(lo, n - n % 16 if rng.random() < 0.5 else n)


def draw(rng):
    kind = rng.choice(["call", "call", "call", "sync", "host", "batch", "batch", "plan", "noalloc", "served"])
    mix = rng.randrange(100, 1 << 20)
    if kind in ("call", "sync"):
        return {"kind": kind, "nbytes": _size(rng, KIB, (256 if kind == "call" else 16) * MIB),
                "bits": rng.choice([128, 192, 256])}
    if kind == "host":
        return {"kind": kind, "nbytes": _size(rng, 64 * KIB, 32 * MIB), "bits": rng.choice([128, 256])}
    if kind == "served":
        if rng.random() < 0.5:
            return {"kind": kind, "n": 1, "fixed": _size(rng, 4 * KIB, 8 * MIB), "mix": mix}
        return {"kind": kind, "n": _size(rng, 16, 512), "fixed": 0, "mix": mix}
    lo = _size(rng, 256, 64 * KIB)
    hi = _size(rng, 2 * lo, 8 * MIB)
    # at most the listed plan's bytes in all (the mean of a log-uniform length)
    most = min({"batch": 1024, "plan": 4096, "noalloc": 1024}[kind], int(3e9 / ((hi - lo) / math.log(hi / lo))))
    return {"kind": kind, "n": _size(rng, 8, most), "lo": lo, "hi": hi, "mix": mix}


def _lengths(case):
    """Request lengths and key sizes of a case, from the case alone."""
    seed = W.SEED_BASE + int(case["mix"])
    n = int(case["n"])
    if case["kind"] == "served":
        sizes = np.full(n, int(case["fixed"]), np.int64) if case["fixed"] else W.served_sizes(n, seed)
        return sizes, W.key_set(n, seed=seed)[0]
    w = W.batch_varlen(n, int(case["lo"]), int(case["hi"]), seed=seed, with_payload=False)
    return w.lengths, w.bits


def work(case):
    if case["kind"] in ("call", "sync", "host"):
        total = int(case["nbytes"])
    else:
        total = int(_lengths(case)[0].sum())
    return {"bytes": 2 * total, "flops": 0}  # payload in, ciphertext out


def _payload(n, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    # whole 8-byte words of random bits, cut to size
    return torch.randint(-(1 << 63), (1 << 63) - 1, (-(-n // 8),), dtype=torch.int64, device="cuda",
                         generator=g).view(torch.uint8)[:n]


# One server per process, as a serving program has; its keys are registered
# as connections come.  The idle limit lets other work have the SMs soon.
_SERVER = None


def _server():
    global _SERVER
    if _SERVER is None:
        _SERVER = aes.Server(max_keys=4096, idle_timeout_us=1000)
    return _SERVER


def prepare(case, seed):
    kind = case["kind"]
    g = W.rng(seed)
    if kind in ("call", "sync", "host"):
        n, bits = int(case["nbytes"]), int(case["bits"])
        state = {"kind": kind, "n": n, "ctx": aes.Context(W.random_bytes(g, bits // 8).tobytes(), bits),
                 "iv": W.random_bytes(g, 16).tobytes(), "src": _payload(n, seed)}
        state["dst"] = torch.zeros(n, dtype=torch.uint8, device="cuda")
        if kind == "host":
            state["src"] = state["src"].cpu().pin_memory()
            state["dst"] = torch.zeros(n, dtype=torch.uint8).pin_memory()
        return state
    lengths, bits = _lengths(case)
    padded = (lengths + W.ARENA_ALIGN - 1) // W.ARENA_ALIGN * W.ARENA_ALIGN
    offsets = np.concatenate([[0], np.cumsum(padded)[:-1]])
    total = int(padded.sum())
    src = _payload(total, seed)
    dst = torch.zeros(total, dtype=torch.uint8, device="cuda")
    n = len(lengths)
    keys = W.random_bytes(g, 32 * n).reshape(n, 32)
    ivs = W.random_bytes(g, 16 * n).reshape(n, 16)
    state = {"kind": kind, "src": src, "dst": dst}
    if kind == "served":
        srv = _server()
        # a few keys per program: requests of many connections share them
        slots = [srv.key_register(keys[i % n].tobytes()[: b // 8], b) for i, b in enumerate((128, 256))]
        state["requests"] = [(slots[0 if bits[i] == 128 else 1], ivs[i].tobytes(),
                              src.data_ptr() + int(offsets[i]), dst.data_ptr() + int(offsets[i]), int(lengths[i]))
                             for i in range(n)]
        return state
    state["requests"] = [(aes.Context(keys[i].tobytes()[: int(bits[i]) // 8], int(bits[i])), ivs[i].tobytes(),
                          src.data_ptr() + int(offsets[i]), dst.data_ptr() + int(offsets[i]), int(lengths[i]))
                         for i in range(n)]
    if kind == "plan":
        state["plan"] = aes.BatchPlan(state["requests"])
    return state


def run(state):
    kind = state["kind"]
    if kind in ("call", "host"):
        aes.ctr(state["ctx"], state["iv"], state["src"], state["dst"], state["n"])
    elif kind == "sync":
        aes.ctr_sync(state["ctx"], state["iv"], state["src"], state["dst"], state["n"])
    elif kind == "batch":
        aes.batch(state["requests"])
    elif kind == "plan":
        state["plan"].launch()
    elif kind == "noalloc":
        rc = aes.batch_noalloc_status(state["requests"])
        if rc != aes.AES_OK:
            raise aes.AesError(rc, "aes_ctr_batch_noalloc")
    else:
        _serve(_server(), state["requests"])
    return state["dst"]


def _serve(srv, requests):
    """Submit every request and wait for all of them, as a completion thread
    does; a full server is polled and the submit tried again."""
    if len(requests) == 1:
        rc = srv.wait(srv.submit(*requests[0]))
        if rc != aes.AES_OK:
            raise aes.AesError(rc, "offload_wait")
        return
    pending = []
    for r in requests:
        rc, ticket = srv.submit_status(*r)
        while rc == aes.AES_EAGAIN:
            pending = _poll(srv, pending)
            rc, ticket = srv.submit_status(*r)
        if rc != aes.AES_OK:
            raise aes.AesError(rc, "offload_submit")
        pending.append(ticket)
    while pending:
        pending = _poll(srv, pending)


def _poll(srv, tickets):
    """The tickets still in flight after one bounded wait."""
    _, status = srv.poll_many(tickets)
    left = []
    for t, s in zip(tickets, status.tolist()):
        if s == aes.AES_PENDING:
            left.append(t)
        elif s != aes.AES_OK:
            raise aes.AesError(s, "offload_poll_many")
    return left
