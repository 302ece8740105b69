// tile.cuh -- xor the AES-CTR keystream into a run of 32-block chunks of one
// message with T-table rounds and counter-mode caching (the batch kernel's
// work on a request).
#pragma once
#include "internal.h"
#include "common.cuh"
#include "aes_ttable.cuh"

namespace aestile {

// Chunks.  Block j of a message sits at counter position v0 + j, v0 = the IV's
// low byte; 32 consecutive positions are a chunk (position >> 5), the work of
// one warp-wide step: lane l holds the block whose counter low byte is
// l + 32m, m = chunk & 7, and every load/store moves 512 contiguous bytes.
__device__ __forceinline__ uint64_t first_chunk(uint64_t iv_lo) { return (iv_lo & 255u) >> 5; }

constexpr uint32_t kRunChunks = 248;  // chunks whose group constants a warp holds at once
constexpr uint32_t kRunGroups = 32;   // the groups a run touches at most: one per lane

// How many of the chunks k0, k0 + 1, ... of a message one run may take: at
// most 248, and none past a carry into counter byte 10 (every 2^40 blocks),
// up to which lane_round2 holds for all groups.
__device__ __forceinline__ uint32_t run_chunks(uint64_t iv_lo, uint64_t k0, uint64_t nk)
{
    const uint64_t low = ((iv_lo & ~(uint64_t)255u) + ((k0 >> 3) << 8)) & ((1ull << 40) - 1);
    const uint64_t same = (((1ull << 40) - low) >> 5) - (k0 & 7u);
    const uint32_t n = nk < kRunChunks ? (uint32_t)nk : kRunChunks;
    return same < n ? (uint32_t)same : n;
}

// A run: chunks [k0, k0 + n) of one message, n <= run_chunks, done by the
// calling warp alone.  The lanes compute the round-2 constants of the run's
// groups side by side (one group per lane, 27 wavefronts for all of them, kept
// in the warp's s_group slice), then walk the chunks with the same counter low
// bytes one after the other, so that a lane's part of round 2 (lane_round2) is
// computed once for all groups.  Per 64 chunks that is 27 + 43 wavefronts and
// one broadcast load per chunk, 2.1 a chunk (1.5 at 128); constants per group
// and warp and five lookups per block were 8.4.  The next chunk's plaintext is
// loaded before the current chunk's rounds.  Nothing past len is touched; the
// final partial block is done bytewise.
template <int NR, class RK>
__device__ __forceinline__ void xor_run(const uint4 *__restrict__ in, uint4 *__restrict__ out, uint64_t len,
                                        uint64_t iv_hi, uint64_t iv_lo, uint64_t k0, uint32_t n, uint4 *s_group,
                                        const aestt::Lanes &ln, const RK &rk)
{
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t v0 = iv_lo & 255u, base_lo = iv_lo & ~(uint64_t)255u;
    const uint64_t nfull = len >> 4;
    const uint32_t tail = (uint32_t)(len & 15);
    const uint64_t l0 = base_lo + ((k0 >> 3) << 8);  // counter of the run's first group
    const uint64_t h0 = iv_hi + (l0 < base_lo ? 1 : 0);
    const int64_t j0 = (int64_t)(k0 << 5) - (int64_t)v0;  // below 0 in a message's first chunk only
    const uint4 *ip = in + j0 + lane;
    uint4 *op = out + j0 + lane;
    const uint32_t lo = j0 < 0 ? (uint32_t)-j0 : 0;  // blocks lo.. of the run exist
    const int64_t left = (int64_t)nfull - j0;        // whole blocks from the run's start on
    const uint32_t hi = left > (int64_t)(n * 32u) ? n * 32u : (uint32_t)left;
    const uint32_t partial = tail && left < (int64_t)(n * 32u) ? (uint32_t)left : ~0u;
    uint4 next = make_uint4(0, 0, 0, 0);
    if (lane >= lo && lane < hi)
        next = aesdev::ld_stream(ip);
    {
        const uint64_t l = l0 + ((uint64_t)lane << 8);
        const uint4 q = aestt::group_round2(aestt::CounterWords(h0 + (l < l0 ? 1 : 0), l), ln, rk);
        __syncwarp();  // every lane is done with the previous run's constants
        s_group[lane] = q;
        __syncwarp();
    }
    const uint32_t column0 = aestt::column0_round1(aestt::CounterWords(h0, l0), ln, rk);
    const uint32_t m0 = (uint32_t)k0 & 7u, cols = n < 8u ? n : 8u;
#pragma unroll 1
    for (uint32_t c0 = 0; c0 < cols; ++c0) {
        const uint4 mine = aestt::lane_round2(column0, ((m0 + c0) & 7u) * 32u + lane, ln, rk);
#pragma unroll 1
        for (uint32_t c = c0; c < n; c += 8u) {
            const uint4 pt = next;
            const uint32_t cn = c + 8u < n ? c + 8u : c0 + 1 < cols ? c0 + 1 : n;
            const uint32_t in_ = cn * 32u + lane;
            if (in_ >= lo && in_ < hi)
                next = aesdev::ld_stream(ip + cn * 32u);
            const uint4 group = s_group[(m0 + c) >> 3];
            uint32_t s[4] = {group.x ^ mine.x, group.y ^ mine.y, group.z ^ mine.z, group.w ^ mine.w};
            aestt::rounds<3, NR>(s, ln, rk);
            const uint32_t i = c * 32u + lane;
            if (i >= lo && i < hi)
                aesdev::st_stream(op + c * 32u, make_uint4(pt.x ^ s[0], pt.y ^ s[1], pt.z ^ s[2], pt.w ^ s[3]));
            else if (i == partial)
                aesdev::xor_tail(reinterpret_cast<const uint8_t *>(ip + c * 32u),
                                 reinterpret_cast<uint8_t *>(op + c * 32u), s[0], s[1], s[2], s[3], tail);
        }
    }
}

// The same run for payloads in pinned host memory, where the link and the
// host's memory bound the kernel: chunks in address order, two at a time,
// loaded together and stored together, so that each warp moves 1 KiB bursts
// (1024 requests of 1 KiB to 8 MiB in pinned memory, 0.9 GB each way: 144 GB/s
// each way, 168 being the link's measured most; claimed by fixed pieces 141,
// and 134 with xor_run).  The lane's
// part of round 2 is derived for each chunk; the lookups do not bound here.
template <int NR, class RK>
__device__ __forceinline__ void xor_run_host(const uint4 *__restrict__ in, uint4 *__restrict__ out, uint64_t len,
                                             uint64_t iv_hi, uint64_t iv_lo, uint64_t k0, uint32_t n, uint4 *s_group,
                                             const aestt::Lanes &ln, const RK &rk)
{
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t v0 = iv_lo & 255u, base_lo = iv_lo & ~(uint64_t)255u;
    const uint64_t nfull = len >> 4;
    const uint32_t tail = (uint32_t)(len & 15);
    const uint64_t l0 = base_lo + ((k0 >> 3) << 8);
    const uint64_t h0 = iv_hi + (l0 < base_lo ? 1 : 0);
    {
        const uint64_t l = l0 + ((uint64_t)lane << 8);
        const uint4 q = aestt::group_round2(aestt::CounterWords(h0 + (l < l0 ? 1 : 0), l), ln, rk);
        __syncwarp();
        s_group[lane] = q;
        __syncwarp();
    }
    const uint32_t column0 = aestt::column0_round1(aestt::CounterWords(h0, l0), ln, rk);
    const uint32_t m0 = (uint32_t)k0 & 7u;
#pragma unroll 1
    for (uint32_t c = 0; c < n; c += 2u) {
        uint4 x[2];
        // a block before the message's first wraps to a huge index and fails j <= nfull
        const uint64_t j0 = ((k0 + c) << 5) + lane - v0;
#pragma unroll
        for (int b = 0; b < 2; ++b)
            x[b] = c + b < n && j0 + 32u * b < nfull ? aesdev::ld_stream(in + j0 + 32u * b) : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const uint4 mine = aestt::lane_round2(column0, ((m0 + c + b) & 7u) * 32u + lane, ln, rk);
            const uint4 group = s_group[(m0 + (c + b < n ? c + b : c)) >> 3];
            uint32_t s[4] = {group.x ^ mine.x, group.y ^ mine.y, group.z ^ mine.z, group.w ^ mine.w};
            aestt::rounds<3, NR>(s, ln, rk);
            x[b] = make_uint4(x[b].x ^ s[0], x[b].y ^ s[1], x[b].z ^ s[2], x[b].w ^ s[3]);
        }
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const uint64_t j = j0 + 32u * b;
            if (c + b >= n)
                continue;
            if (j < nfull)
                aesdev::st_stream(out + j, x[b]);
            else if (j == nfull && tail)  // x holds the keystream: no plaintext was loaded
                aesdev::xor_tail(reinterpret_cast<const uint8_t *>(in + j), reinterpret_cast<uint8_t *>(out + j),
                                 x[b].x, x[b].y, x[b].z, x[b].w, tail);
        }
    }
}

}  // namespace aestile
