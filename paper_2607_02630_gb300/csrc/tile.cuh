// tile.cuh -- xor the AES-CTR keystream into a range of 16-byte blocks of
// one message with T-table rounds and counter-mode caching (shared by the
// single-buffer, batch and served kernels).
#pragma once
#include "internal.h"
#include "common.cuh"
#include "aes_ttable.cuh"

namespace aestile {

// Blocks [first, last) of a message (in/out, len bytes, initial counter
// (iv_hi, iv_lo) as big-endian halves) are walked by counter group: group g
// holds blocks j = 256g - v0 + L, v0 = the IV's low byte, L = 0..255 the
// counter's low byte.  Lane l of a warp owns L = l + 32m (m = 0..7), so every
// 16-byte load/store instruction of a warp covers 32 consecutive blocks.  A
// group is split into `parts` work units (1, 2, 4 or 8; unit p covers
// m in [p*8/parts, (p+1)*8/parts)); warp w0, w0 + stride, ... take the units
// in order.  Whole groups amortise the 27 group-constant lookups best; parts
// spread a short message over more warps.  NB blocks per lane are in flight
// at once with their plaintext loaded before the keystream is computed.  The
// final partial block is done bytewise and nothing past len is touched.
template <int NR, int NB, class RK>
__device__ __forceinline__ void xor_range(const uint4 *__restrict__ in, uint4 *__restrict__ out, uint64_t len,
                                          uint64_t iv_hi, uint64_t iv_lo, uint64_t first, uint64_t last,
                                          uint64_t warp0, uint64_t warp_stride, uint32_t parts,
                                          const aestt::Lanes &ln, const RK &rk)
{
    if (first >= last)
        return;
    const uint64_t nfull = len >> 4;
    const uint32_t tail = (uint32_t)(len & 15);
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t v0 = iv_lo & 255u;
    const uint64_t base_lo = iv_lo & ~(uint64_t)255u;
    const uint64_t g_first = (v0 + first) >> 8, g_end = ((v0 + last - 1) >> 8) + 1;
    const uint32_t per = 8u / parts;
    const uint64_t u_end = (g_end - g_first) * parts;
    uint64_t gc_for = ~0ull;
    aestt::Group gc;
    const uint64_t pf_end = last < nfull ? last : nfull;  // full blocks only: never past the input
    for (uint64_t u = warp0; u < u_end; u += warp_stride) {
        const uint64_t g = g_first + u / parts;
        const uint32_t m_begin = (uint32_t)(u % parts) * per;
        if (NB == 1 && lane == 0 && u + warp_stride < u_end) {
            // With one block per lane in flight a warp has little of its own
            // to hide the payload's DRAM latency with: ask L2 now for the
            // plaintext of the warp's next unit (one bulk prefetch, a hint
            // that reads nothing into registers; the range stays inside the
            // input's full blocks).  Measured on the batch workload: 833 ->
            // 868 GB/s with one block per lane; with two it cost ~1.5 %, so
            // it is not compiled in there.
            const uint64_t un = u + warp_stride;
            const uint64_t jb = ((g_first + un / parts) << 8) - v0 + 32u * ((uint32_t)(un % parts) * per);
            const uint64_t a = jb < first ? first : jb;
            const uint64_t b = jb + 32u * per < pf_end ? jb + 32u * per : pf_end;
            if (a < b)  // also false when jb wrapped below 0 (the first group)
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(in + a), "r"((uint32_t)((b - a) * 16u))
                             : "memory");
        }
        if (g != gc_for) {
            uint32_t base[4];
            const uint64_t l = base_lo + (g << 8);
            const uint64_t h = iv_hi + (l < base_lo ? 1ull : 0ull);
            base[0] = aesdev::bswap32((uint32_t)(h >> 32));
            base[1] = aesdev::bswap32((uint32_t)h);
            base[2] = aesdev::bswap32((uint32_t)(l >> 32));
            base[3] = aesdev::bswap32((uint32_t)l);
            gc = aestt::group_consts(base, ln, rk);
            gc_for = g;
        }
        const uint64_t j0 = (g << 8) - v0;  // block of L = 0 (wraps below 0 in the first group)
#pragma unroll 1
        for (uint32_t m0 = m_begin; m0 < m_begin + per; m0 += NB) {
            uint32_t L[NB], s[NB][4];
            uint4 pt[NB];
            bool ok[NB];
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                L[b] = lane + 32u * (m0 + (uint32_t)b);
                const uint64_t j = j0 + L[b];
                // a wrapped index is huge and fails j < last; m past the unit is skipped
                ok[b] = m0 + (uint32_t)b < m_begin + per && j >= first && j < last;
                pt[b] = (ok[b] && j < nfull) ? aesdev::ld_stream(in + j) : make_uint4(0, 0, 0, 0);
            }
            aestt::encrypt_group<NR, NB>(s, L, gc, ln, rk);
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const uint64_t j = j0 + L[b];
                if (!ok[b])
                    continue;
                if (j < nfull) {
                    aesdev::st_stream(out + j, make_uint4(pt[b].x ^ s[b][0], pt[b].y ^ s[b][1],
                                                          pt[b].z ^ s[b][2], pt[b].w ^ s[b][3]));
                } else if (tail) {  // j == nfull: the final partial block
                    aesdev::xor_tail(reinterpret_cast<const uint8_t *>(in + j),
                                     reinterpret_cast<uint8_t *>(out + j), s[b][0], s[b][1], s[b][2],
                                     s[b][3], tail);
                }
            }
        }
    }
}

// Blocks [first, last) of the `tile`-th run of `tile_groups` counter groups
// of a request with nb blocks and IV low byte v0 (tiles are group-aligned so
// no group is split between two tiles).
__device__ __forceinline__ void tile_blocks_of(uint64_t tile, uint32_t tile_groups, uint64_t v0, uint64_t nb,
                                               uint64_t *first, uint64_t *last)
{
    const uint64_t g0 = tile * tile_groups, g1 = g0 + tile_groups;
    *first = g0 == 0 ? 0 : (g0 << 8) - v0;
    const uint64_t e = (g1 << 8) - v0;
    *last = e < nb ? e : nb;
}

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
// and warp and five lookups per block were 8.4.  The next chunk's plaintext is loaded
// before the current chunk's rounds.  Nothing past len is touched; the final
// partial block is done bytewise.
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
            uint32_t s[1][4] = {{group.x ^ mine.x, group.y ^ mine.y, group.z ^ mine.z, group.w ^ mine.w}};
            aestt::rounds<3, NR, 1>(s, ln, rk);
            const uint32_t i = c * 32u + lane;
            if (i >= lo && i < hi)
                aesdev::st_stream(op + c * 32u, make_uint4(pt.x ^ s[0][0], pt.y ^ s[0][1], pt.z ^ s[0][2],
                                                           pt.w ^ s[0][3]));
            else if (i == partial)
                aesdev::xor_tail(reinterpret_cast<const uint8_t *>(ip + c * 32u),
                                 reinterpret_cast<uint8_t *>(op + c * 32u), s[0][0], s[0][1], s[0][2], s[0][3],
                                 tail);
        }
    }
}

}  // namespace aestile
