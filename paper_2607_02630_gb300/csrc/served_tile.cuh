// served_tile.cuh -- a served request's tile: blocks [first, last) of one
// message by counter groups, two blocks per lane in flight.
//
// The batch kernel's chunk runs (tile.cuh) need fewer lookups, and served
// bursts of large requests ran 8 % faster with them (640 against 594 GB/s on
// the served mix from native submitters), but 4096 requests of log-uniform
// lengths 26 % slower (300 against 403 GB/s), with one block in flight or two:
// so the served workers keep this walk.
#pragma once
#include "internal.h"
#include "common.cuh"
#include "aes_ttable.cuh"

namespace aesserved {

using aestt::Lanes;
using aestt::te;

// Rounds R0..NR-1 (full) and the final round NR on NB blocks held as
// s[b][0..3] (little-endian column words), in place.  The state passed in is
// the output of round R0 - 1.
template <int R0, int NR, int NB, class RK>
__device__ __forceinline__ void rounds(uint32_t (&s)[NB][4], const Lanes &ln,
                                       const RK &rk)
{
#pragma unroll
    for (int r = R0; r < NR; ++r) {
        const uint4 k = rk.get(r);
        const uint32_t kk[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const uint32_t a[4] = {s[b][0], s[b][1], s[b][2], s[b][3]};
#pragma unroll
            for (int c = 0; c < 4; ++c)
                s[b][c] = te<0, 0>(a[c], ln) ^ te<1, 1>(a[(c + 1) & 3], ln) ^
                          te<2, 2>(a[(c + 2) & 3], ln) ^ te<3, 3>(a[(c + 3) & 3], ln) ^ kk[c];
        }
    }
    {
        // Final round: byte r of output column c is S(s_{c+r}.b_r), taken
        // from the byte of a T-table entry that holds the plain S-box value:
        // Te2 byte 0, Te3 byte 1, Te0 byte 2, Te1 byte 3.
        const uint4 k = rk.get(NR);
        const uint32_t kk[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const uint32_t a[4] = {s[b][0], s[b][1], s[b][2], s[b][3]};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint32_t x0 = te<2, 0>(a[c], ln);            // byte 0
                const uint32_t x1 = te<3, 1>(a[(c + 1) & 3], ln);  // byte 1
                const uint32_t x2 = te<0, 2>(a[(c + 2) & 3], ln);  // byte 2
                const uint32_t x3 = te<1, 3>(a[(c + 3) & 3], ln);  // byte 3
                const uint32_t lo = __byte_perm(x0, x1, 0x3250);
                const uint32_t hi = __byte_perm(x2, x3, 0x7210);
                s[b][c] = __byte_perm(lo, hi, 0x7610) ^ kk[c];
            }
        }
    }
}

// Counter-mode caching.  The 256 counter blocks T = G*256 + L (L = 0..255)
// of one counter group share bytes 0..14, so after AddRoundKey only byte 15
// (row 3 of column 3, through Te3 into output column 0) varies in round 1:
// round 1 gives columns (P0 ^ Te3[L ^ k15], C1, C2, C3) with P0, C1..C3 fixed
// for the group.  In round 2 the varying column 0 feeds exactly one lookup of
// each output column (row r of column 0 reaches column -r mod 4), so round 2
// is Q_c ^ (one lookup) with Q0..Q3 fixed for the group.  A block then needs 5
// lookups for rounds 1-2 instead of 32; the group constants cost 27 lookups
// once per group.
struct Group {
    uint32_t p0, c1, c2, c3, q0, q1, q2, q3, k15;
};

// base: the group's first counter block (byte 15 = 0) as column words.
template <class RK>
__device__ __forceinline__ Group group_consts(const uint32_t base[4], const Lanes &ln,
                                              const RK &rk)
{
    const uint4 k0 = rk.get(0), k1 = rk.get(1), k2 = rk.get(2);
    const uint32_t s0 = base[0] ^ k0.x, s1 = base[1] ^ k0.y, s2 = base[2] ^ k0.z, s3 = base[3] ^ k0.w;
    Group g;
    g.k15 = k0.w >> 24;
    g.p0 = te<0, 0>(s0, ln) ^ te<1, 1>(s1, ln) ^ te<2, 2>(s2, ln) ^ k1.x;
    g.c1 = te<0, 0>(s1, ln) ^ te<1, 1>(s2, ln) ^ te<2, 2>(s3, ln) ^ te<3, 3>(s0, ln) ^ k1.y;
    g.c2 = te<0, 0>(s2, ln) ^ te<1, 1>(s3, ln) ^ te<2, 2>(s0, ln) ^ te<3, 3>(s1, ln) ^ k1.z;
    g.c3 = te<0, 0>(s3, ln) ^ te<1, 1>(s0, ln) ^ te<2, 2>(s1, ln) ^ te<3, 3>(s2, ln) ^ k1.w;
    g.q0 = te<1, 1>(g.c1, ln) ^ te<2, 2>(g.c2, ln) ^ te<3, 3>(g.c3, ln) ^ k2.x;
    g.q1 = te<0, 0>(g.c1, ln) ^ te<1, 1>(g.c2, ln) ^ te<2, 2>(g.c3, ln) ^ k2.y;
    g.q2 = te<0, 0>(g.c2, ln) ^ te<1, 1>(g.c3, ln) ^ te<3, 3>(g.c1, ln) ^ k2.z;
    g.q3 = te<0, 0>(g.c3, ln) ^ te<2, 2>(g.c1, ln) ^ te<3, 3>(g.c2, ln) ^ k2.w;
    return g;
}

// Keystream of NB blocks of one group, L[b] = the blocks' low counter bytes.
template <int NR, int NB, class RK>
__device__ __forceinline__ void encrypt_group(uint32_t (&s)[NB][4], const uint32_t (&L)[NB], const Group &g,
                                              const Lanes &ln, const RK &rk)
{
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        const uint32_t r10 = g.p0 ^ te<3, 0>(L[b] ^ g.k15, ln);  // Te3[byte 15]
        s[b][0] = g.q0 ^ te<0, 0>(r10, ln);
        s[b][1] = g.q1 ^ te<3, 3>(r10, ln);
        s[b][2] = g.q2 ^ te<2, 2>(r10, ln);
        s[b][3] = g.q3 ^ te<1, 1>(r10, ln);
    }
    rounds<3, NR, NB>(s, ln, rk);
}

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
                                          const Lanes &ln, const RK &rk)
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
    Group gc;
    for (uint64_t u = warp0; u < u_end; u += warp_stride) {
        const uint64_t g = g_first + u / parts;
        const uint32_t m_begin = (uint32_t)(u % parts) * per;
        if (g != gc_for) {
            uint32_t base[4];
            const uint64_t l = base_lo + (g << 8);
            const uint64_t h = iv_hi + (l < base_lo ? 1ull : 0ull);
            base[0] = aesdev::bswap32((uint32_t)(h >> 32));
            base[1] = aesdev::bswap32((uint32_t)h);
            base[2] = aesdev::bswap32((uint32_t)(l >> 32));
            base[3] = aesdev::bswap32((uint32_t)l);
            gc = group_consts(base, ln, rk);
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
            encrypt_group<NR, NB>(s, L, gc, ln, rk);
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

}  // namespace aesserved
