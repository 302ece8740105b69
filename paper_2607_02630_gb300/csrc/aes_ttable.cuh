// aes_ttable.cuh -- AES rounds from T-tables in bank-replicated shared memory.
//
// One full round (FIPS-197 Sec. 5.1: SubBytes, ShiftRows, MixColumns,
// AddRoundKey) is, per output column c,
//   t_c = Te0[s_c.b0] ^ Te1[s_{c+1}.b1] ^ Te2[s_{c+2}.b2] ^ Te3[s_{c+3}.b3] ^ k_c
// where s_c is column c of the state as a little-endian word (byte r = row
// r), s_c.b_r its byte r, and Te_r[x] the column r of the MixColumns matrix
// times S(x): Te0[x] = (2S, S, S, 3S) in bytes 0..3 and Te_r = Te0 rotated
// left by 8r bits.  The final round has no MixColumns and takes S(x) out of
// the byte of Te_r that holds the plain S(x).
//
// Layout (32 KiB a table, 128 KiB per CTA): entry e of Te_r, copy for lane l, is the word at
// byte r*32768 + e*128 + l*4.  Every lane reads its own copy, so the 32 lanes
// of a warp always hit 32 distinct banks (conflict-free).  The byte offset of
// a lookup is 128 * (state byte K) + 4 * lane: one four-way byte dot product
// with the weights 0x80 << 8K (dp4a), the table's base being the load's
// immediate.  The dot product issues on the multiply pipe, 64 lanes a clock
// beside the logic pipe's 64 (measured: the two alternating reach 117), so a
// round's 16 offsets no longer share the logic pipe with its xors, as byte
// permutes did.  The pipe that bounds the rounds stays the shared-memory
// lookups, 32 lanes a clock.  One 8 MiB AES-128 buffer: 10.99 us with byte
// permutes, 10.68 us so; 256 MiB 243.5 and 240.1 us.
//
// With TABLES == 2 only Te0 and Te1 are kept: Te2 and Te3 are their halves
// swapped, and a column's two lookups there are swapped together by one more
// permute.  That halves the fill and the shared memory, for 8 more logic
// operations a round.
#pragma once
#include <stdint.h>

namespace aestt {

constexpr uint32_t kOneTable = 32768;
template <int TABLES>
constexpr uint32_t kTableBytesOf = TABLES * kOneTable;
constexpr uint32_t kTableBytes = kTableBytesOf<4>;

// The shared address of the calling lane's copy of entry 0 of Te0; made after
// the barrier that follows fill_tables.  The address rides in the dot
// product's accumulator, so a lookup is the dot product and the load and
// nothing else: left to the compiler, some instantiations added the tables'
// base to every offset (131 more instructions per 32 AES-128 blocks in the
// batch kernel, 64 MiB 84.2 us instead of 76.3).
template <int TABLES>
struct LanesOf {
    static constexpr int kTables = TABLES;
    uint32_t a;
    __device__ __forceinline__ explicit LanesOf(const uint8_t *tables)
        : a((uint32_t)__cvta_generic_to_shared(tables) + (threadIdx.x & 31u) * 4u)
    {
        // every lookup depends on this value and so stays behind the barrier
        asm volatile("" : "+r"(a)::"memory");
    }
};
using Lanes = LanesOf<4>;

__device__ __forceinline__ uint32_t swap_halves(uint32_t v) { return __byte_perm(v, 0, 0x1032); }

// Te_T[byte K of x].
template <int T, int K, class LN>
__device__ __forceinline__ uint32_t te(uint32_t x, const LN &ln)
{
    constexpr int kAt = LN::kTables == 4 ? T : T & 1;
    uint32_t v;
    asm("ld.shared.u32 %0, [%1 + %2];" : "=r"(v) : "r"(__dp4a(x, 0x80u << (8 * K), ln.a)), "n"(kAt * kOneTable));
    return kAt == T ? v : swap_halves(v);
}

// Fill the replicated tables from Te0 (256 words in global memory).  Must be
// followed by __syncthreads() before the first lookup.  Te0 is first staged
// in a 1 KiB shared array (one global round trip for the whole CTA); then
// each thread takes an entry's 16-byte chunk of four lane copies and writes
// it to every table, consecutive threads to consecutive chunks (no bank
// conflicts).  The fill is most of a short launch's fixed cost.
template <int TABLES = 4>
__device__ __forceinline__ void fill_tables(uint8_t *smem, const uint32_t *__restrict__ te0)
{
    __shared__ uint32_t s_te0[256];
    for (uint32_t e = threadIdx.x; e < 256u; e += blockDim.x)
        s_te0[e] = __ldg(te0 + e);
    __syncthreads();
#pragma unroll 2
    for (uint32_t q = threadIdx.x; q < kOneTable / 16; q += blockDim.x) {
        const uint32_t v = s_te0[q >> 3];  // entry e = q / 8
#pragma unroll
        for (int t = 0; t < TABLES; ++t) {
            const uint32_t val = t ? __funnelshift_l(v, v, 8 * t) : v;
            *reinterpret_cast<uint4 *>(smem + t * kOneTable + q * 16u) = make_uint4(val, val, val, val);
        }
    }
}

// Round keys stored as kernel parameters (constant bank) -- the single-key
// launch.  Indices are compile-time after unrolling, so the words are
// instruction operands and cost no registers or loads.
struct RkConst {
    const uint32_t *w;
    __device__ __forceinline__ uint4 get(int r) const
    {
        return make_uint4(w[4 * r], w[4 * r + 1], w[4 * r + 2], w[4 * r + 3]);
    }
};

// Round keys staged in shared memory (per-request keys in batch CTAs of more
// than 512 threads); one broadcast 16-byte load per round.
struct RkShared {
    const uint4 *w;
    __device__ __forceinline__ uint4 get(int r) const { return w[r]; }
};

// Round keys held in registers -- the batch kernel's warps, one request at a
// time.  The schedule is read once per run (NR + 1 uniform 16-byte loads);
// indices are compile-time after unrolling, so every round's key is four
// register operands and costs no shared-memory wavefront.  The price is
// 4 * (NR + 1) registers a thread, which the 512-thread batch CTA can pay.
template <int NR>
struct RkRegs {
    uint4 w[NR + 1];
    __device__ __forceinline__ explicit RkRegs(const uint4 *__restrict__ g)
    {
#pragma unroll
        for (int r = 0; r <= NR; ++r)
            w[r] = __ldg(g + r);
    }
    __device__ __forceinline__ uint4 get(int r) const { return w[r]; }
};

// Rounds R0..NR-1 (full) and the final round NR on one block held as s[0..3]
// (little-endian column words), in place.  The state passed in is the output
// of round R0 - 1.
template <int R0, int NR, class LN, class RK>
__device__ __forceinline__ void rounds(uint32_t (&s)[4], const LN &ln, const RK &rk)
{
    constexpr bool kFour = LN::kTables == 4;
#pragma unroll
    for (int r = R0; r < NR; ++r) {
        const uint4 k = rk.get(r);
        const uint32_t kk[4] = {k.x, k.y, k.z, k.w};
        const uint32_t a[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if constexpr (kFour)
                s[c] = te<0, 0>(a[c], ln) ^ te<1, 1>(a[(c + 1) & 3], ln) ^ te<2, 2>(a[(c + 2) & 3], ln) ^
                       te<3, 3>(a[(c + 3) & 3], ln) ^ kk[c];
            else
                s[c] = te<0, 0>(a[c], ln) ^ te<1, 1>(a[(c + 1) & 3], ln) ^ kk[c] ^
                       swap_halves(te<0, 2>(a[(c + 2) & 3], ln) ^ te<1, 3>(a[(c + 3) & 3], ln));
        }
    }
    // Final round: byte r of output column c is S(s_{c+r}.b_r), taken from a
    // byte of a T-table entry that holds the plain S-box value: Te2 byte 0,
    // Te3 byte 1, Te0 byte 2 and Te1 byte 3, which need no moving, or byte 1
    // of Te0.
    const uint4 k = rk.get(NR);
    const uint32_t kk[4] = {k.x, k.y, k.z, k.w};
    const uint32_t a[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const uint32_t a0 = a[c], a1 = a[(c + 1) & 3], a2 = a[(c + 2) & 3], a3 = a[(c + 3) & 3];
        const uint32_t lo = kFour ? __byte_perm(te<2, 0>(a0, ln), te<3, 1>(a1, ln), 0x3250)
                                  : __byte_perm(te<0, 0>(a0, ln), te<0, 1>(a1, ln), 0x3251);
        const uint32_t hi = kFour ? __byte_perm(te<0, 2>(a2, ln), te<1, 3>(a3, ln), 0x7210)
                                  : __byte_perm(te<0, 2>(a2, ln), te<0, 3>(a3, ln), 0x5110);
        s[c] = __byte_perm(lo, hi, 0x7610) ^ kk[c];
    }
}

// Counter-mode caching.  The 256 counter blocks T = G*256 + L (L = 0..255)
// of one counter group share bytes 0..14, so after AddRoundKey only byte 15
// (row 3 of column 3, through Te3 into output column 0) varies in round 1:
// round 1 gives columns (P0 ^ Te3[L ^ k15], C1, C2, C3) with P0, C1..C3 fixed
// for the group.  In round 2 the varying column 0 feeds exactly one lookup of
// each output column (row r of column 0 reaches column -r mod 4), so round 2
// is Q_c ^ (one lookup) with Q0..Q3 fixed for the group.  The two halves are
// each computed once for a whole run, and a block's state after round 2 is
// one xor of four words:
//   round-2 state = group_round2(upper 15 counter bytes) ^ lane_round2(L)
// group_round2 holds what byte 15 does not touch (Q0..Q3 above).  lane_round2
// is byte 15's part: through P0 it also depends on counter bytes 0, 5 and 10,
// i.e. it is the same for every group until the counter carries into byte 10
// (every 2^40 blocks), so a lane that stays on one L keeps it in registers.
// ctr: a counter block's upper and lower 64 bits (byte 15 is ignored).
struct CounterWords {
    uint32_t w[4];
    __device__ __forceinline__ CounterWords(uint64_t hi, uint64_t lo)
    {
        w[0] = __byte_perm((uint32_t)(hi >> 32), 0, 0x0123);
        w[1] = __byte_perm((uint32_t)hi, 0, 0x0123);
        w[2] = __byte_perm((uint32_t)(lo >> 32), 0, 0x0123);
        w[3] = __byte_perm((uint32_t)lo, 0, 0x0123);
    }
};

// 27 lookups.
template <class LN, class RK>
__device__ __forceinline__ uint4 group_round2(const CounterWords &ctr, const LN &ln, const RK &rk)
{
    const uint4 k0 = rk.get(0), k1 = rk.get(1), k2 = rk.get(2);
    const uint32_t s0 = ctr.w[0] ^ k0.x, s1 = ctr.w[1] ^ k0.y, s2 = ctr.w[2] ^ k0.z, s3 = ctr.w[3] ^ k0.w;
    const uint32_t c1 = te<0, 0>(s1, ln) ^ te<1, 1>(s2, ln) ^ te<2, 2>(s3, ln) ^ te<3, 3>(s0, ln) ^ k1.y;
    const uint32_t c2 = te<0, 0>(s2, ln) ^ te<1, 1>(s3, ln) ^ te<2, 2>(s0, ln) ^ te<3, 3>(s1, ln) ^ k1.z;
    const uint32_t c3 = te<0, 0>(s3, ln) ^ te<1, 1>(s0, ln) ^ te<2, 2>(s1, ln) ^ te<3, 3>(s2, ln) ^ k1.w;
    return make_uint4(te<1, 1>(c1, ln) ^ te<2, 2>(c2, ln) ^ te<3, 3>(c3, ln) ^ k2.x,
                      te<0, 0>(c1, ln) ^ te<1, 1>(c2, ln) ^ te<2, 2>(c3, ln) ^ k2.y,
                      te<0, 0>(c2, ln) ^ te<1, 1>(c3, ln) ^ te<3, 3>(c1, ln) ^ k2.z,
                      te<0, 0>(c3, ln) ^ te<2, 2>(c1, ln) ^ te<3, 3>(c2, ln) ^ k2.w);
}

// The part of lane_round2 that all lanes share: round 1's column 0 without
// byte 15's lookup.
template <class LN, class RK>
__device__ __forceinline__ uint32_t column0_round1(const CounterWords &ctr, const LN &ln, const RK &rk)
{
    const uint4 k0 = rk.get(0), k1 = rk.get(1);
    return te<0, 0>(ctr.w[0] ^ k0.x, ln) ^ te<1, 1>(ctr.w[1] ^ k0.y, ln) ^ te<2, 2>(ctr.w[2] ^ k0.z, ln) ^ k1.x;
}

template <class LN, class RK>
__device__ __forceinline__ uint4 lane_round2(uint32_t column0, uint32_t L, const LN &ln, const RK &rk)
{
    const uint32_t r10 = column0 ^ te<3, 0>(L ^ (rk.get(0).w >> 24), ln);
    return make_uint4(te<0, 0>(r10, ln), te<3, 3>(r10, ln), te<2, 2>(r10, ln), te<1, 1>(r10, ln));
}

}  // namespace aestt
