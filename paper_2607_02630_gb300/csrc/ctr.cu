// ctr.cu -- single-buffer AES-CTR kernels (SP 800-38A Sec. 6.5).
//
// Two variants of the block cipher, same contract:
//   T-table  : each CTA owns a contiguous run of 32-block chunks of the
//              counter space, its warps take them in turn (lane l the block
//              whose counter low byte is l + 32m, so every load/store
//              instruction of the warp moves 512 contiguous bytes); rounds from
//              T-tables in bank-replicated shared memory with counter-mode
//              caching of rounds 1-2 (aes_ttable.cuh).  About 136 KiB of shared
//              memory, or 72 KiB with two tables; one CTA per SM.
//   bitsliced: each warp owns 1024 consecutive blocks; lane l holds blocks
//              base + l + 32k (k = 0..31) as 128 bit planes (aes_bitslice.cuh),
//              so loads/stores are again 512 contiguous bytes per instruction.
// Both compute the counter block T_1 + j in registers, xor the keystream
// into the plaintext with 16-byte streaming loads/stores, and handle the
// final partial block bytewise without touching bytes past len.
#include "internal.h"
#include "common.cuh"
#include "aes_ttable.cuh"
#include "bs_tile.cuh"

namespace {

using aesrt::CtrParams;

// Counter groups whose round-2 constants a CTA holds at once (16 bytes each).
constexpr uint32_t kGroupsPerPass = 512;
template <int TABLES>
constexpr size_t kCtrSmem = aestt::kTableBytesOf<TABLES> + kGroupsPerPass * sizeof(uint4);

// Single-buffer T-table kernel, bound by shared-memory wavefronts: per
// 32-block chunk the 16 * (NR - 2) lookups of rounds 3..NR, one broadcast
// load of the group's round-2 constants and 8 for the payload in and out.
//
// Split: with v0 the IV's low byte, block j sits at counter position
// v0 + j, and position >> 5 is its chunk.  The chunks are cut into gridDim.x
// equal contiguous runs, one per CTA, so SMs differ by at most one chunk
// (whole 256-block groups dealt out to warps left the busiest SM 1.3 times
// the mean at 8 and 64 MiB).  In the run, warp w takes chunks w, w + W, ...;
// W is a multiple of 8 in the usual shapes, so a lane's counter low byte
// never changes and its part of round 2 (lane_round2) is computed once.  The
// groups' part (group_round2) is computed once per CTA, one group per
// thread.  Both cost 27 + 40 lookups per group and warp when each warp
// derived them for itself: 8.4 of 144 wavefronts per chunk.
// The next chunk's plaintext is loaded before the current one's rounds, so
// a chunk's whole time (about 1 us with 16 warps) covers the DRAM latency.
// One block per lane in flight: two gave 1.27 (1 MiB), 1.06 (8 MiB) and
// 0.99-1.01 (256 MiB) times the time of one.
// Measured (AES-128, launches in a CUDA graph): 1 MiB 5.05 -> 4.05 us, 8 MiB
// 13.4 -> 10.7 us, 256 MiB 263 -> 240 us (1.12 TB/s; 137 wavefronts per
// chunk at the measured rate and 2070 MHz are 228 us).  Back to back on a
// stream, with the set-up overlapped (launch_overlapped): 1 MiB 3.5 us, 8 MiB
// 10.2 us (9.4 with two tables).
//
// With two tables (64 KiB) and 512 threads, two CTAs fit an SM, so the next
// launch's CTAs set up beside the running ones instead of after them.
template <int NR, int TABLES>
__global__ void __launch_bounds__(TABLES == 2 ? 512 : 1024, TABLES == 2 ? 2 : 1)
    ctr_ttable_kernel(const __grid_constant__ CtrParams p)
{
    extern __shared__ __align__(128) uint8_t smem[];
    uint4 *s_group = reinterpret_cast<uint4 *>(smem + aestt::kTableBytesOf<TABLES>);
    aesdev::let_next_launch_start();
    aestt::fill_tables<TABLES>(smem, p.te0);
    __syncthreads();
    const aestt::LanesOf<TABLES> ln(smem);
    const aestt::RkConst rk{p.rk};
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const uint64_t nblocks = (p.len + 15) >> 4, nfull = p.len >> 4;
    const uint64_t v0 = p.iv_lo & 255u, base_lo = p.iv_lo & ~(uint64_t)255u;
    const uint64_t first = v0 >> 5, chunks = ((v0 + nblocks - 1) >> 5) - first + 1;
    // this CTA's run; q * CTAs + r = chunks avoids the product chunks * blockIdx.x
    const uint64_t q = chunks / gridDim.x, r = chunks % gridDim.x;
    const uint64_t k_begin = first + q * blockIdx.x + (blockIdx.x < r ? blockIdx.x : r);
    const uint64_t k_end = k_begin + q + (blockIdx.x < r ? 1 : 0);
    uint4 mine = make_uint4(0, 0, 0, 0);  // lane_round2 of the lane's counter low byte
    uint64_t mine_for = ~0ull;            // (counter bits 40.., m) it belongs to
    for (uint64_t ka = k_begin; ka < k_end;) {
        const uint64_t ga = ka >> 3;
        const uint64_t kb = k_end < (ga + kGroupsPerPass) << 3 ? k_end : (ga + kGroupsPerPass) << 3;
        const uint32_t ng = (uint32_t)(((kb - 1) >> 3) - ga) + 1;
        if (ka != k_begin)
            __syncthreads();  // every warp is done with the previous constants
        for (uint32_t t = threadIdx.x; t < ng; t += blockDim.x) {
            const uint64_t l = base_lo + ((ga + t) << 8);
            s_group[t] = aestt::group_round2(aestt::CounterWords(p.iv_hi + (l < base_lo ? 1 : 0), l), ln, rk);
        }
        if (ka == k_begin)
            aesdev::wait_for_previous_launch();  // no payload byte is touched before
        // a block index before the message's first (first chunk) wraps and fails j < nfull
        uint64_t k = ka + warp, j = (k << 5) + lane - v0;
        uint4 next = make_uint4(0, 0, 0, 0);
        if (k < kb && j < nfull)
            next = aesdev::ld_stream(p.in + j);
        __syncthreads();
        for (; k < kb; k += nwarps) {
            const uint4 pt = next;
            const uint64_t jn = j + 32u * nwarps;
            if (k + nwarps < kb && jn < nfull)
                next = aesdev::ld_stream(p.in + jn);
            const uint64_t g = k >> 3, l = base_lo + (g << 8);
            const uint64_t tag = (l >> 40) << 3 | (k & 7u);
            if (tag != mine_for) {
                const aestt::CounterWords ctr(p.iv_hi + (l < base_lo ? 1 : 0), l);
                mine = aestt::lane_round2(aestt::column0_round1(ctr, ln, rk), ((uint32_t)k & 7u) * 32u + lane, ln, rk);
                mine_for = tag;
            }
            const uint4 group = s_group[g - ga];
            uint32_t s[4] = {group.x ^ mine.x, group.y ^ mine.y, group.z ^ mine.z, group.w ^ mine.w};
            aestt::rounds<3, NR>(s, ln, rk);
            if (j < nfull)
                aesdev::st_stream(p.out + j, make_uint4(pt.x ^ s[0], pt.y ^ s[1], pt.z ^ s[2], pt.w ^ s[3]));
            else if (j == nfull && (p.len & 15))  // the final partial block
                aesdev::xor_tail(reinterpret_cast<const uint8_t *>(p.in + j), reinterpret_cast<uint8_t *>(p.out + j),
                                 s[0], s[1], s[2], s[3], (uint32_t)(p.len & 15));
            j = jn;
        }
        ka = kb;
    }
}

template <int NR>
__global__ void __launch_bounds__(128) ctr_bitslice_kernel(const __grid_constant__ CtrParams p)
{
    __shared__ __align__(16) uint32_t bsk[(NR + 1) * 128];
    aesbs::build_masks(bsk, p.rk, NR, threadIdx.x, blockDim.x);
    __syncthreads();
    const uint32_t rk0[4] = {p.rk[0], p.rk[1], p.rk[2], p.rk[3]};
    const uint64_t gwarp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    aesbs::xor_range<NR>(p.in, p.out, p.len, p.iv_hi, p.iv_lo, rk0, 0, (p.len + 15) >> 4, gwarp, nwarps,
                         aesbs::MaskKeys{reinterpret_cast<const uint4 *>(bsk)});
}

template <int NR>
cudaError_t set_tt_attr()
{
    const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const cudaError_t e = cudaFuncSetAttribute(ctr_ttable_kernel<NR, 4>, attr, (int)kCtrSmem<4>);
    return e ? e : cudaFuncSetAttribute(ctr_ttable_kernel<NR, 2>, attr, (int)kCtrSmem<2>);
}

// Two tables from 2 to 16 MiB, where a launch's set-up counts and the extra
// logic operations hide behind the lookups; four below (one chunk per warp:
// the longer chain of a round counts) and above.  Launches in a row, four and
// two tables, AES-128 and AES-256:
//   1 MiB     3.26 3.29 us   3.72 4.16 us      8 MiB    9.9  9.4    13.2  12.75
//   1.25 MiB  3.67 3.88      4.34 3.74         16 MiB   17.4 17.1   24.0  23.7
//   1.5 MiB   3.87 3.14      4.57 3.84         20 MiB   20.94 20.82  29.3 29.1
//   2 MiB     4.18 3.47      5.01 4.32         32 MiB   32.0 32.1   45.3  45.3
//   4 MiB     6.30 5.65      8.03 7.39         256 MiB  241.9 245.3  348  352
// The upper line is where they meet; the lower one is on the safe side (1.25
// MiB goes either way, 1.5 MiB would gain).
bool two_tables(uint64_t len, int threads) { return len >= (2u << 20) && len <= (16u << 20) && threads == 512; }

template <int NR>
cudaError_t launch_tt(const CtrParams &p, int ctas, int threads, cudaStream_t stream)
{
    if (two_tables(p.len, threads))
        return aesrt::launch_overlapped(ctr_ttable_kernel<NR, 2>, ctas, threads, kCtrSmem<2>, stream, p);
    return aesrt::launch_overlapped(ctr_ttable_kernel<NR, 4>, ctas, threads, kCtrSmem<4>, stream, p);
}

}  // namespace

namespace aesrt {

cudaError_t ctr_set_attributes()
{
    cudaError_t e;
    if ((e = set_tt_attr<10>()) || (e = set_tt_attr<12>()) || (e = set_tt_attr<14>()))
        return e;
    return cudaSuccess;
}

// CTAs per SM of one launch: one T-table CTA (it keeps the lookups busy, and
// four tables fill most of an SM's shared memory); bitsliced CTAs of 128
// threads are bound by registers.
int ctr_max_ctas(const CtrShape &s, int nsm)
{
    if (s.variant == 2)
        return nsm * (s.threads <= 128 ? 2 : 1);
    return nsm;
}

int ctr_ctas(uint64_t nblocks, uint32_t v0, const CtrShape &s, int nsm)
{
    const uint64_t cap = (uint64_t)ctr_max_ctas(s, nsm);
    uint64_t want;
    if (s.ctas > 0) {
        want = (uint64_t)s.ctas;
    } else if (s.variant == 2) {
        const uint64_t warps = (uint64_t)(s.threads / 32);
        want = ((nblocks + 1023) / 1024 + warps - 1) / warps;  // a bitsliced warp takes 1024 blocks per pass
    } else {
        // One CTA per 8 chunks of 32 blocks until every SM has one.  One per
        // chunk is done 0.2 us sooner on an idle GPU (16 and 64 KiB in a CUDA
        // graph: 3.6 and 3.8 us, 3.85 and 4.0 with 8 chunks, 4.4 and 4.5 with
        // 16; calls in a row 2.5 us with each), but every CTA fills its tables
        // for what may be one warp's work, and where SMs are wanted by others
        // that is the cost: 64 KiB calls from 8 streams 2.24 us a call with 1
        // chunk, 1.19 with 2, 0.68 with 4, 0.61 with 8, 0.66 with 16; one such
        // call beside the resident server (4 SMs free) 77.8, 43, 24.7, 16.8
        // and 12.8 us.
        const uint64_t chunks = nblocks ? ((v0 + nblocks - 1) >> 5) - (v0 >> 5) + 1 : 1;
        const uint64_t per = s.threads < 256 ? (uint64_t)(s.threads / 32) : 8;  // a warp takes one
        want = (chunks + per - 1) / per;
    }
    if (want > cap)
        want = cap;
    return want < 1 ? 1 : (int)want;
}

cudaError_t launch_ctr(const CtrParams &p, int nr, const CtrShape &s, int nsm, cudaStream_t stream)
{
    const uint64_t nblocks = aesrt::blocks_of(p.len);
    if (!nblocks)
        return cudaSuccess;
    const int ctas = ctr_ctas(nblocks, (uint32_t)(p.iv_lo & 255u), s, nsm);
    if (s.variant == 2) {
        if (s.threads != 128)
            return cudaErrorInvalidValue;
        switch (nr) {
        case 10: ctr_bitslice_kernel<10><<<ctas, 128, 0, stream>>>(p); break;
        case 12: ctr_bitslice_kernel<12><<<ctas, 128, 0, stream>>>(p); break;
        case 14: ctr_bitslice_kernel<14><<<ctas, 128, 0, stream>>>(p); break;
        default: return cudaErrorInvalidValue;
        }
        return cudaGetLastError();
    }
    switch (nr) {
    case 10: return launch_tt<10>(p, ctas, s.threads, stream);
    case 12: return launch_tt<12>(p, ctas, s.threads, stream);
    case 14: return launch_tt<14>(p, ctas, s.threads, stream);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace aesrt
