// batch.cu -- many independent AES-CTR requests in one launch.
//
// Work is measured in shared-memory wavefronts, the unit of the kernel's
// bound: a 32-block chunk (tile.cuh) of a request with Nr rounds costs about
// 16 (Nr - 2) + 9 of them.  The requests' chunks, one request after the other,
// are one line of cost.  Its tiles are claimed in one of two ways.
//   By pieces: CTA c of G (one per SM) owns the c-th of G equal pieces of the
// line, so every SM gets the same number of lookups whatever the mix of
// lengths and key sizes, and neither a table of tiles nor a counter in device
// memory is needed.  The CTA's warps claim tiles of the piece through one
// counter in shared memory, each tile a warps-th of what is left, at most
// tile_blocks and at least about one chunk: large tiles amortise a request's
// set-up, small ones at the end let the warps finish together, and a batch of
// a few short requests is spread one chunk to a warp.
//   From the whole line (WHOLE): every warp of the grid claims through one
// counter in device memory, each tile a share of what the line has left, at
// least 4 chunks.  SMs that other work holds, or that get less of the host
// link, then cost only their own share (measured at kWholeFrom); a claim costs
// a trip to L2 and back instead of one to shared memory.
// A warp finds its tile's request by a 32-way search over the requests' first
// costs.
//
// The cipher is the same T-table round code as the single-buffer kernel.
// Round keys: CTAs of up to 512 threads (the default) hold the current
// request's schedule in registers, so the shared-memory pipe, the kernel's
// bound, serves lookups only; larger CTAs stage it in each warp's slice of
// shared memory (one broadcast wavefront per round).
//
// The bitsliced kernel, the autotuner's alternative to the T-tables, cuts its
// work in passes of 1024 blocks: by pieces where the requests are in kernel
// parameters, else one pass to a claim from the whole line: 4096 requests of
// 1 KiB to 8 MiB 22.9 ms, by pieces 32.3, two passes to a claim 38.4 (probably
// because the warps of an SM then run the same unrolled rounds, of one key
// size, at the same time: the more neighbouring passes run together, the
// faster).
//
// With a tile order (a test aid) the line is cut into equal tiles instead,
// and tile t is processed as tile (a*t + b) mod T for a host-chosen a coprime
// to T (a permutation), so tiles complete in a scrambled order; results must
// not change.
#include "../../include/aesoffload.h"
#include "internal.h"
#include "runtime.h"
#include "common.cuh"
#include "aes_ttable.cuh"
#include "bs_tile.cuh"
#include "tile.cuh"

#include <algorithm>
#include <cstring>
#include <mutex>
#include <new>
#include <type_traits>
#include <vector>

namespace {

using aesrt::BatchReq;

struct TileOrder {
    uint64_t a, b;   // t -> (a*t + b) mod tiles
    uint64_t tiles;  // 0: no order, tiles are cut as they are claimed
};

// A request's work is cut in units: chunks for the T-table kernel, passes of 32
// chunks (1024 blocks) for the bitsliced one, which spends a whole pass on any
// part of it.  A chunk costs its shared-memory wavefronts: 16 lookups in each
// of the NR - 2 rounds that are not cached, and about 9 for the payload and
// the group constants.  A pass costs its rounds and, about as much as 5 of
// them, the transposes and the payload (323 and 254 GB/s at 10 and 14 rounds
// on a 256 MiB buffer).
struct TtUnit {
    static constexpr bool kEven = false;
    static constexpr uint32_t kChunks = 1;
    __host__ __device__ static constexpr uint32_t cost(uint32_t nr) { return 16u * (nr - 2u) + 9u; }
    static __device__ __forceinline__ uint32_t run(uint64_t iv_lo, uint64_t k0, uint64_t nk)
    {
        return aestile::run_chunks(iv_lo, k0, nk);
    }
};
// EVEN: every pass counts 1, for launches whose warps claim passes one by one.
template <bool EVEN>
struct BsUnitOf {
    static constexpr bool kEven = EVEN;
    static constexpr uint32_t kChunks = 32;
    __host__ __device__ static constexpr uint32_t cost(uint32_t nr) { return EVEN ? 1u : 16u * (nr + 5u); }
    static __device__ __forceinline__ uint32_t run(uint64_t, uint64_t, uint64_t nk)
    {
        return nk < kChunks ? (uint32_t)nk : kChunks;
    }
};

template <class UNIT>
__device__ __forceinline__ uint64_t ceil_units(uint64_t cost, uint32_t nr)
{
    switch (nr) {
    case 10: return (cost + UNIT::cost(10) - 1) / UNIT::cost(10);
    case 12: return (cost + UNIT::cost(12) - 1) / UNIT::cost(12);
    default: return (cost + UNIT::cost(14) - 1) / UNIT::cost(14);
    }
}

// One launch over n requests, none of them empty: in the kernel's own
// parameters (CAP of them at most) or, CAP == 0, in device memory, which is
// read only after wait_for_previous_launch.
struct BatchArgs {
    const BatchReq *reqs;  // CAP == 0
    uint32_t n;
    uint64_t total_cost;
    uint64_t tile_cost;  // largest tile
    const uint32_t *te0;
    TileOrder order;
};
template <int CAP>
struct BatchParams : BatchArgs {
    BatchReq in_params[CAP];
    __device__ __forceinline__ const BatchReq *requests() const { return in_params; }
    __device__ __forceinline__ unsigned long long *whole_line() const { return nullptr; }
    __device__ __forceinline__ void clear_next() const {}
};
static_assert(sizeof(BatchArgs) == 64, "requests in parameters start on a 64-byte line");
template <>
struct BatchParams<0> : BatchArgs {
    // Kernels that claim from the whole line: this launch's counter, zero when
    // it starts, and the next one's, which it clears.
    unsigned long long *claimed, *cleared;
    __device__ __forceinline__ const BatchReq *requests() const { return reqs; }
    __device__ __forceinline__ unsigned long long *whole_line() const { return claimed; }
    __device__ __forceinline__ void clear_next() const
    {
        if (blockIdx.x == 0 && threadIdx.x == 0)
            *cleared = 0;
    }
};

// Requests that fit the kernel's parameters (32764 bytes at most): a batch of
// up to so many needs no descriptor table in device memory, hence no
// allocation, no copy and no wait for one.  The small size keeps the launch
// of a small batch from copying 32 KB: calls of 1000-byte requests in a row,
// with it and with the large size, 1 request 3.8 and 4.3 us, 64 7.8 and 7.9
// (enqueued in 4.7-4.9 and 5.1-5.5); 65 requests, in the large size, 8.7.
constexpr int kFewInParams = 64;
constexpr int kMostInParams = 500;
static_assert(sizeof(BatchParams<kMostInParams>) <= 32764, "kernel parameters");
// Batches of up to so many requests never use a table in device memory.
constexpr int kMostByParams = AES_NOALLOC_MAX_REQUESTS;

// CTA sizes up to this hold round keys in registers.
constexpr int kRegsMaxThreads = 512;
// The bitsliced batch kernel's CTA size (its warps are register-bound).
constexpr int kBsThreads = 128;

// The last request of [lo, hi) whose first cost is <= x (reqs[lo] is one).
// The whole warp searches: every step reads 32 requests spread over the range
// and keeps the stretch between two of them, so 2^20 requests take 4 steps;
// near tells that the answer is probably within 32 requests of lo.
__device__ __forceinline__ uint32_t owner_of(const BatchReq *reqs, uint32_t lo, uint32_t hi, uint64_t x, bool near)
{
    const uint32_t lane = threadIdx.x & 31u;
    while (hi - lo > 1) {
        const uint32_t step = near ? 1u : (hi - lo + 31u) / 32u;
        const uint64_t i = (uint64_t)lo + (uint64_t)lane * step;
        const bool below = i < hi && reqs[i].cost_begin <= x;
        const uint32_t cnt = (uint32_t)__popc(__ballot_sync(0xffffffffu, below));  // >= 1: lane 0's is reqs[lo]
        lo += (cnt - 1u) * step;
        if (cnt < 32u && hi - lo > step)
            hi = lo + step;
        near = false;
    }
    return lo;
}

// Where a warp stands: what is left of its tile's cost range, and a request
// at or before it.  Kept in shared memory between runs: held in registers it
// was spilled around the bitsliced rounds and took registers from the
// lookups in flight.
struct WarpState {
    unsigned long long xa, xb;
    uint32_t ri, pad;
};

// The warp's next run: n > 0 chunks from chunk k0 on of request rq (every
// lane gets the same), or false when the CTA's piece (WHOLE: the line) is done.
// pos: the piece's counter in shared memory, the line's in device memory; st:
// this warp's state, which like the piece's counter is zeroed before the CTA's
// last barrier.
template <class UNIT, bool WHOLE>
__device__ __forceinline__ bool next_run(const BatchArgs &p, const BatchReq *reqs, unsigned long long *pos,
                                         WarpState *st, BatchReq &rq, uint64_t &k0, uint32_t &n)
{
    const uint32_t lane = threadIdx.x & 31u;
    __syncwarp();  // lane 0's last store to the state
    uint64_t xa = st->xa, xb = st->xb;
    uint32_t ri = st->ri;
    __syncwarp();  // before lane 0 writes the next
    for (;;) {
        bool near = true;  // the request is probably the last one or one of the next
        if (xa >= xb) {    // claim a tile of [u0, u0 + size)
            const uint64_t units = p.order.tiles ? p.order.tiles : p.total_cost;
            const uint64_t q = units / gridDim.x, r = units % gridDim.x;
            const uint64_t u0 = WHOLE ? 0 : q * blockIdx.x + (blockIdx.x < r ? blockIdx.x : r);
            const uint64_t size = WHOLE ? units : q + (blockIdx.x < r ? 1 : 0);
            unsigned long long at = 0, take = 1;
            if (lane == 0) {
                if (!p.order.tiles && !UNIT::kEven) {
                    const unsigned long long cur = *(volatile unsigned long long *)pos;
                    const uint32_t warps = (blockDim.x >> 5) * (WHOLE ? gridDim.x : 1u);
                    const uint32_t least = (WHOLE ? 4u : 1u) * UNIT::cost(10);
                    take = cur < size ? (size - cur) / warps : 0;
                    take = take < least ? least : take > p.tile_cost ? p.tile_cost : take;
                }
                at = atomicAdd(pos, take);
            }
            at = __shfl_sync(0xffffffffu, at, 0);
            take = __shfl_sync(0xffffffffu, take, 0);
            if (at >= size)
                return false;
            if (p.order.tiles) {
                const uint64_t t = (p.order.a * (u0 + at) + p.order.b) % p.order.tiles;
                xa = t * p.tile_cost;
                xb = xa + p.tile_cost < p.total_cost ? xa + p.tile_cost : p.total_cost;
                ri = 0;
                near = false;
            } else {
                near = xb != 0;  // the first tile may lie anywhere
                xa = u0 + at;
                xb = u0 + (at + take < size ? at + take : size);
            }
        }
        ri = owner_of(reqs, ri, p.n, xa, near);
        rq = reqs[ri];
        // a unit belongs to the tile that holds the first of its cost
        const uint64_t nb = (rq.len + 15) >> 4, v0 = rq.iv_lo & 255u, first = aestile::first_chunk(rq.iv_lo);
        const uint64_t nch = ((v0 + nb - 1) >> 5) - first + 1;
        const uint64_t all = (nch + UNIT::kChunks - 1) / UNIT::kChunks;
        const uint64_t ua = ceil_units<UNIT>(xa - rq.cost_begin, rq.nr);
        uint64_t ub = ceil_units<UNIT>(xb - rq.cost_begin, rq.nr);
        ub = ub < all ? ub : all;
        if (ua < ub) {
            const uint64_t c = ua * UNIT::kChunks, end = ub * UNIT::kChunks;
            k0 = first + c;
            n = UNIT::run(rq.iv_lo, k0, (end < nch ? end : nch) - c);
            if (lane == 0) {
                st->xa = rq.cost_begin + (ua + (n + UNIT::kChunks - 1) / UNIT::kChunks) * UNIT::cost(rq.nr);
                st->xb = xb;
                st->ri = ri;
            }
            return true;
        }
        xa = rq.cost_begin + all * UNIT::cost(rq.nr);  // on to the next request, or past the tile
    }
}

// The T-table batch kernel, bound by shared-memory wavefronts (95 % of the
// pipe busy on a 256 MiB AES-128 request).  Measured as plans against the
// kernel with a tile map, a device counter and two blocks per lane: 4096
// requests of 1 KiB to 8 MiB (3.66 GB) 4396 -> 4029 us, 512 of them 638 ->
// 562, 256 of 4 KiB to 1 MiB 111 -> 58, 64 of 1 to 16 KiB 37 -> 5.1 (one warp
// used to take up to 8 groups of a short request in turn).  Other CTA sizes
// on the 4096: 1024 threads (keys in shared memory) 4491 us, 256 threads
// 5148; 384 threads with up to 168 registers were 2 % faster on AES-256
// alone and 3 % slower on AES-128.  MAXT: largest CTA it is launched with;
// RK_REGS: round keys in registers (else in the warp's slice of shared
// memory); HOST: some payload lies in pinned host memory, and every request
// of the launch takes that walk (256 device requests of 4 KiB to 1 MiB 62.7
// us, one of them in pinned memory 65.6, or 63.0 with the device's walk for
// all; one in 16 62.7 and 59.6); WHOLE: claims from the whole line.
template <int MAXT, bool RK_REGS, int CAP, bool HOST, bool WHOLE>
__global__ void __launch_bounds__(MAXT, 1) batch_ttable_kernel(const __grid_constant__ BatchParams<CAP> p)
{
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ uint4 s_group[MAXT / 32][aestile::kRunGroups];
    __shared__ uint4 s_rk[RK_REGS ? 1 : MAXT / 32][15];  // round keys of each warp's current request
    __shared__ unsigned long long s_pos;
    __shared__ WarpState s_state[MAXT / 32];
    aesdev::let_next_launch_start();
    if (threadIdx.x == 0)
        s_pos = 0;
    if (threadIdx.x < MAXT / 32)
        s_state[threadIdx.x] = WarpState{0, 0, 0, 0};
    aestt::fill_tables(smem, p.te0);
    __syncthreads();
    aesdev::wait_for_previous_launch();
    if constexpr (WHOLE)
        p.clear_next();
    const aestt::Lanes ln(smem);
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    uint4 *w_group = s_group[warp];
    uint4 *w_rk = s_rk[RK_REGS ? 0 : warp];
    auto xor_with = [&](const BatchReq &rq, uint64_t k0, uint32_t n, auto nr) {
        constexpr int NR = decltype(nr)::value;
        auto go = [&](const auto &rk) {
            if constexpr (HOST)
                aestile::xor_run_host<NR>(rq.in, rq.out, rq.len, rq.iv_hi, rq.iv_lo, k0, n, w_group, ln, rk);
            else
                aestile::xor_run<NR>(rq.in, rq.out, rq.len, rq.iv_hi, rq.iv_lo, k0, n, w_group, ln, rk);
        };
        if constexpr (RK_REGS) {
            go(aestt::RkRegs<NR>(rq.rk));
        } else {
            if (lane <= NR)
                w_rk[lane] = rq.rk[lane];
            __syncwarp();
            go(aestt::RkShared{w_rk});
        }
    };
    BatchReq rq;
    uint64_t k0;
    uint32_t n;
    while (next_run<TtUnit, WHOLE>(p, p.requests(), WHOLE ? p.whole_line() : &s_pos, &s_state[warp], rq, k0, n)) {
        switch (rq.nr) {
        case 10: xor_with(rq, k0, n, std::integral_constant<int, 10>()); break;
        case 12: xor_with(rq, k0, n, std::integral_constant<int, 12>()); break;
        default: xor_with(rq, k0, n, std::integral_constant<int, 14>()); break;
        }
    }
}

// The bitsliced batch kernel: the same pieces and claims, each run encrypted
// by one warp 1024 blocks at a time (bs_tile.cuh) with the request's
// round-key bit planes in the warp's slice of shared memory (rebuilt when the
// warp moves to a request with another key).
template <int CAP>
__global__ void __launch_bounds__(kBsThreads) batch_bitslice_kernel(const __grid_constant__ BatchParams<CAP> p)
{
    __shared__ __align__(16) uint32_t s_mask[kBsThreads / 32][15 * 128];
    __shared__ unsigned long long s_pos;
    __shared__ WarpState s_state[kBsThreads / 32];
    aesdev::let_next_launch_start();
    if (threadIdx.x == 0)
        s_pos = 0;
    if (threadIdx.x < kBsThreads / 32)
        s_state[threadIdx.x] = WarpState{0, 0, 0, 0};
    __syncthreads();
    aesdev::wait_for_previous_launch();
    p.clear_next();
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t *mask = s_mask[threadIdx.x >> 5];
    const uint4 *cur = nullptr;  // schedule whose masks are in `mask`
    BatchReq rq;
    uint64_t k0;
    uint32_t n;
    while (next_run<BsUnitOf<CAP == 0>, CAP == 0>(p, p.requests(), CAP == 0 ? p.whole_line() : &s_pos,
                                               &s_state[threadIdx.x >> 5], rq, k0, n)) {
        const uint64_t v0 = rq.iv_lo & 255u, nb = (rq.len + 15) >> 4;
        const uint64_t first = k0 << 5 > v0 ? (k0 << 5) - v0 : 0;
        const uint64_t end = ((k0 + n) << 5) - v0, last = end < nb ? end : nb;
        if (rq.rk != cur) {
            __syncwarp();  // every lane is done with the previous masks
            aesbs::build_masks(mask, reinterpret_cast<const uint32_t *>(rq.rk), (int)rq.nr, lane, 32);
            __syncwarp();
            cur = rq.rk;
        }
        const uint4 k0w = __ldg(rq.rk);
        const uint32_t rk0[4] = {k0w.x, k0w.y, k0w.z, k0w.w};
        const aesbs::MaskKeys keys{reinterpret_cast<const uint4 *>(mask)};
        switch (rq.nr) {
        case 10: aesbs::xor_range<10>(rq.in, rq.out, rq.len, rq.iv_hi, rq.iv_lo, rk0, first, last, 0, 1, keys); break;
        case 12: aesbs::xor_range<12>(rq.in, rq.out, rq.len, rq.iv_hi, rq.iv_lo, rk0, first, last, 0, 1, keys); break;
        default: aesbs::xor_range<14>(rq.in, rq.out, rq.len, rq.iv_hi, rq.iv_lo, rk0, first, last, 0, 1, keys); break;
        }
    }
}

template <int MAXT, bool RK_REGS, int CAP, bool WHOLE = false>
cudaError_t set_smem()
{
    const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const cudaError_t e = cudaFuncSetAttribute(batch_ttable_kernel<MAXT, RK_REGS, CAP, false, WHOLE>, attr,
                                               (int)aestt::kTableBytes);
    return e ? e
             : cudaFuncSetAttribute(batch_ttable_kernel<MAXT, RK_REGS, CAP, true, WHOLE>, attr,
                                    (int)aestt::kTableBytes);
}

int g_bs_ctas_per_sm = 1;  // resident bitsliced batch CTAs per SM (set with the attributes)

}  // namespace

namespace aesrt {

cudaError_t batch_set_attributes()
{
    cudaError_t e;
    if ((e = set_smem<kRegsMaxThreads, true, 0>()) || (e = set_smem<kRegsMaxThreads, true, kFewInParams>()) ||
        (e = set_smem<kRegsMaxThreads, true, kMostInParams>()) || (e = set_smem<kRegsMaxThreads, true, 0, true>()) ||
        (e = set_smem<1024, false, 0>()) || (e = set_smem<1024, false, 0, true>()) ||
        (e = set_smem<1024, false, kMostInParams>()))
        return e;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_bitslice_kernel<0>, kBsThreads, 0)))
        return e;
    g_bs_ctas_per_sm = per_sm > 0 ? per_sm : 1;
    return cudaSuccess;
}

// More tiles (of BatchShape::counted blocks) than this are AES_ETOOBIG: the
// lengths of one batch stay far below what would overflow its summed cost.
// The built-in shape counts tiles of 2048 blocks (128 TiB in all), whatever
// size it claims them in.
constexpr uint64_t kMostTiles = 0xffffffffull;
constexpr int kBuiltInCounted = 2048;

static uint64_t gcd64(uint64_t a, uint64_t b)
{
    while (b) {
        const uint64_t t = a % b;
        a = b;
        b = t;
    }
    return a;
}

static TileOrder make_order(uint64_t total, uint32_t seed)
{
    TileOrder o{1, 0, 0};
    if (!seed || total < 2 || total > kMostTiles)  // a * t must fit 64 bits
        return o;
    o.tiles = total;
    uint64_t x = seed * 0x9E3779B97F4A7C15ull + 0x632BE59BD9B4E019ull;
    for (int tries = 0; tries < 64; ++tries) {
        x ^= x >> 29;
        x *= 0xBF58476D1CE4E5B9ull;
        x ^= x >> 32;
        const uint64_t a = 1 + x % (total - 1);
        if (gcd64(a, total) == 1 && a != 1) {
            o.a = a;
            break;
        }
    }
    o.b = (x >> 7) % total;
    return o;
}

// From so many units on (chunks; 128 MiB) a launch with its table in device
// memory claims from the whole line.  Plans in a row, by pieces and from the
// whole line, on a free GPU and beside a server that holds 52 of the 152 SMs:
// 96 requests of 1 to 2 MiB (140 MB) 169.2 and 171.1 us, 335 and 267; 256 of
// 1 KiB to 8 MiB 341.4 and 341.6, 679 and 524; 4096 of them 4262 and 4237, 8471
// and 6439; 300 of them in pinned host memory 2126 and 2092, 2069 and 1974.
// Below it the claims show: 46 MB 62.6 and 68.9 on a free GPU (122.7 and 105.8
// beside the server), 16 MB 24.1 and 29.3 (47.2 and 46.3).
constexpr uint64_t kWholeFrom = 1u << 18;

// What a launch needs to know of its requests.
struct BatchSums {
    size_t n = 0;       // requests that hold any bytes
    bool table = false;  // for a launch with its table in device memory
    bool host = false;   // some payload lies in pinned host memory
    uint64_t cost = 0, units = 0;
    uint64_t tiles = 0;  // of BatchShape::counted blocks; stays at kMostTiles + 1 once past it
    int64_t bytes = 0;
    // Appends r: sets its first cost, adds its units.
    void add(BatchReq &r, const BatchShape &s)
    {
        const uint32_t v0 = (uint32_t)(r.iv_lo & 255u);
        const uint64_t chunks = chunks_of(r.len, v0);
        const bool bs = s.variant == AES_VARIANT_BITSLICE;
        if (s.counted)
            tiles = std::min(tiles + tiles_of(r.len, v0, s.counted), kMostTiles + 1);
        const uint64_t u = bs ? (chunks + 31) / 32 : chunks;
        r.cost_begin = cost;
        cost += u * (!bs ? TtUnit::cost(r.nr) : table ? BsUnitOf<true>::cost(r.nr) : BsUnitOf<false>::cost(r.nr));
        units += u;
        bytes += (int64_t)r.len;
        ++n;
    }
};

int validate_batch_shape(BatchShape &s)
{
    if (s.variant == AES_VARIANT_AUTO)
        s.variant = AES_VARIANT_TTABLE;
    if (s.variant == AES_VARIANT_BITSLICE) {
        if (s.threads != kBsThreads)
            return AES_EINVAL;  // one instantiation: 128-thread CTAs
    } else if (s.variant != AES_VARIANT_TTABLE) {
        return AES_EINVAL;
    }
    if (s.nb != 1 && s.nb != 2 && s.nb != 4)
        return AES_EINVAL;
    if (s.threads < 32 || s.threads > 1024 || (s.threads & 31))
        return AES_EINVAL;
    if (s.tile_blocks < 256 || s.tile_blocks % 256 || s.tile_blocks > (1 << 22))
        return AES_EINVAL;
    if (s.ctas < 0)
        return AES_EINVAL;
    return AES_OK;
}

static BatchShape pick_batch_shape(const DeviceState &st, const aes_batch_opts_t *opts)
{
    BatchShape s = st.batch_tuned;
    if (opts) {
        if (opts->variant && opts->variant != s.variant) {
            // another variant than the tuned one: start from its defaults
            s = opts->variant == AES_VARIANT_BITSLICE ? BatchShape{AES_VARIANT_BITSLICE, kBsThreads, 2048, 0, 1}
                                                      : BatchShape{opts->variant, 512, kBuiltInTile, 0, 1};
        }
        if (opts->threads)
            s.threads = opts->threads;
        if (opts->tile_blocks)
            s.tile_blocks = opts->tile_blocks;
        if (opts->ctas)
            s.ctas = opts->ctas;
        if (opts->blocks_per_thread)
            s.nb = opts->blocks_per_thread;
    }
    s.counted = s.tile_blocks == kBuiltInTile && !(opts && opts->tile_blocks) ? kBuiltInCounted : s.tile_blocks;
    return s;
}

// One request (r.len == 0: no work) after its checks, or the status of the one
// that failed.
static int request_of(const aes_desc_t &d, int dev, PayloadChecks &payloads, BatchReq &r, bool *host)
{
    r.len = 0;
    if (!d.ctx || d.ctx->device != dev)
        return AES_EINVAL;
    if (!d.len)
        return AES_OK;
    const void *din = nullptr;
    void *dout = nullptr;
    const int rc = payloads.check(d.in, d.out, d.len, &din, &dout, host);
    if (rc || !blocks_of(d.len))
        return rc;
    r.in = static_cast<const uint4 *>(din);
    r.out = static_cast<uint4 *>(dout);
    r.len = d.len;
    iv_halves(d.iv, &r.iv_hi, &r.iv_lo);
    r.rk = reinterpret_cast<const uint4 *>(d.ctx->d_rk);
    r.nr = (uint32_t)d.ctx->nr;
    r.pad = 0;
    return AES_OK;
}

// The non-empty requests of descs[0..n) into out (room for n), their sums into
// `sum`; the first bad request's status.
static int fill_reqs(const aes_desc_t *descs, int n, int dev, const BatchShape &s, BatchReq *out, BatchSums &sum)
{
    PayloadChecks payloads(dev);
    for (int i = 0; i < n; ++i) {
        BatchReq r;
        bool host = false;
        const int rc = request_of(descs[i], dev, payloads, r, &host);
        if (rc)
            return rc;
        if (!r.len)
            continue;
        sum.host |= host;
        const size_t at = sum.n;
        sum.add(r, s);
        out[at] = r;
    }
    return sum.tiles > kMostTiles ? AES_ETOOBIG : AES_OK;
}

// Chunks of the largest T-table tile for a shape's tile_blocks.  A warp does a
// tile in runs of at most 248 chunks (7936 blocks), so from half a run on a
// tile is whole runs: one of 4096 blocks, the tuner's largest, was half a run
// (4096 requests of 1 KiB to 8 MiB 4054 us, 4029 as a run), one of 8192 a run
// and a short one.
static uint32_t tile_chunks(int tile_blocks)
{
    constexpr uint32_t run = aestile::kRunChunks;
    const uint32_t chunks = (uint32_t)tile_blocks / 32u;
    return chunks <= run / 2 ? chunks : (chunks + run / 2) / run * run;
}

// Everything of a launch but its requests; returns the grid size.
static int set_args(BatchArgs &p, const BatchSums &sum, const DeviceState &st, const BatchShape &s, uint32_t seed)
{
    p.reqs = nullptr;
    p.n = (uint32_t)sum.n;
    p.total_cost = sum.cost;
    const bool bs = s.variant == AES_VARIANT_BITSLICE;
    p.tile_cost = !bs         ? (uint64_t)tile_chunks(s.tile_blocks) * TtUnit::cost(10)
                  : sum.table ? BsUnitOf<true>::cost(10)
                              : (uint64_t)std::max(1, s.tile_blocks / 1024) * BsUnitOf<false>::cost(10);
    p.te0 = st.te0;
    p.order = make_order((sum.cost + p.tile_cost - 1) / p.tile_cost, seed);
    // as many CTAs as are resident at once (one T-table CTA per SM: its
    // tables take 128 KiB of shared memory), each with a unit of work at
    // least.  A T-table CTA gets 8 chunks, one for a warp, as a single call's
    // does (ctr_ctas): plans of 64 requests of 1 to 16 KiB take 5.16 us in a
    // row with 1 chunk, 5.13 with 8, 6.81 with 16, and beside the resident
    // server (4 SMs free) 174, 107 and 70 us; 8 such requests 4.2, 4.6, 5.5
    // and 107, 25, 17 us.
    const int resident = bs ? st.nsm * g_bs_ctas_per_sm : st.nsm;
    const int ctas = s.ctas > 0 ? std::min(s.ctas, resident) : resident;
    const uint64_t per = bs || s.ctas > 0 ? 1 : std::min(8, s.threads / 32);
    return (int)std::min((uint64_t)ctas, (sum.units + per - 1) / per);
}

// The table in device memory and, in one more entry behind it, the counters of
// a kernel that claims from the whole line; both are zero before its first launch.
static size_t table_entries(const BatchSums &sum) { return sum.n + 1; }
static void set_table(BatchParams<0> &p, BatchReq *table, const BatchSums &sum, const BatchShape &s)
{
    p.reqs = table;
    if (s.variant == AES_VARIANT_BITSLICE || sum.units >= kWholeFrom) {
        p.claimed = reinterpret_cast<unsigned long long *>(table + sum.n);
        p.cleared = p.claimed + 1;
    }
}

template <int MAXT, bool RK_REGS, int CAP>
static cudaError_t launch_ttable(const BatchParams<CAP> &p, int ctas, int threads, bool host, cudaStream_t stream)
{
    auto kernel = host ? batch_ttable_kernel<MAXT, RK_REGS, CAP, true, false>
                       : batch_ttable_kernel<MAXT, RK_REGS, CAP, false, false>;
    if constexpr (CAP == 0)
        if (p.claimed)
            kernel = host ? batch_ttable_kernel<MAXT, RK_REGS, CAP, true, true>
                          : batch_ttable_kernel<MAXT, RK_REGS, CAP, false, true>;
    return launch_overlapped(kernel, ctas, threads, aestt::kTableBytes, stream, p);
}

template <int CAP>
static cudaError_t launch_batch(const BatchParams<CAP> &p, int ctas, const BatchShape &s, bool host,
                                cudaStream_t stream)
{
    if constexpr (CAP != kFewInParams) {  // the small size exists for the default shape's kernel only
        if (s.variant == AES_VARIANT_BITSLICE)
            return launch_overlapped(batch_bitslice_kernel<CAP>, ctas, kBsThreads, 0, stream, p);
        if (s.threads > kRegsMaxThreads)
            return launch_ttable<1024, false>(p, ctas, s.threads, host, stream);
    }
    return launch_ttable<kRegsMaxThreads, true>(p, ctas, s.threads, host, stream);
}

// n <= CAP requests in one launch whose parameters hold them.
template <int CAP>
static int launch_in_params(const aes_desc_t *descs, int n, const DeviceState &st, const BatchShape &s, uint32_t seed,
                            cudaStream_t stream)
{
    BatchParams<CAP> p;
    BatchSums sum;
    const int rc = fill_reqs(descs, n, st.device, s, p.in_params, sum);
    if (rc || !sum.n)
        return rc;
    const int ctas = set_args(p, sum, st, s, seed);
    const cudaError_t e = launch_batch(p, ctas, s, sum.host, stream);
    return e ? cuda_fail(e, "aes_ctr_batch launch") : AES_OK;
}

int batch_by_params(const aes_desc_t *descs, int n, const DeviceState &st, const BatchShape &s, uint32_t seed,
                    cudaStream_t stream)
{
    if (n <= kFewInParams && s.variant == AES_VARIANT_TTABLE && s.threads <= kRegsMaxThreads)
        return launch_in_params<kFewInParams>(descs, n, st, s, seed, stream);
    if (n <= kMostInParams)
        return launch_in_params<kMostInParams>(descs, n, st, s, seed, stream);
    // Nothing runs unless every request is good: one pass checks and counts
    // them, a second fills the launches (no-alloc callers may have no heap to
    // hold them in between).  Addresses are looked up again only if some
    // payload's differs from the one the caller knows it by.
    BatchSums sum;
    bool as_given = true;
    PayloadChecks payloads(st.device);
    for (int i = 0; i < n; ++i) {
        BatchReq r;
        bool host = false;
        const int rc = request_of(descs[i], st.device, payloads, r, &host);
        if (rc)
            return rc;
        if (!r.len)
            continue;
        sum.host |= host;
        sum.add(r, s);
        as_given &= r.in == descs[i].in && r.out == descs[i].out;
    }
    if (sum.tiles > kMostTiles)
        return AES_ETOOBIG;
    // equal numbers of requests per launch
    const size_t launches = (sum.n + kMostInParams - 1) / kMostInParams;
    payloads.accept_all = as_given;
    BatchParams<kMostInParams> p;
    int i = 0;
    for (size_t k = 0; k < launches; ++k) {
        const size_t want = sum.n * (k + 1) / launches - sum.n * k / launches;
        BatchSums part;
        while (part.n < want) {
            BatchReq r;
            bool host = false;
            const int rc = request_of(descs[i++], st.device, payloads, r, &host);
            if (rc)
                return rc;
            if (!r.len)
                continue;
            const size_t at = part.n;
            part.add(r, s);
            p.in_params[at] = r;
        }
        const int ctas = set_args(p, part, st, s, seed);
        const cudaError_t e = launch_batch(p, ctas, s, sum.host, stream);
        if (e)
            return cuda_fail(e, "aes_ctr_batch launch");
    }
    return AES_OK;
}

}  // namespace aesrt

using namespace aesrt;

namespace {

// The calling thread's current device, put back when the scope ends.
class OnDevice {
public:
    OnDevice() { error = cudaGetDevice(&before_); }
    ~OnDevice() { set(before_); }
    int before() const { return before_; }
    cudaError_t set(int device)
    {
        int now = -1;
        const cudaError_t e = cudaGetDevice(&now);
        return e || now == device ? e : cudaSetDevice(device);
    }
    cudaError_t error;

private:
    int before_ = 0;
};

}  // namespace

// A prepared batch.  It runs on the device it was created on, whichever is
// current, in any device's stream, and its launches run one after the other on
// whatever streams they are made (two launches at once of a plan that encrypts
// in place would race): a launch waits for the event that the last one left,
// unless both are on one stream.  Recording the event costs 0.4 us of host
// time and leaves launches in a row overlapped (64 requests of 1 to 16 KiB
// 5.1 us a launch with it and without; as a CUDA graph, which has the same
// guarantees, 8.2 us).
struct aes_batch_plan_s {
    int device = 0;
    BatchSums sum;
    BatchShape shape{};
    BatchParams<0> params{};
    int ctas = 0;
    BatchReq *reqs = nullptr;  // device
    std::mutex mu;
    cudaEvent_t done = nullptr;     // the last launch
    bool launched = false;
    unsigned long long last_id = 0;  // cudaStreamGetId of its stream
    cudaStream_t own = nullptr;      // for launches into another device's stream

    ~aes_batch_plan_s()
    {
        OnDevice on;
        on.set(device);
        cudaFree(reqs);
        if (done)
            cudaEventDestroy(done);
        if (own)
            cudaStreamDestroy(own);
    }

    // One launch on a stream of the plan's device, which is current.
    cudaError_t launch_on(cudaStream_t stream)
    {
        unsigned long long id = 0;
        cudaError_t e = cudaStreamGetId(stream, &id);
        if (!e && launched && id != last_id)
            e = cudaStreamWaitEvent(stream, done, 0);
        if (e || (e = launch_batch(params, ctas, shape, sum.host, stream)))
            return e;
        launched = true;
        last_id = id;
        std::swap(params.claimed, params.cleared);
        return cudaEventRecord(done, stream);
    }

    // One launch into a stream of `stream_device`: on the plan's own stream,
    // between what that stream holds and what follows there.
    cudaError_t launch_from(int stream_device, cudaStream_t stream, OnDevice &on)
    {
        cudaEvent_t before = nullptr;
        cudaError_t e = on.set(stream_device);
        if (!e)
            e = cudaEventCreateWithFlags(&before, cudaEventDisableTiming);
        if (!e)
            e = cudaEventRecord(before, stream);
        if (!e)
            e = on.set(device);
        if (!e && !own)
            e = cudaStreamCreateWithFlags(&own, cudaStreamNonBlocking);
        if (!e)
            e = cudaStreamWaitEvent(own, before, 0);
        if (!e)
            e = launch_on(own);
        if (!e)
            e = on.set(stream_device);
        if (!e)
            e = cudaStreamWaitEvent(stream, done, 0);
        if (before)
            cudaEventDestroy(before);
        return e;
    }
};

extern "C" {

int aes_ctr_batch_ex(const aes_desc_t *descs, int n, void *stream, const aes_batch_opts_t *opts)
{
    if (n < 0 || (n > 0 && !descs))
        return AES_EINVAL;
    if (n > AES_BATCH_MAX)
        return AES_ETOOBIG;
    if (n == 0)
        return AES_OK;
    DeviceState *st = nullptr;
    int rc = device_state(&st);
    if (rc)
        return rc;
    BatchShape s = pick_batch_shape(*st, opts);
    if ((rc = validate_batch_shape(s)))
        return rc;
    const uint32_t seed = opts ? opts->tile_order_seed : 0;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    // Up to two or three launches with the requests in their parameters cost
    // what one launch with a table in device memory does (1000 requests of 1
    // to 16 KiB: 175.5 and 176.9 us a call in a row of calls; 512 of 1 KiB to
    // 8 MiB: 539 and 537), and a call on an idle GPU is sooner done without
    // the allocation and the copy (209 and 359 us, 639 and 800).  A capture
    // must not record the copy: its host source is gone when the graph runs.
    if (n <= kMostByParams || capturing(cs))
        return batch_by_params(descs, n, *st, s, seed, cs);
    std::vector<BatchReq> host;
    try {
        host.resize((size_t)n + 1);
    } catch (const std::bad_alloc &) {
        return AES_ENOMEM;
    }
    BatchSums sum;
    sum.table = true;
    if ((rc = fill_reqs(descs, n, st->device, s, host.data(), sum)) || !sum.n)
        return rc;
    BatchParams<0> p{};
    const int ctas = set_args(p, sum, *st, s, seed);
    BatchReq *reqs = nullptr;
    const size_t bytes = table_entries(sum) * sizeof(BatchReq);
    cudaError_t e = cudaMallocFromPoolAsync(reinterpret_cast<void **>(&reqs), bytes, st->pool, cs);
    if (e)
        return e == cudaErrorMemoryAllocation ? AES_ENOMEM : cuda_fail(e, "cudaMallocFromPoolAsync");
    set_table(p, reqs, sum, s);
    // Pageable source: the copy has finished reading the host vector when
    // cudaMemcpyAsync returns, so it may be destroyed afterwards.
    e = cudaMemcpyAsync(reqs, host.data(), bytes, cudaMemcpyHostToDevice, cs);
    if (!e)
        e = launch_batch(p, ctas, s, sum.host, cs);
    cudaError_t e2 = cudaFreeAsync(reqs, cs);
    if (e)
        return cuda_fail(e, "aes_ctr_batch");
    if (e2)
        return cuda_fail(e2, "cudaFreeAsync");
    return AES_OK;
}

int aes_ctr_batch(const aes_desc_t *descs, int n, void *stream)
{
    return aes_ctr_batch_ex(descs, n, stream, nullptr);
}

int aes_batch_plan_create(aes_batch_plan_t *out, const aes_desc_t *descs, int n,
                          const aes_batch_opts_t *opts)
{
    if (!out)
        return AES_EINVAL;
    *out = nullptr;
    if (n < 1 || !descs)
        return AES_EINVAL;
    if (n > AES_BATCH_MAX)
        return AES_ETOOBIG;
    DeviceState *st = nullptr;
    int rc = device_state(&st);
    if (rc)
        return rc;
    BatchShape s = pick_batch_shape(*st, opts);
    if ((rc = validate_batch_shape(s)))
        return rc;
    aes_batch_plan_s *plan = new (std::nothrow) aes_batch_plan_s();
    if (!plan)
        return AES_ENOMEM;
    plan->device = st->device;
    plan->shape = s;
    plan->sum.table = true;
    std::vector<BatchReq> host;
    try {
        host.resize((size_t)n + 1);
    } catch (const std::bad_alloc &) {
        delete plan;
        return AES_ENOMEM;
    }
    if ((rc = fill_reqs(descs, n, st->device, s, host.data(), plan->sum))) {
        delete plan;
        return rc;
    }
    if (plan->sum.n) {
        const size_t bytes = table_entries(plan->sum) * sizeof(BatchReq);
        cudaError_t e = cudaMalloc(reinterpret_cast<void **>(&plan->reqs), bytes);
        if (e) {
            delete plan;
            return e == cudaErrorMemoryAllocation ? AES_ENOMEM : cuda_fail(e, "cudaMalloc(plan)");
        }
        e = cudaMemcpyAsync(plan->reqs, host.data(), bytes, cudaMemcpyHostToDevice, st->setup);
        if (!e)
            e = cudaStreamSynchronize(st->setup);
        if (!e)
            e = cudaEventCreateWithFlags(&plan->done, cudaEventDisableTiming);
        if (e) {
            delete plan;
            return cuda_fail(e, "aes_batch_plan_create");
        }
        plan->ctas = set_args(plan->params, plan->sum, *st, s, opts ? opts->tile_order_seed : 0);
        set_table(plan->params, plan->reqs, plan->sum, s);
    }
    *out = plan;
    return AES_OK;
}

int aes_batch_plan_launch(aes_batch_plan_t plan, void *stream)
{
    if (!plan)
        return AES_EINVAL;
    if (!plan->sum.n)
        return AES_OK;  // nothing to encrypt (all lengths zero)
    if (capturing(static_cast<cudaStream_t>(stream)))
        return cuda_fail(cudaErrorStreamCaptureUnsupported, "aes_batch_plan_launch");
    const cudaStream_t cs = static_cast<cudaStream_t>(stream);
    OnDevice on;
    cudaError_t e = on.error;
    int stream_device = on.before();
    if (!e && cs && cs != cudaStreamLegacy && cs != cudaStreamPerThread)
        e = cudaStreamGetDevice(cs, &stream_device);
    if (!e) {
        std::lock_guard<std::mutex> lock(plan->mu);
        if (stream_device != plan->device)
            e = plan->launch_from(stream_device, cs, on);
        else if (!(e = on.set(plan->device)))
            e = plan->launch_on(cs);
    }
    return e ? cuda_fail(e, "aes_batch_plan_launch") : AES_OK;
}

int64_t aes_batch_plan_bytes(aes_batch_plan_t plan) { return plan ? plan->sum.bytes : AES_EINVAL; }

int aes_batch_plan_destroy(aes_batch_plan_t plan)
{
    delete plan;
    return AES_OK;
}

}  // extern "C"
