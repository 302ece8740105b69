// batch.cu -- many independent AES-CTR requests in one launch.
//
// Work is measured in shared-memory wavefronts, the unit of the kernel's
// bound: a 32-block chunk (tile.cuh) of a request with Nr rounds costs
// chunk_cost(Nr) of them.  The requests' chunks, one request after the other,
// are one line of cost; CTA c of G (one per SM) owns the c-th of G equal
// pieces of it, so every SM gets the same number of lookups whatever the mix
// of lengths and key sizes, and neither a table of tiles nor a counter in
// device memory is needed.  In a CTA's piece the warps claim tiles through
// one counter in shared memory, each tile a warps-th of what is left, at
// most tile_blocks and at least about one chunk: large tiles amortise a
// request's set-up, small ones at the end let the warps finish together, and
// a batch of a few short requests is spread one chunk to a warp.  A warp
// finds its tile's request by a 32-way search over the requests' first costs.
// The cipher is the same T-table round code as the single-buffer kernel.
// Round keys: CTAs of up to 512 threads (the default) hold the current
// request's schedule in registers, so the shared-memory pipe, the kernel's
// bound, serves lookups only; larger CTAs stage it in each warp's slice of
// shared memory (one broadcast wavefront per round).
//
// The bitsliced kernel takes the same pieces and tiles, 1024 blocks at a time,
// as the autotuner's alternative to the T-tables.
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
#include <new>
#include <type_traits>
#include <vector>

namespace {

using aesrt::BatchReq;

struct TileOrder {
    uint64_t a, b;   // t -> (a*t + b) mod tiles
    uint64_t tiles;  // 0: no order, tiles are cut as they are claimed
};

// Shared-memory wavefronts of one 32-block chunk: 16 lookups in each of the
// NR - 2 rounds that are not cached, and about 9 for the payload and the
// group constants.
__host__ __device__ constexpr uint32_t chunk_cost(uint32_t nr) { return 16u * (nr - 2u) + 9u; }
// The smallest tile: one AES-128 chunk.
constexpr uint64_t kMinTileCost = chunk_cost(10);

__device__ __forceinline__ uint64_t ceil_chunks(uint64_t cost, uint32_t nr)
{
    switch (nr) {
    case 10: return (cost + chunk_cost(10) - 1) / chunk_cost(10);
    case 12: return (cost + chunk_cost(12) - 1) / chunk_cost(12);
    default: return (cost + chunk_cost(14) - 1) / chunk_cost(14);
    }
}

// One launch.  reqs (device memory, no empty requests) is read only after
// wait_for_previous_launch.
struct BatchArgs {
    const BatchReq *reqs;
    uint32_t n;
    uint64_t total_cost;
    uint64_t tile_cost;  // largest tile
    const uint32_t *te0;
    TileOrder order;
};

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

// Calls run(request, first chunk, chunks <= kRunChunks) for every piece of
// work of the calling warp (every lane with the same arguments).  s_pos: the CTA's
// counter, zeroed before the CTA's last barrier.
template <class RUN>
__device__ __forceinline__ void for_each_run(const BatchArgs &p, unsigned long long *s_pos, RUN &&run)
{
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t units = p.order.tiles ? p.order.tiles : p.total_cost;  // this CTA's piece [u0, u1)
    const uint64_t q = units / gridDim.x, r = units % gridDim.x;
    const uint64_t u0 = q * blockIdx.x + (blockIdx.x < r ? blockIdx.x : r);
    const uint64_t size = q + (blockIdx.x < r ? 1 : 0);
    const uint64_t guide = blockDim.x >> 5;
    uint32_t ri = 0;
    bool near = false;
    for (;;) {
        unsigned long long at = 0, take = 1;
        if (lane == 0) {
            if (!p.order.tiles) {
                const unsigned long long cur = *(volatile unsigned long long *)s_pos;
                take = cur < size ? (size - cur) / guide : 0;
                take = take < kMinTileCost ? kMinTileCost : take > p.tile_cost ? p.tile_cost : take;
            }
            at = atomicAdd(s_pos, take);
        }
        at = __shfl_sync(0xffffffffu, at, 0);
        take = __shfl_sync(0xffffffffu, take, 0);
        if (at >= size)
            break;
        uint64_t xa, xb;  // the tile's cost range
        if (p.order.tiles) {
            const uint64_t t = (p.order.a * (u0 + at) + p.order.b) % p.order.tiles;
            xa = t * p.tile_cost;
            xb = xa + p.tile_cost < p.total_cost ? xa + p.tile_cost : p.total_cost;
            ri = 0;
        } else {
            xa = u0 + at;
            xb = u0 + (at + take < size ? at + take : size);
        }
        ri = owner_of(p.reqs, ri, p.n, xa, near);
        near = !p.order.tiles;  // later tiles lie further along
        for (uint32_t i = ri; i < p.n; ++i) {
            const BatchReq rq = p.reqs[i];
            if (rq.cost_begin >= xb)
                break;
            // chunk c belongs to the tile that holds its first cost unit
            const uint64_t nb = (rq.len + 15) >> 4, v0 = rq.iv_lo & 255u, first = aestile::first_chunk(rq.iv_lo);
            const uint64_t nch = ((v0 + nb - 1) >> 5) - first + 1;
            const uint64_t ca = xa > rq.cost_begin ? ceil_chunks(xa - rq.cost_begin, rq.nr) : 0;
            uint64_t cb = ceil_chunks(xb - rq.cost_begin, rq.nr);
            cb = cb < nch ? cb : nch;
            for (uint64_t c = ca; c < cb;) {
                const uint32_t m = aestile::run_chunks(rq.iv_lo, first + c, cb - c);
                run(rq, first + c, m);
                c += m;
            }
        }
    }
}

// The T-table batch kernel, bound by shared-memory wavefronts (95 % of the
// pipe busy on a 256 MiB AES-128 request, 146 wavefronts a chunk of which 128
// are lookups of rounds 3..10).  Measured as plans: 4096 requests of 1 KiB to
// 8 MiB (3.66 GB) 4390 -> 4153 us, 64 requests of 1 to 16 KiB 39 -> 6.4 us
// (one warp used to take up to 8 groups of a short request in turn), against
// the kernel with a tile map, a device counter and two blocks per lane.
// Registers: 384-thread CTAs with 168 a thread are faster on AES-256 alone
// (4870 against 4957 us for the same lengths) and slower on AES-128 (3459
// against 3356), as are 448 (5258 and 3401).  MAXT: largest CTA it is launched with; RK_REGS:
// round keys in registers (else in the warp's slice of shared memory).
template <int MAXT, bool RK_REGS>
__global__ void __launch_bounds__(MAXT, 1) batch_ttable_kernel(const __grid_constant__ BatchArgs p)
{
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ uint4 s_group[MAXT / 32][aestile::kRunGroups];
    __shared__ uint4 s_rk[RK_REGS ? 1 : MAXT / 32][15];  // round keys of each warp's current request
    __shared__ unsigned long long s_pos;
    aesdev::let_next_launch_start();
    if (threadIdx.x == 0)
        s_pos = 0;
    aestt::fill_tables(smem, p.te0);
    __syncthreads();
    aesdev::wait_for_previous_launch();
    const aestt::Lanes ln(smem);
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    uint4 *w_group = s_group[warp];
    uint4 *w_rk = s_rk[RK_REGS ? 0 : warp];
    auto xor_with = [&](const BatchReq &rq, uint64_t k0, uint32_t n, auto nr) {
        constexpr int NR = decltype(nr)::value;
        if constexpr (RK_REGS) {
            const aestt::RkRegs<NR> rk(rq.rk);
            aestile::xor_run<NR>(rq.in, rq.out, rq.len, rq.iv_hi, rq.iv_lo, k0, n, w_group, ln, rk);
        } else {
            __syncwarp();  // every lane is done with the previous keys
            if (lane <= NR)
                w_rk[lane] = rq.rk[lane];
            __syncwarp();
            const aestt::RkShared rk{w_rk};
            aestile::xor_run<NR>(rq.in, rq.out, rq.len, rq.iv_hi, rq.iv_lo, k0, n, w_group, ln, rk);
        }
    };
    for_each_run(p, &s_pos, [&](const BatchReq &rq, uint64_t k0, uint32_t n) {
        switch (rq.nr) {
        case 10: xor_with(rq, k0, n, std::integral_constant<int, 10>()); break;
        case 12: xor_with(rq, k0, n, std::integral_constant<int, 12>()); break;
        default: xor_with(rq, k0, n, std::integral_constant<int, 14>()); break;
        }
    });
}

// The bitsliced batch kernel: the same tiles and claims, each run encrypted
// by one warp 1024 blocks at a time (bs_tile.cuh) with the request's
// round-key bit planes in the warp's slice of shared memory (rebuilt when the
// warp moves to a request with another key).
__global__ void __launch_bounds__(kBsThreads) batch_bitslice_kernel(const __grid_constant__ BatchArgs p)
{
    __shared__ __align__(16) uint32_t s_mask[kBsThreads / 32][15 * 128];
    __shared__ unsigned long long s_pos;
    aesdev::let_next_launch_start();
    if (threadIdx.x == 0)
        s_pos = 0;
    __syncthreads();
    aesdev::wait_for_previous_launch();
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t *mask = s_mask[threadIdx.x >> 5];
    const uint4 *cur = nullptr;  // schedule whose masks are in `mask`
    for_each_run(p, &s_pos, [&](const BatchReq &rq, uint64_t k0, uint32_t n) {
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
    });
}

int g_bs_ctas_per_sm = 1;  // resident bitsliced batch CTAs per SM (set with the attributes)

}  // namespace

namespace aesrt {

cudaError_t batch_set_attributes()
{
    cudaError_t e;
    const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if ((e = cudaFuncSetAttribute(batch_ttable_kernel<kRegsMaxThreads, true>, attr, (int)aestt::kTableBytes)) ||
        (e = cudaFuncSetAttribute(batch_ttable_kernel<1024, false>, attr, (int)aestt::kTableBytes)))
        return e;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_bitslice_kernel, kBsThreads, 0)))
        return e;
    g_bs_ctas_per_sm = per_sm > 0 ? per_sm : 1;
    return cudaSuccess;
}

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
    if (!seed || total < 2)
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

// Host-side preparation shared by aes_ctr_batch and the plans: the requests
// that hold any bytes.
struct BatchTables {
    std::vector<BatchReq> reqs;
    uint64_t total_cost = 0;
    uint64_t total_chunks = 0;
    int64_t bytes = 0;
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
                                                      : BatchShape{opts->variant, 512, 2048, 0, 1};
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
    return s;
}

static int build_tables(const aes_desc_t *descs, int n, int dev, BatchTables &bt)
{
    bt.reqs.reserve((size_t)n);
    for (int i = 0; i < n; ++i) {
        const aes_desc_t &d = descs[i];
        if (!d.ctx)
            return AES_EINVAL;
        if (d.ctx->device != dev)
            return AES_EINVAL;
        if (!d.len)
            continue;
        const void *din = nullptr;
        void *dout = nullptr;
        const int rc = check_payload(d.in, d.out, d.len, dev, &din, &dout);
        if (rc)
            return rc;
        BatchReq r{};
        r.in = static_cast<const uint4 *>(din);
        r.out = static_cast<uint4 *>(dout);
        r.len = d.len;
        iv_halves(d.iv, &r.iv_hi, &r.iv_lo);
        r.rk = reinterpret_cast<const uint4 *>(d.ctx->d_rk);
        r.nr = (uint32_t)d.ctx->nr;
        r.cost_begin = bt.total_cost;
        const uint64_t chunks = chunks_of(d.len, d.iv[15]);
        bt.total_chunks += chunks;
        bt.total_cost += chunks * chunk_cost(r.nr);
        bt.bytes += (int64_t)d.len;
        bt.reqs.push_back(r);
    }
    return AES_OK;
}

uint32_t batch_chunk_cost(int nr) { return chunk_cost((uint32_t)nr); }

cudaError_t launch_batch(const BatchReq *reqs, size_t n, uint64_t total_cost, uint64_t total_chunks,
                                const uint32_t *te0, const BatchShape &s, int nsm, uint32_t seed, cudaStream_t stream)
{
    BatchArgs p{};
    p.reqs = reqs;
    p.n = (uint32_t)n;
    p.total_cost = total_cost;
    p.tile_cost = (uint64_t)(s.tile_blocks / 32) * chunk_cost(10);
    p.te0 = te0;
    p.order = make_order((total_cost + p.tile_cost - 1) / p.tile_cost, seed);
    // as many CTAs as are resident at once (one T-table CTA per SM: its
    // tables take 128 KiB of shared memory), none without a chunk
    const int resident = s.variant == AES_VARIANT_BITSLICE ? nsm * g_bs_ctas_per_sm : nsm;
    int ctas = s.ctas > 0 ? std::min(s.ctas, resident) : resident;
    if ((uint64_t)ctas > total_chunks)
        ctas = (int)total_chunks;
    if (s.variant == AES_VARIANT_BITSLICE)
        return launch_overlapped(batch_bitslice_kernel, ctas, kBsThreads, 0, stream, p);
    return s.threads <= kRegsMaxThreads
               ? launch_overlapped(batch_ttable_kernel<kRegsMaxThreads, true>, ctas, s.threads, aestt::kTableBytes,
                                   stream, p)
               : launch_overlapped(batch_ttable_kernel<1024, false>, ctas, s.threads, aestt::kTableBytes, stream, p);
}

}  // namespace aesrt

using namespace aesrt;

struct aes_batch_plan_s {
    int device;
    BatchTables bt;
    BatchShape shape;
    uint32_t seed = 0;
    BatchReq *reqs = nullptr;  // device
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
    BatchTables bt;
    if ((rc = build_tables(descs, n, st->device, bt)))
        return rc;
    if (bt.reqs.empty())
        return AES_OK;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    BatchReq *reqs = nullptr;
    const size_t bytes = bt.reqs.size() * sizeof(BatchReq);
    cudaError_t e = cudaMallocAsync(reinterpret_cast<void **>(&reqs), bytes, cs);
    if (e)
        return e == cudaErrorMemoryAllocation ? AES_ENOMEM : cuda_fail(e, "cudaMallocAsync");
    // Pageable source: the copy has finished reading the host vector when
    // cudaMemcpyAsync returns, so bt may be destroyed afterwards.
    e = cudaMemcpyAsync(reqs, bt.reqs.data(), bytes, cudaMemcpyHostToDevice, cs);
    if (!e)
        e = launch_batch(reqs, bt.reqs.size(), bt.total_cost, bt.total_chunks, st->te0, s, st->nsm,
                         opts ? opts->tile_order_seed : 0, cs);
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
    plan->seed = opts ? opts->tile_order_seed : 0;
    if ((rc = build_tables(descs, n, st->device, plan->bt))) {
        delete plan;
        return rc;
    }
    const size_t bytes = plan->bt.reqs.size() * sizeof(BatchReq);
    if (bytes) {
        cudaError_t e = cudaMalloc(reinterpret_cast<void **>(&plan->reqs), bytes);
        if (e) {
            delete plan;
            return e == cudaErrorMemoryAllocation ? AES_ENOMEM : cuda_fail(e, "cudaMalloc(plan)");
        }
        e = cudaMemcpyAsync(plan->reqs, plan->bt.reqs.data(), bytes, cudaMemcpyHostToDevice, st->setup);
        if (!e)
            e = cudaStreamSynchronize(st->setup);
        if (e) {
            cudaFree(plan->reqs);
            delete plan;
            return cuda_fail(e, "aes_batch_plan_create");
        }
    }
    *out = plan;
    return AES_OK;
}

int aes_batch_plan_launch(aes_batch_plan_t plan, void *stream)
{
    if (!plan)
        return AES_EINVAL;
    if (plan->bt.reqs.empty())
        return AES_OK;  // nothing to encrypt (all lengths zero)
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(static_cast<cudaStream_t>(stream), &cap) == cudaSuccess &&
        cap != cudaStreamCaptureStatusNone)
        return cuda_fail(cudaErrorStreamCaptureUnsupported, "aes_batch_plan_launch");
    DeviceState *st = nullptr;
    int rc = device_state(&st);
    if (rc)
        return rc;
    if (st->device != plan->device)
        return AES_EINVAL;
    const cudaError_t e =
        launch_batch(plan->reqs, plan->bt.reqs.size(), plan->bt.total_cost, plan->bt.total_chunks, st->te0,
                     plan->shape, st->nsm, plan->seed, static_cast<cudaStream_t>(stream));
    return e ? cuda_fail(e, "aes_batch_plan_launch") : AES_OK;
}

int64_t aes_batch_plan_bytes(aes_batch_plan_t plan) { return plan ? plan->bt.bytes : AES_EINVAL; }

int aes_batch_plan_destroy(aes_batch_plan_t plan)
{
    if (!plan)
        return AES_OK;
    cudaFree(plan->reqs);
    delete plan;
    return AES_OK;
}

}  // extern "C"
