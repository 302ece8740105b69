// internal.h -- host-side interfaces between the library's translation units.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>
#include <type_traits>

namespace aesrt {

constexpr int kMaxRoundKeyWords = 60;  // 4 * (14 + 1)

// Parameters of one single-key CTR launch.  Passed by value (kernel
// parameter space), so the round keys are constant-bank operands.
struct CtrParams {
    const uint4 *in;
    uint4 *out;
    uint64_t len;           // payload bytes
    uint64_t iv_hi, iv_lo;  // initial counter block as big-endian halves
    const uint32_t *te0;    // 256-word T-table seed (device)
    uint32_t rk[kMaxRoundKeyWords];  // round keys, little-endian column words
};

struct CtrShape {
    int variant;  // 1 = T-table, 2 = bitsliced
    int threads;
    int nb;       // T-table: accepted as 1, 2 or 4; the kernel keeps one block per lane in flight
    int ctas;     // 0 = derive
};

// 16-byte blocks of `len` bytes.  A length within 15 bytes of 2^64 (a negative
// one made unsigned) wraps to none: the entry points do nothing with it, and
// no count of chunks may be derived from it.
inline uint64_t blocks_of(uint64_t len) { return (len + 15) / 16; }

// Device tables and key expansion (tables.cu).
cudaError_t launch_te0_init(uint32_t *te0, cudaStream_t stream);
cudaError_t launch_key_expand(const uint8_t *keys, const int32_t *bits, const uint32_t *te0,
                              uint32_t *w, int n, cudaStream_t stream);

// Whether the stream is being captured into a graph.
inline bool capturing(cudaStream_t stream)
{
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    return cudaStreamIsCapturing(stream, &cap) == cudaSuccess && cap != cudaStreamCaptureStatusNone;
}

// Launch a kernel that calls let_next_launch_start and
// wait_for_previous_launch: its CTAs may be set up (table fill, constants)
// while the stream's previous kernel drains, instead of after it has ended
// and been flushed.  A 4 KiB message costs 3.2 us per launch in a row of
// plain launches inside a CUDA graph and 6.2 us on a stream; overlapped
// launches 1.7 us on a stream, 1 MiB 6.9 -> 3.5 us.  While the stream is
// being captured the launch is a plain one, so captured graphs hold ordinary
// full dependencies.
template <class P>
inline cudaError_t launch_overlapped(void (*kernel)(P), int ctas, int threads, size_t smem, cudaStream_t stream,
                                     const std::remove_const_t<P> &params)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    if (!capturing(stream)) {
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
    }
    void *args[1] = {const_cast<void *>(static_cast<const void *>(&params))};  // copied by the launch
    const cudaError_t e = cudaLaunchKernelExC(&cfg, reinterpret_cast<const void *>(kernel), args);
    if (e)
        cudaGetLastError();  // the caller reports it; leave no stale error behind
    return e;
}

// Single-buffer CTR (ctr.cu).
cudaError_t ctr_set_attributes();  // once per device
int ctr_max_ctas(const CtrShape &s, int nsm);
// Grid size of one launch of `nblocks` blocks whose initial counter has low
// byte v0.
int ctr_ctas(uint64_t nblocks, uint32_t v0, const CtrShape &s, int nsm);
cudaError_t launch_ctr(const CtrParams &p, int nr, const CtrShape &s, int nsm, cudaStream_t stream);

// Batched varlen CTR (batch.cu).
struct BatchReq {        // one request, device-side descriptor (64 bytes)
    const uint4 *in;
    uint4 *out;
    uint64_t len;
    uint64_t iv_hi, iv_lo;
    const uint4 *rk;     // device round keys (4*(Nr+1) words as uint4 per round)
    uint32_t nr;
    uint32_t pad;
    uint64_t cost_begin; // batch: summed cost of the requests before this one
};
static_assert(sizeof(BatchReq) == 64, "descriptor is one 64-byte line");

constexpr int kBuiltInTile = 7936;  // tile_blocks of the shape used until a tuner picks another

struct BatchShape {
    int variant;      // AES_VARIANT_TTABLE or AES_VARIANT_BITSLICE
    int threads;
    int tile_blocks;  // a multiple of 256: the largest tile a warp claims
    int ctas;
    int nb;           // T-table: accepted as 1, 2 or 4; the kernel keeps one block per lane in flight
    int counted;      // the batch may hold 2^32 - 1 tiles of so many blocks (0: no limit)
};

// Tiles of `tile_blocks` blocks (whole 256-block counter groups) that `len`
// bytes make when the initial counter has low byte `iv_low_byte`.
inline uint64_t tiles_of(uint64_t len, uint32_t iv_low_byte, int tile_blocks)
{
    const uint64_t nb = blocks_of(len);
    if (!nb)
        return 0;
    const uint64_t groups = ((iv_low_byte + nb - 1) >> 8) + 1, per = (uint64_t)tile_blocks / 256u;
    return (groups + per - 1) / per;
}

// 32-block chunks of the counter space that `len` bytes (of at least one
// block) touch when the initial counter has low byte `iv_low_byte`.
inline uint64_t chunks_of(uint64_t len, uint32_t iv_low_byte)
{
    const uint64_t nb = blocks_of(len);
    return ((iv_low_byte + nb - 1) >> 5) - (iv_low_byte >> 5) + 1;
}

cudaError_t batch_set_attributes();

}  // namespace aesrt
