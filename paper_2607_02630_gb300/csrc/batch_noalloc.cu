// batch_noalloc.cu -- aes_ctr_batch_noalloc: the batched launch for callers
// that cannot allocate device memory.
//
// aes_ctr_batch allocates a descriptor table in device memory for batches of
// more requests than a kernel's parameters hold.  Some callers cannot have
// that: a process whose whole HBM budget is already reserved by another
// framework's memory pool, a latency-critical path that must not pay for
// cudaMalloc/cudaFree (both can synchronise the device), or an embedded
// runtime that forbids dynamic allocation once it has started.  This entry
// point passes every request in kernel parameters instead, in as many
// launches as that takes (500 requests each), so it needs no memory, the
// host's heap included, but 32 KB of stack, and its calls share no state.  The caller still owns the payload buffers
// and the key contexts (which must exist already: creating them is the only
// step that allocates).
#include "../../include/aesoffload.h"
#include "internal.h"
#include "runtime.h"

using namespace aesrt;

extern "C" int aes_ctr_batch_noalloc(const aes_desc_t *descs, int n, void *stream)
{
    if (n < 0 || (n > 0 && !descs))
        return AES_EINVAL;
    if (n > AES_NOALLOC_MAX_REQUESTS)
        return AES_ETOOBIG;
    if (n == 0)
        return AES_OK;
    DeviceState *st = nullptr;
    const int rc = device_state_ready(&st);  // never initialises, so never allocates
    if (rc)
        return rc;
    // the tuned T-table shape
    BatchShape s = st->batch_tuned;
    if (s.variant != AES_VARIANT_TTABLE)
        s = BatchShape{AES_VARIANT_TTABLE, 512, kBuiltInTile, 0, 1};
    return batch_by_params(descs, n, *st, s, 0, static_cast<cudaStream_t>(stream));
}
