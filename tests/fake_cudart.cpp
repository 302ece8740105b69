// A CUDA runtime that runs nothing and writes down what it is asked to do:
// linked with the library's own objects, it shows on the CPU which launches an
// entry point makes, on which device and stream and with which grid.  Two
// devices; device memory is host memory; streams and events keep which launches
// run behind which.  Not modelled: capture, time beyond given costs, and what
// kernels compute.
#include <cuda_runtime_api.h>

#include <atomic>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <new>
#include <set>
#include <string>
#include <utility>
#include <vector>

namespace {

struct Launch {
    int device;        // the device the kernel runs on
    int grid, block;
    int programmatic;  // 1: may start before the stream's previous kernel has ended
    uint64_t stream;
    char args[80];     // the first bytes of the first parameter
    char name[128];
};

struct Stream {
    int device;
    std::set<int> before;  // launches that its next operation runs behind
};
struct Event {
    int device;
    std::set<int> before;
    size_t at = 0;  // launches made before it
};

int g_device = 0, g_sms = 152;
size_t g_segment = 1ull << 40;    // size of an allocation that payloads lie in
std::map<int, std::pair<float, float>> g_costs;  // by CTA size: us of a launch after an event, of one in a row
long g_queries = 0, g_lookups = 0;  // pointers asked about, allocations looked up
std::atomic<long> g_news{0};
std::vector<Launch> g_log;
std::vector<std::set<int>> g_before;  // of each launch: those it runs behind
std::set<Stream *> g_streams;
std::map<const void *, std::string> g_names;
std::set<std::pair<const void *, int>> g_big_smem;  // (kernel, device): more than 48 KiB allowed
thread_local dim3 t_grid, t_block;
thread_local size_t t_smem;
thread_local cudaStream_t t_stream;

Stream g_null[2] = {{0}, {1}};

Stream *stream_of(cudaStream_t s)
{
    return !s ? &g_null[g_device] : g_streams.count((Stream *)s) ? (Stream *)s : nullptr;
}

void enqueue(Stream *st, const Launch &l)
{
    g_before.push_back(st->before);
    st->before.insert((int)g_log.size());
    if (st->before.size() > 256)  // enough to check, and a long row stays quick
        st->before.erase(st->before.begin());
    g_log.push_back(l);
}

cudaError_t launch(const void *fn, dim3 grid, dim3 block, size_t smem, cudaStream_t s, void **args, bool programmatic,
                   bool copy_args)
{
    Stream *st = stream_of(s);
    if (!st || st->device != g_device)
        return cudaErrorInvalidResourceHandle;
    if (smem > 49152 && !g_big_smem.count({fn, g_device}))
        return cudaErrorInvalidValue;
    const long news = g_news;
    Launch l{};
    l.device = g_device;
    l.grid = (int)grid.x;
    l.block = (int)block.x;
    l.programmatic = programmatic;
    l.stream = (uint64_t)(uintptr_t)s;
    if (copy_args)
        std::memcpy(l.args, args[0], sizeof(l.args));
    std::strncpy(l.name, g_names[fn].c_str(), sizeof(l.name) - 1);
    enqueue(st, l);
    g_news = news;  // the record's own are not the library's
    return cudaSuccess;
}

}  // namespace

// Allocations of the library itself.
void *operator new(size_t n)
{
    ++g_news;
    if (void *p = std::malloc(n ? n : 1))
        return p;
    throw std::bad_alloc();
}
void *operator new(size_t n, const std::nothrow_t &) noexcept
{
    ++g_news;
    return std::malloc(n ? n : 1);
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, size_t) noexcept { std::free(p); }
void operator delete(void *p, const std::nothrow_t &) noexcept { std::free(p); }

extern "C" {

// --- what a test asks and sets ---
long fake_news() { return g_news; }
void fake_set_device(int d) { g_device = d; }
int fake_device() { return g_device; }
void fake_set_sms(int n) { g_sms = n; }
void *fake_stream(int device)
{
    Stream *s = new Stream{device};
    g_streams.insert(s);
    return s;
}
void fake_set_segment(size_t bytes) { g_segment = bytes; }
long fake_queries() { return g_queries; }
long fake_lookups() { return g_lookups; }
void fake_clear_costs() { g_costs.clear(); }
void fake_cost(int threads, float first, float next) { g_costs[threads] = {first, next}; }
void fake_reset()
{
    g_queries = g_lookups = 0;
    g_log.clear();
    g_before.clear();
    for (Stream &n : g_null)
        n.before.clear();
    for (Stream *s : g_streams)
        s->before.clear();
}
int fake_launches() { return (int)g_log.size(); }
void fake_launch(int i, Launch *out) { *out = g_log[(size_t)i]; }
// whether launch i runs behind launch j
int fake_behind(int i, int j) { return (int)g_before[(size_t)i].count(j); }
// a kernel of the caller's own, in a stream of the current device if null
void fake_other_kernel(void *stream)
{
    Launch l{};
    Stream *st = stream_of((cudaStream_t)stream);
    l.device = st->device;
    l.stream = (uint64_t)(uintptr_t)stream;
    enqueue(st, l);
}

// --- the runtime ---
cudaError_t cudaGetDevice(int *d) { return *d = g_device, cudaSuccess; }
cudaError_t cudaSetDevice(int d) { return g_device = d, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = g_sms, cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int)
{
    std::memset(p, 0, sizeof(*p));
    std::strcpy(p->name, "fake");
    p->multiProcessorCount = g_sms;
    return cudaSuccess;
}
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) { return *p = std::calloc(n ? n : 1, 1), cudaSuccess; }
cudaError_t cudaFree(void *p) { return std::free(p), cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) { return *p = nullptr, cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t, cudaStream_t) { return cudaMalloc(p, n); }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return cudaFree(p); }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *p, int v, size_t n) { return std::memset(p, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) { return cudaMemset(p, v, n); }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p)
{
    ++g_queries;
    std::memset(a, 0, sizeof(*a));
    a->type = cudaMemoryTypeDevice;
    a->devicePointer = const_cast<void *>(p);
    return cudaSuccess;  // every address is memory of device 0
}
// the driver calls behind an allocation's bounds: allocations of g_segment bytes
static int retain(void *, void *) { return 1; }  // not of mapped ranges
static int release(unsigned long long) { return 0; }
static int attribute(void *v, int, unsigned long long) { return *(void **)v = nullptr, 0; }
static int range(unsigned long long *base, size_t *size, unsigned long long p)
{
    ++g_lookups;
    *base = p / g_segment * g_segment;
    *size = g_segment;
    return 0;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *name, void **fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *r)
{
    const std::string n = name;
    *fn = n == "cuMemGetAddressRange"          ? (void *)range
          : n == "cuPointerGetAttribute"       ? (void *)attribute
          : n == "cuMemRetainAllocationHandle" ? (void *)retain
          : n == "cuMemRelease"                ? (void *)release
                                               : nullptr;
    *r = *fn ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned)
{
    *s = (cudaStream_t)fake_stream(g_device);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s)
{
    g_streams.erase((Stream *)s);
    delete (Stream *)s;
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *c)
{
    return *c = cudaStreamCaptureStatusNone, cudaSuccess;
}
cudaError_t cudaStreamGetDevice(cudaStream_t s, int *d)
{
    Stream *st = stream_of(s);
    return st ? (*d = st->device, cudaSuccess) : cudaErrorInvalidResourceHandle;
}
cudaError_t cudaStreamGetId(cudaStream_t s, unsigned long long *id)
{
    return *id = (unsigned long long)(uintptr_t)stream_of(s), cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned)
{
    Stream *st = stream_of(s);
    if (!st)
        return cudaErrorInvalidResourceHandle;
    st->before.insert(((Event *)e)->before.begin(), ((Event *)e)->before.end());
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned)
{
    *e = (cudaEvent_t) new Event{g_device, {}};
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return delete (Event *)e, cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s)
{
    Stream *st = stream_of(s);
    if (!st || st->device != ((Event *)e)->device)
        return cudaErrorInvalidResourceHandle;
    ((Event *)e)->before = st->before;
    ((Event *)e)->at = g_log.size();
    return cudaSuccess;
}
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t a, cudaEvent_t b)
{
    *ms = 0;
    for (size_t i = ((Event *)a)->at; i < ((Event *)b)->at; ++i) {
        const auto c = g_costs.find(g_log[i].block);
        *ms += 1e-3f * (c == g_costs.end() ? 1.f : i == ((Event *)a)->at ? c->second.first : c->second.second);
    }
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *fn, cudaFuncAttribute, int v)
{
    if (v > 49152)
        g_big_smem.insert({fn, g_device});
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned)
{
    return *n = 2, cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *fn, void **args)
{
    bool programmatic = false;
    for (unsigned i = 0; i < c->numAttrs; ++i)
        programmatic |= c->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization;
    return launch(fn, c->gridDim, c->blockDim, c->dynamicSmemBytes, c->stream, args, programmatic, true);
}

// --- what nvcc's host code calls for <<<>>> and for the embedded kernels ---
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void *s)
{
    t_grid = grid, t_block = block, t_smem = smem, t_stream = (cudaStream_t)s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *s)
{
    *grid = t_grid, *block = t_block, *smem = t_smem, *(cudaStream_t *)s = t_stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fn) { return *k = (cudaKernel_t)fn, cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void **args, size_t smem, cudaStream_t s)
{
    return launch((const void *)k, grid, block, smem, s, args, false, false);
}
void **__cudaRegisterFatBinary(void *) { return (void **)std::malloc(8); }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **h) { std::free(h); }
void __cudaRegisterFunction(void **, const char *fn, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *)
{
    g_names[fn] = name;
}

}  // extern "C"
