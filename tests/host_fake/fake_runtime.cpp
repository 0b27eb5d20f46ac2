// Stand-ins for the CUDA runtime, linked with the host pipeline's object (and fake_launch.cu) so that its order of copies,
// kernels, events and waits can be followed without a GPU.  Nothing runs: every call is written to a log, with the bytes that it
// reads and writes.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <cstdarg>
#include <cstdio>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <set>
#include <string>

static std::string g_log;
static long g_next = 1;
static std::set<long> g_live;                          // streams and events of the context that is current
static unsigned long long g_ctx = 1;
static bool g_bound = false;                           // whether the calling thread has a context
static long long g_rows = 0;
static int g_status = 0;

void say(const char *fmt, ...)
{
    char line[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(line, sizeof line, fmt, ap);
    va_end(ap);
    g_log += line;
    g_log += '\n';
}
long num(const void *h) { return (long)reinterpret_cast<intptr_t>(h); }
const char *dead(const void *h) { return g_live.count(num(h)) ? "" : " dead"; }
template <typename H> static cudaError_t make(H *h)
{
    g_live.insert(g_next);
    *h = reinterpret_cast<H>((intptr_t)g_next++);
    return cudaSuccess;
}
template <typename H> static cudaError_t drop(H h)
{
    say("destroy %ld%s", num(h), dead(h));
    g_live.erase(num(h));
    return cudaSuccess;
}

extern "C" {
const char *fake_log() { return g_log.c_str(); }
void fake_reset(long long rows, int status) { g_log.clear(); g_rows = rows; g_status = status; }
void fake_new_context() { ++g_ctx; g_bound = false; g_live.clear(); }    // what cudaDeviceReset leaves: the same handle, another context
long fake_live() { return (long)g_live.size(); }

static CUresult ctx_current(CUcontext *c) { *c = reinterpret_cast<CUcontext>((intptr_t)(g_bound ? 0x1000 : 0)); return CUDA_SUCCESS; }
static CUresult ctx_id(CUcontext, unsigned long long *id) { *id = g_ctx; return CUDA_SUCCESS; }
cudaError_t cudaGetDriverEntryPoint(const char *name, void **fn, unsigned long long, cudaDriverEntryPointQueryResult *r)
{
    *fn = !strcmp(name, "cuCtxGetCurrent") ? (void *)ctx_current : !strcmp(name, "cuCtxGetId") ? (void *)ctx_id : nullptr;
    if (r) *r = *fn ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { g_bound = true; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { *p = malloc(n); say("pinned %ld", num(*p)); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { say("unpinned %ld", num(p)); free(p); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return make(s); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return make(e); }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return drop(s); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return drop(e); }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { say("record %ld %ld%s%s", num(s), num(e), dead(s), dead(e)); return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) { say("wait %ld %ld%s%s", num(s), num(e), dead(s), dead(e)); return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { say("hostwait %ld%s", num(e), dead(e)); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { say("hostsync %ld%s", num(s), dead(s)); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int, size_t n, cudaStream_t s) { say("op %ld memset w %ld %zu%s", num(s), num(p), n, dead(s)); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t st)
{
    say("op %ld copy r %ld %zu w %ld %zu%s", num(st), num(s), n, num(d), n, dead(st));
    return cudaSuccess;
}

static struct { dim3 g, b; size_t smem; void *stream; } g_cfg;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st *stream) { g_cfg = {g, b, smem, stream}; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *stream)
{
    *g = g_cfg.g; *b = g_cfg.b; *smem = g_cfg.smem;
    *static_cast<void **>(stream) = g_cfg.stream;
    return cudaSuccess;
}
// the one kernel of the pipeline itself: (rows, status) of a layer into pinned memory
cudaError_t cudaLaunchKernel(const void *, dim3, dim3, void **args, size_t, cudaStream_t s)
{
    struct Meta { long long rows; int32_t status; };
    const void *rows = *static_cast<void **>(args[0]), *status = *static_cast<void **>(args[1]);
    Meta *out = *static_cast<Meta **>(args[2]);
    say("op %ld meta r %ld 8 r %ld 4 w %ld %zu%s", num(s), num(rows), num(status), num(out), sizeof(Meta), dead(s));
    *out = {g_rows, g_status};
    return cudaSuccess;
}
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
}
