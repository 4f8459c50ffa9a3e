// Stand-ins for the CUDA runtime and the kernel launchers, so that api.cu's host side (the order of what it queues, what it
// does when a call fails) can be run without a device: every call is written to a log, device memory is host memory, and the
// n-th call of a name can be made to fail.
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <string>
#include <vector>

#include <cuda.h>

#include "common.cuh"

namespace {

std::string g_log;
std::map<std::string, int> g_fail;                       // name -> calls until one fails
struct Range { const char *lo; size_t bytes; };
std::vector<Range> g_pinned;
const void *g_device = nullptr;                          // a pointer that is said to be the device's
const int kSms = 148;
bool g_capturing = false;

cudaError_t call(const char *name, const char *fmt = "", ...)
{
    char buf[256];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_log += std::string(name) + " " + buf + "\n";
    auto it = g_fail.find(name);
    if (it != g_fail.end() && --it->second == 0) return cudaErrorUnknown;
    return cudaSuccess;
}
const Range *pinned(const void *p)
{
    for (const Range &r : g_pinned)
        if ((const char *)p >= r.lo && (const char *)p < r.lo + r.bytes) return &r;
    return nullptr;
}
unsigned id(const void *p) { return (unsigned)(uintptr_t)p; }

}  // namespace

extern "C" {

const char *fake_log() { return g_log.c_str(); }
void fake_reset() { g_log.clear(); g_fail.clear(); g_pinned.clear(); g_device = nullptr; }
void fake_device(const void *p) { g_device = p; }
void fake_capture(int on) { g_capturing = on != 0; }
void fake_fail(const char *name, int nth) { g_fail[name] = nth; }
void fake_pin(const void *p, size_t bytes) { g_pinned.push_back({(const char *)p, bytes}); }

cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = kSms; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) { *p = aligned_alloc(256, (n + 255) / 256 * 256); return cudaSuccess; }
cudaError_t cudaFree(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemset(void *, int, size_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)0x51; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { static size_t n = 0xe0; *e = (cudaEvent_t)++n; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t s) { return call("event_record", "stream=%x", id(s)); }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t, unsigned) { return call("stream_wait", "stream=%x", id(s)); }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s)
{
    *s = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return call("sync", "stream=%x", id(s)); }
cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t n, cudaMemcpyKind k, cudaStream_t s)
{
    if (k == cudaMemcpyDeviceToHost && n == sizeof(int)) *(int *)dst = 0;      // (the status word)
    return call(k == cudaMemcpyHostToDevice ? "h2d" : k == cudaMemcpyDeviceToHost ? "d2h" : "d2d", "host=%llx bytes=%zu stream=%x",
                (unsigned long long)(uintptr_t)(k == cudaMemcpyHostToDevice ? src : dst), n, id(s));
}
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p)
{
    const bool in = pinned(p) != nullptr;
    a->type = p == g_device ? cudaMemoryTypeDevice : in ? cudaMemoryTypeHost : cudaMemoryTypeUnregistered;
    a->devicePointer = in ? const_cast<void *>(p) : nullptr;
    a->hostPointer = const_cast<void *>(p);
    return cudaSuccess;
}

CUresult fake_pointer_attribute(void *data, CUpointer_attribute what, CUdeviceptr p)
{
    const Range *r = pinned((const void *)p);
    if (!r) return CUDA_ERROR_INVALID_VALUE;
    if (what == CU_POINTER_ATTRIBUTE_RANGE_START_ADDR) *(CUdeviceptr *)data = (CUdeviceptr)r->lo;
    else if (what == CU_POINTER_ATTRIBUTE_RANGE_SIZE) *(size_t *)data = r->bytes;
    else return CUDA_ERROR_INVALID_VALUE;
    return CUDA_SUCCESS;
}
cudaError_t cudaGetDriverEntryPoint(const char *, void **fn, unsigned long long, cudaDriverEntryPointQueryResult *q)
{
    *fn = (void *)fake_pointer_attribute;
    if (q) *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}

}  // extern "C"

int fspad_attn_mtiles(const fspad_ctx *c, int N, int, int) { return (N * (c->cfg.n_q_heads / c->cfg.n_kv_heads) + 127) / 128; }
int fspad_attn_umma_splits(const fspad_ctx *c, int N, int B, int sms)
{
    const int s = (sms > 0 ? sms : kSms) / (B * c->cfg.n_kv_heads * fspad_attn_mtiles(c, N, B, sms)), chunks = (c->cfg.max_len + 127) / 128;
    return chunks <= 5 || s < 1 ? 1 : s < chunks ? s : chunks;
}
int fspad_attn_ranges(const fspad_ctx *c, int N, int B, int sms, int, bool) { return fspad_attn_umma_splits(c, N, B, sms); }
int fspad_draft_expand_pieces(int V) { return (V + 4095) / 4096; }
int fspad_lm_head_tiles(int V) { return (V + 127) / 128; }
int fspad_walk_ctas(fspad_ctx *, int B, int V)
{
    int c = 16;
    while (c > 1 && (V + c - 1) / c < 2048) c >>= 1;
    return B * (c == 16 && B > 7 ? 10 : c);
}
size_t fspad_feature_sampler_scratch_floats(int, int, int) { return 0; }
FspadStatsGeom fspad_lm_head_geom(int, int, bool, int) { return FspadStatsGeom(); }

cudaError_t fspad_launch_tree_attn(fspad_ctx *, const fspad_bf16 *, const fspad_bf16 *, const fspad_bf16 *, const fspad_bf16 *,
                                   const fspad_bf16 *, const int *, const int *, int, int, fspad_bf16 *, cudaStream_t st, int sms,
                                   FspadPaged paged, bool)
{
    return call("attention", "sms=%d early=%d stream=%x", sms, (int)paged.early, id(st));
}
cudaError_t fspad_launch_accept_walk(fspad_ctx *, const float *, const float *draft, const int *, const int *, const float *,
                                     const float *, const FspadStatsGeom &, int, int, int, int *, int *, int *, cudaStream_t st,
                                     FspadWalkCompact kv, bool far)
{
    return call("walk", "draft=%llx far=%d compacts=%d stream=%x", (unsigned long long)(uintptr_t)draft, (int)far, (int)(kv.cache != nullptr), id(st));
}
cudaError_t fspad_launch_stats_partials(fspad_ctx *, const float *, const float *, int, int, int, FspadStatsGeom *geom, cudaStream_t st,
                                        bool, int)
{
    return call("scan", "trees=%d staged=%d stream=%x", (int)(geom->parent != nullptr), (int)(geom->stage != nullptr), id(st));
}
cudaError_t fspad_launch_kv_compact(fspad_ctx *, fspad_bf16 *, const int *, const int *, const int *, int, int *, cudaStream_t st, bool)
{
    return call("compact", "stream=%x", id(st));
}
cudaError_t fspad_launch_tree_scatter(fspad_ctx *, fspad_bf16 *, const fspad_bf16 *, const fspad_bf16 *, const int *, int, int,
                                      cudaStream_t st)
{
    return call("scatter", "stream=%x", id(st));
}
// not reached by what is tested here
cudaError_t fspad_launch_accept_stats(fspad_ctx *, const float *, const float *, int, int, int, float *, double *, int *, cudaStream_t)
{ return cudaErrorUnknown; }
cudaError_t fspad_launch_draft_expand(fspad_ctx *, const float *, const float *, const int *, int, int, int, int, int, int, int *, int *,
                                      float *, int *, float *, cudaStream_t)
{ return cudaErrorUnknown; }
cudaError_t fspad_launch_feature_sampler(fspad_ctx *, const fspad_bf16 *, const fspad_bf16 *, const fspad_bf16 *, const fspad_bf16 *,
                                         const fspad_bf16 *, int, int, int, fspad_bf16 *, fspad_bf16 *, float *, cudaStream_t)
{ return cudaErrorUnknown; }
cudaError_t fspad_launch_kv_append(fspad_ctx *, fspad_bf16 *, const fspad_bf16 *, const int *, const int *, const int *, int, int, int *,
                                   cudaStream_t)
{ return cudaErrorUnknown; }
cudaError_t fspad_launch_kv_compact_paged(fspad_ctx *, fspad_bf16 *, FspadPaged, const int *, const int *, const int *, int, int *,
                                          cudaStream_t)
{ return cudaErrorUnknown; }
cudaError_t fspad_launch_lm_head(fspad_ctx *, const fspad_bf16 *, const fspad_bf16 *, int, int, int, const float *, float *,
                                 const FspadStatsGeom *, float *, double *, int *, cudaStream_t)
{ return cudaErrorUnknown; }
cudaError_t fspad_launch_tree_build(fspad_ctx *, const int *, const int *, const float *, const int *, int, int, int, int *, int *, int *,
                                    unsigned long long *, int *, cudaStream_t)
{ return cudaErrorUnknown; }
cudaError_t fspad_launch_wait_selftest(fspad_ctx *, int, cudaStream_t) { return cudaErrorUnknown; }
cudaError_t fspad_launch_walk_wait_selftest(fspad_ctx *, int, cudaStream_t) { return cudaErrorUnknown; }
