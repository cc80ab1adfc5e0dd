// A stand-in for the CUDA runtime, linked with the library's objects by test_host_calls.py, so that
// the order of the host's calls can be tested without a GPU: it runs no kernel and holds no device
// memory, but keeps, per stream, how much of every other stream's work it is ordered after, can
// make the n-th call that queues work fail, and lists the launches.
#include <cuda_runtime.h>
#include <cuda.h>

#include <algorithm>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {

using Clock = std::map<cudaStream_t, long>;  // work of each stream that is done before

struct Fake {
    std::map<cudaStream_t, Clock> at;         // a stream: the work its next call is ordered after
    std::map<cudaEvent_t, Clock> events;
    Clock done;                               // work the host has waited for
    std::map<const void *, std::string> names;
    std::string log;                          // "name grid.x grid.y grid.z block smem stream\n" a launch
    long ids = 0x1000, calls = 0, fail_at = -1;
    uintptr_t memory = 1ull << 32;
    cudaError_t last = cudaSuccess;
    struct { dim3 grid, block; size_t smem; cudaStream_t st; } config;
} f;

void merge(Clock &into, const Clock &c)
{
    for (auto &k : c) into[k.first] = std::max(into[k.first], k.second);
}
bool fails()  // one of the calls that can be made to fail
{
    if (++f.calls - 1 != f.fail_at) return false;
    f.last = cudaErrorUnknown;
    return true;
}
cudaError_t work(cudaStream_t st)
{
    if (fails()) return cudaErrorUnknown;
    f.at[st][st] += 1;
    return cudaSuccess;
}
cudaError_t launch(const void *fn, dim3 grid, dim3 block, size_t smem, cudaStream_t st)
{
    if (cudaError_t e = work(st)) return e;
    auto n = [](unsigned v) { return std::to_string(v) + " "; };
    f.log += f.names[fn] + " " + n(grid.x) + n(grid.y) + n(grid.z) + n(block.x) + std::to_string(smem) + " " +
             std::to_string((uintptr_t)st) + "\n";
    return cudaSuccess;
}
CUresult encode_tiled(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                      const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                      CUtensorMapL2promotion, CUtensorMapFloatOOBfill)
{
    return CUDA_SUCCESS;
}

}  // namespace

extern "C" {

// ---- the test's side
void fake_reset()  // forget work, waits and launches
{
    f.at.clear(); f.events.clear(); f.done.clear(); f.log.clear();
    f.calls = 0; f.fail_at = -1; f.last = cudaSuccess;
}
void fake_fail_at(long n) { f.calls = 0; f.fail_at = n; }
long fake_calls() { return f.calls; }
const char *fake_log() { return f.log.c_str(); }
// work of other streams that neither `st` nor the host waits for
long fake_unjoined(cudaStream_t st)
{
    long n = 0;
    for (auto &s : f.at)
        if (s.first != st) n += std::max(0L, s.second[s.first] - std::max(f.at[st][s.first], f.done[s.first]));
    return n;
}

// ---- the runtime's
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *)
{
    f.names[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t st)
{
    f.config = {grid, block, smem, st};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *st)
{
    *grid = f.config.grid; *block = f.config.block; *smem = f.config.smem;
    *(cudaStream_t *)st = f.config.st;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fn) { *k = (cudaKernel_t)fn; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void **, size_t smem, cudaStream_t st)
{
    return launch((const void *)k, grid, block, smem, st);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *fn, void **)
{
    return launch(fn, c->gridDim, c->blockDim, c->dynamicSmemBytes, c->stream);
}
cudaError_t cudaGetLastError(void) { return std::exchange(f.last, cudaSuccess); }
const char *cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int *n) { *n = 1; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int)
{
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 227 * 1024 : 0;
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *)
{
    memset(a, 0, sizeof *a);
    a->numRegs = 128;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int threads, size_t smem)
{
    *n = threads <= 256 && smem <= 113 * 1024 ? 2 : 1;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *fn, const cudaLaunchConfig_t *c)
{
    unsigned cl = 1;
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cl = c->attrs[i].val.clusterDim.x;
    int per_sm;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, (int)c->blockDim.x, c->dynamicSmemBytes);
    *n = (int)(per_sm * 152 / cl);
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q)
{
    *fn = (void *)encode_tiled;
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *) { *p = (void *)(1ull << 31); return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n)
{
    *p = (void *)f.memory;
    f.memory += (n + 511) / 256 * 256;
    return cudaSuccess;
}
cudaError_t cudaFree(void *) { return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemset(void *, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemcpy(void *, const void *, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t st) { return work(st); }
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t st) { return work(st); }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)f.ids++; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { merge(f.done, f.at[s]); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)f.ids++; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s)
{
    if (fails()) return cudaErrorUnknown;
    f.events[e] = f.at[s];
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned)
{
    if (fails()) return cudaErrorUnknown;
    merge(f.at[s], f.events[e]);
    return cudaSuccess;
}

}  // extern "C"
