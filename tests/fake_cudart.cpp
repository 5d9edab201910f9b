// A CUDA runtime without a GPU: what the library's host code calls, as far as it calls it.  Every call succeeds unless the test asked
// for its failure, is counted under its name, and kernel launches are counted under the kernel's name as well.  Linked into a build of
// the library in place of the runtime (tests/test_host_paths.py).
#include <cuda_runtime_api.h>
#include <map>
#include <string>

namespace {
struct Plan { int skip, count; cudaError_t code; };
std::map<std::string, Plan> plans;
std::map<std::string, int> calls;
std::map<const void *, std::string> &kernels()           // (filled by constructors that run before this file's)
{
    static std::map<const void *, std::string> names;
    return names;
}
cudaError_t last = cudaSuccess;
int pointer_device = 0, pointer_type = cudaMemoryTypeDevice, max_clusters = 148, capturing = 0;
size_t handles = 4096;

cudaError_t call(const std::string &name)
{
    ++calls[name];
    const auto it = plans.find(name);
    if (it == plans.end() || it->second.count == 0) return cudaSuccess;
    if (it->second.skip > 0) { --it->second.skip; return cudaSuccess; }
    if (it->second.count > 0) --it->second.count;
    return last = it->second.code;
}
template <class T> cudaError_t made(const char *name, T *out)
{
    *out = (T)(handles += 64);
    return call(name);
}
cudaError_t launch(const void *fn)
{
    const cudaError_t e = call("launch");
    if (e == cudaSuccess) ++calls[kernels()[fn]];
    return e;
}
struct { dim3 grid, block; size_t smem; cudaStream_t s; } config;
}

extern "C" {
// ---- what the test says and asks ---------------------------------------------------------------------------------
void fake_reset() { plans.clear(); calls.clear(); last = cudaSuccess; pointer_device = 0; pointer_type = cudaMemoryTypeDevice; max_clusters = 148; capturing = 0; }
void fake_fail(const char *name, int skip, int count, int code) { plans[name] = Plan{skip, count, (cudaError_t)code}; }   // count -1: always
void fake_pointers(int device, int type) { pointer_device = device; pointer_type = type; }
void fake_clusters(int n) { max_clusters = n; }
void fake_capturing(int on) { capturing = on; }
int fake_calls(const char *part)                       // calls whose name contains `part`
{
    int n = 0;
    for (const auto &c : calls)
        if (c.first.find(part) != std::string::npos) n += c.second;
    return n;
}

// ---- the runtime ---------------------------------------------------------------------------------------------------
void **__cudaRegisterFatBinary(void *) { return (void **)&config; }
char __cudaInitModule(void **) { return 1; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *)
{
    kernels()[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st *s)
{
    config = {grid, block, smem, s};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *s)
{
    *grid = config.grid;
    *block = config.block;
    *smem = config.smem;
    *(cudaStream_t *)s = config.s;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void *fn, dim3, dim3, void **, size_t, cudaStream_t) { return launch(fn); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *fn, void **) { return launch(fn); }
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return call("cudaGetDevice"); }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr, int) { *v = 148; return call("cudaDeviceGetAttribute"); }
cudaError_t cudaFuncSetAttribute(const void *, enum cudaFuncAttribute, int) { return call("cudaFuncSetAttribute"); }
cudaError_t cudaGetSymbolAddress(void **p, const void *) { return made("cudaGetSymbolAddress", p); }
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *)
{
    *n = max_clusters;
    return call("cudaOccupancyMaxActiveClusters");
}
cudaError_t cudaPointerGetAttributes(struct cudaPointerAttributes *a, const void *p)
{
    *a = cudaPointerAttributes();
    a->type = (enum cudaMemoryType)pointer_type;
    a->device = pointer_device;
    a->devicePointer = a->hostPointer = const_cast<void *>(p);
    return call("cudaPointerGetAttributes");
}
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, enum cudaMemcpyKind, cudaStream_t) { return call("cudaMemcpyAsync"); }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return call("cudaMemsetAsync"); }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return made("cudaStreamCreateWithFlags", s); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return call("cudaStreamDestroy"); }
cudaError_t cudaStreamGetDevice(cudaStream_t, int *d) { *d = 0; return call("cudaStreamGetDevice"); }
cudaError_t cudaStreamIsCapturing(cudaStream_t, enum cudaStreamCaptureStatus *st)
{
    *st = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return call("cudaStreamIsCapturing");
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return call("cudaStreamSynchronize"); }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return call("cudaStreamWaitEvent"); }
cudaError_t cudaThreadExchangeStreamCaptureMode(enum cudaStreamCaptureMode *) { return call("cudaThreadExchangeStreamCaptureMode"); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return made("cudaEventCreateWithFlags", e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return call("cudaEventDestroy"); }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return call("cudaEventRecord"); }
cudaError_t cudaGraphCreate(cudaGraph_t *g, unsigned) { return made("cudaGraphCreate", g); }
cudaError_t cudaGraphAddNode_v2(cudaGraphNode_t *n, cudaGraph_t, const cudaGraphNode_t *, const cudaGraphEdgeData *, size_t,
                                struct cudaGraphNodeParams *)
{
    return made("cudaGraphAddNode", n);
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long)
{
    const cudaError_t e = made("cudaGraphInstantiate", x);
    if (e != cudaSuccess) *x = nullptr;
    return e;
}
cudaError_t cudaGraphExecNodeSetParams(cudaGraphExec_t, cudaGraphNode_t, struct cudaGraphNodeParams *) { return call("cudaGraphExecNodeSetParams"); }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return call("cudaGraphLaunch"); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return call("cudaGraphDestroy"); }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return call("cudaGraphExecDestroy"); }
}
