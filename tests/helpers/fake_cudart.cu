// Test helper, not part of the library: a CUDA runtime without a GPU. The library's host code is linked against it
// in place of the real one; "device" memory is host memory, no kernel runs, and every launch is written down, with
// what the tests ask about. So the order and the form of the launches can be tested on a machine without a GPU.
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <string>
#include <vector>

#include "od_draw.cuh"

namespace {

std::map<const void *, std::string> &kernels() { static std::map<const void *, std::string> k; return k; }
std::string &log_text() { static std::string s; return s; }
struct Range { const char *p; size_t bytes; };
std::vector<Range> &pinned() { static std::vector<Range> v; return v; }
bool no_driver_functions = false;
unsigned cluster_limit = 16;                                 // blocks of the largest cluster that the device has room for

unsigned cluster_of(const cudaLaunchConfig_t *cfg)
{
    unsigned blocks = 1;
    for (unsigned i = 0; i < cfg->numAttrs; ++i)
        if (cfg->attrs[i].id == cudaLaunchAttributeClusterDimension)
            blocks = cfg->attrs[i].val.clusterDim.x * cfg->attrs[i].val.clusterDim.y * cfg->attrs[i].val.clusterDim.z;
    return blocks;
}

const char *const NAMES[] = {"od_map_kernel", "od_verify_stream_kernel", "od_verify_decide_kernel", "od_verify_finish_kernel",
                             "od_verify_rows_kernel", "od_sample_kernel", "od_sample_shard_kernel", "od_step_kernel",
                             "fetch_logits_kernel", "fetch_drafter_kernel", "od_exit_kernel"};

// one line per launch: name, grid, and what of the launch in front the kernel may read ahead (-1: not a question)
cudaError_t launched(const void *func, dim3 grid, void **args)
{
    std::string name = kernels()[func];
    for (const char *n : NAMES)
        if (name.find(n) != std::string::npos) name = n;
    int early = -1;
    if (name == "od_map_kernel") early = *(const int32_t *)args[11];
    if (name == "od_sample_kernel" || name == "od_sample_shard_kernel") early = ((const SampleArgs *)args[0])->early;
    char line[256];
    snprintf(line, sizeof(line), "%.100s %u %u %u %d\n", name.c_str(), grid.x, grid.y, grid.z, early);
    log_text() += line;
    return cudaSuccess;
}

int context_id(void *, unsigned long long *id) { *id = 1; return 0; }
int pointer_attribute(void *data, int what, unsigned long long p)
{
    for (const Range &r : pinned())
        if ((uintptr_t)r.p <= p && p < (uintptr_t)r.p + r.bytes) {
            const unsigned long long value = what == 11 ? (unsigned long long)(uintptr_t)r.p : (unsigned long long)r.bytes;
            memcpy(data, &value, 8);
            return 0;
        }
    return 1;
}

struct Config { dim3 grid, block; size_t smem; cudaStream_t stream; } pushed;

}  // namespace

extern "C" {

// ---- for the tests
const char *fake_log(void) { static std::string last; last = log_text(); log_text().clear(); return last.c_str(); }
void fake_pin(const void *p, size_t bytes) { pinned().push_back({(const char *)p, bytes}); }
void fake_unpin_all(void) { pinned().clear(); }
void fake_no_driver_functions(int none) { no_driver_functions = none != 0; }
void fake_cluster_limit(int blocks) { cluster_limit = (unsigned)blocks; }

// ---- the runtime
#ifndef __CUDA_ARCH__                                        // (the device's has some of the same names)
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
char __cudaInitModule(void **) { return 0; }
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) { kernels()[host] = name; }
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t s) { pushed = {grid, block, smem, s}; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *s)
{
    *grid = pushed.grid; *block = pushed.block; *smem = pushed.smem; *(cudaStream_t *)s = pushed.stream;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void *func, dim3 grid, dim3, void **args, size_t, cudaStream_t) { return launched(func, grid, args); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *cfg, const void *func, void **args)
{
    return cluster_of(cfg) > cluster_limit ? cudaErrorInvalidClusterSize : launched(func, cfg->gridDim, args);
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int)
{
    *v = a == cudaDevAttrMultiProcessorCount ? 148 : a == cudaDevAttrComputeCapabilityMajor ? 10 : 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaFree(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) { return posix_memalign(p, 256, n ? n : 1) == 0 ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind kind, cudaStream_t)
{
    memcpy(d, s, n);
    char line[64];
    snprintf(line, sizeof(line), "%s %zu\n", kind == cudaMemcpyHostToDevice ? "to_device" : "to_host", n);
    log_text() += line;
    return cudaSuccess;
}
cudaError_t cudaMemset(void *p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int *n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *s) { *p = const_cast<void *>(s); return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *cfg)
{
    *n = cluster_of(cfg) > cluster_limit ? 0 : 148 / (int)cluster_of(cfg);
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *name, void **fn, unsigned, unsigned long long, cudaDriverEntryPointQueryResult *)
{
    *fn = no_driver_functions ? nullptr : !strcmp(name, "cuCtxGetId") ? (void *)context_id : (void *)pointer_attribute;
    return *fn ? cudaSuccess : cudaErrorSymbolNotFound;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *at, const void *p)
{
    memset(at, 0, sizeof(*at));
    at->type = cudaMemoryTypeUnregistered;
    for (const Range &r : pinned())
        if (r.p <= (const char *)p && (const char *)p < r.p + r.bytes) {
            at->type = cudaMemoryTypeHost;
            at->hostPointer = at->devicePointer = const_cast<void *>(p);
        }
    return cudaSuccess;
}
#endif

}  // extern "C"
