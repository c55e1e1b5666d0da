// A stand-in for the CUDA runtime: libmpr's host code runs against it on the CPU, without a GPU.
// Device memory is host memory, copies are done at once, kernels do nothing but what the host code needs to
// go on (range and sample energy of a creation). Launches are recorded in order; a test reads them,
// limits memory, or has launches refused.
#include "fake_cudart.h"

#include <cuda_runtime.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <mutex>

namespace fake {

std::vector<Launch> launches;
std::function<int(const Launch&)> on_launch;
size_t alloc_limit = ~(size_t)0;
int refused_allocs = 0;

namespace {

std::mutex mu;
std::map<const void*, std::string>& names()
{
    static std::map<const void*, std::string> m;   // filled by the objects' static initialisers
    return m;
}
std::map<const void*, size_t> smem_limit;

void* get_memory(size_t n)
{
    if (n > alloc_limit) {
        ++refused_allocs;
        return nullptr;
    }
    return calloc(1, n ? n : 1);
}

cudaError_t launch(const void* f, unsigned grid, void** args, size_t smem, bool programmatic, bool cooperative)
{
    Launch l;
    {
        std::lock_guard<std::mutex> lock(mu);
        l.name = names()[f];
    }
    l.grid = grid;
    l.smem = smem;
    l.programmatic = programmatic;
    l.cooperative = cooperative;
    l.args = args;
    if (on_launch) {
        const int e = on_launch(l);
        if (e != cudaSuccess) return (cudaError_t)e;
    }
    std::lock_guard<std::mutex> lock(mu);
    const size_t most = smem_limit.count(f) ? smem_limit[f] : 48 * 1024;
    if (smem > most) return cudaErrorInvalidValue;
    if (l.name.find("minmax_final") != std::string::npos) {
        double* const out = *static_cast<double**>(args[2]);   // zmin, zmax, measured, not finite
        out[0] = 0.0;
        out[1] = 1.0;
        out[2] = 100.0;
    }
    if (l.name.find("sample_energy_final") != std::string::npos) {
        double* const out = *static_cast<double**>(args[3]);   // e_s, pairs
        out[0] = -0.5;
        out[1] = 10.0;
    }
    launches.push_back(l);
    return cudaSuccess;
}

struct Config {
    dim3 grid, block;
    size_t smem;
    void* stream;
};
thread_local Config pushed;

}  // namespace
}  // namespace fake

extern "C" {

void** __cudaRegisterFatBinary(void*)
{
    static void* h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*,
                            dim3*, int*)
{
    fake::names()[host] = name;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f)
{
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, CUstream_st* st)
{
    fake::pushed = fake::Config{grid, block, smem, st};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* st)
{
    *grid = fake::pushed.grid;
    *block = fake::pushed.block;
    *smem = fake::pushed.smem;
    *static_cast<void**>(st) = fake::pushed.stream;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void** args, size_t smem, cudaStream_t)
{
    return fake::launch((const void*)k, grid.x, args, smem, false, false);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args)
{
    bool pdl = false, coop = false;
    for (unsigned i = 0; i < c->numAttrs; ++i) {
        pdl |= c->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization &&
               c->attrs[i].val.programmaticStreamSerializationAllowed;
        coop |= c->attrs[i].id == cudaLaunchAttributeCooperative && c->attrs[i].val.cooperative;
    }
    return fake::launch(f, c->gridDim.x, args, c->dynamicSmemBytes, pdl, coop);
}
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3 grid, dim3, void** args, size_t smem, cudaStream_t)
{
    return fake::launch(f, grid.x, args, smem, false, true);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v)
{
    std::lock_guard<std::mutex> lock(fake::mu);
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) fake::smem_limit[f] = (size_t)v;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int)
{
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d)
{
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t)
{
    *n = 4;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned)
{
    *n = 4;
    return cudaSuccess;
}

cudaError_t cudaMalloc(void** p, size_t n)
{
    return (*p = fake::get_memory(n)) ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) { return cudaMalloc(p, n); }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned)
{
    return (*p = calloc(1, n)) ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void* p)
{
    free(p);
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return cudaFree(p); }
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*)
{
    static int pool;
    *p = (cudaMemPool_t)&pool;
    return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n)
{
    memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { return cudaMemset(p, v, n); }
cudaError_t cudaGetSymbolAddress(void**, const void*) { return cudaErrorInvalidSymbol; }

cudaError_t cudaEventCreate(cudaEvent_t* e)
{
    static int event;
    *e = (cudaEvent_t)&event;
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t)
{
    *ms = 1.0f;
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "error of the stand-in runtime"; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void**, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult*)
{
    return cudaErrorNotSupported;   // no tensor maps
}

// graphs: batches are not run against this runtime
cudaError_t cudaGraphCreate(cudaGraph_t*, unsigned) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphAddKernelNode(cudaGraphNode_t*, cudaGraph_t, const cudaGraphNode_t*, size_t,
                                   const cudaKernelNodeParams*)
{
    return cudaErrorNotSupported;
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t*, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*,
                             size_t, cudaGraphNodeParams*)
{
    return cudaErrorNotSupported;
}
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle*, cudaGraph_t, unsigned, unsigned)
{
    return cudaErrorNotSupported;
}
cudaError_t cudaGraphKernelNodeSetAttribute(cudaGraphNode_t, cudaLaunchAttributeID, const cudaLaunchAttributeValue*)
{
    return cudaErrorNotSupported;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphUpload(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaErrorNotSupported; }

}  // extern "C"
