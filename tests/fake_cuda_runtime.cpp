// A stand-in for the CUDA runtime, linked with the library's host code so that its launches can be looked at on a machine
// without a GPU: every kernel launch, memset and copy is written down as one line of text, and a launch can be made to fail.
// Nothing here runs device code.
#include <cuda.h>
#include <cuda_runtime.h>

#include <map>
#include <string>

static std::map<const void*, std::string> names;         // host stub -> mangled kernel name
static std::string log_text;
static int refuse_clusters = 0, refuse_cooperative = 0;  // status of such launches (0: they go through)
static cudaError_t last = cudaSuccess;

extern "C" {
const char* fake_log() { return log_text.c_str(); }
void fake_reset(int clusters, int cooperative)
{
    log_text.clear();
    refuse_clusters = clusters;
    refuse_cooperative = cooperative;
    last = cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) { static void* handle; return &handle; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 0; }
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* stub, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) { names[stub] = name; }
unsigned __cudaPushCallConfiguration(dim3 grid, dim3, size_t, cudaStream_t)
{
    log_text += "grid " + std::to_string(grid.x) + " ";
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* stream)
{
    *grid = *block = dim3(1);
    *smem = 0;
    *static_cast<cudaStream_t*>(stream) = nullptr;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void* stub, dim3, dim3, void**, size_t, cudaStream_t)
{
    log_text += names[stub] + "\n";
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* cfg, const void* stub, void**)
{
    unsigned cluster = 1;
    int cooperative = 0;
    for (unsigned i = 0; i < cfg->numAttrs; ++i) {
        if (cfg->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = cfg->attrs[i].val.clusterDim.x;
        if (cfg->attrs[i].id == cudaLaunchAttributeCooperative) cooperative = cfg->attrs[i].val.cooperative;
    }
    const int status = cluster > 1 && refuse_clusters ? refuse_clusters : cooperative && refuse_cooperative ? refuse_cooperative : 0;
    log_text += "grid " + std::to_string(cfg->gridDim.x) + " cluster " + std::to_string(cluster) + (cooperative ? " cooperative " : " ") +
                (status ? "refused " : "") + names[stub] + "\n";
    if (status) last = static_cast<cudaError_t>(status);
    return static_cast<cudaError_t>(status);
}
cudaError_t cudaGetLastError()
{
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
cudaError_t cudaMemsetAsync(void* p, int value, size_t n, cudaStream_t)
{
    log_text += "memset " + std::to_string(reinterpret_cast<size_t>(p)) + " " + std::to_string(value) + " " + std::to_string(n) + "\n";
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpyFromSymbol(void*, const void*, size_t, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemcpyToSymbol(const void*, const void*, size_t, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = reinterpret_cast<void*>(0x100000); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetDevice(int* dev) { *dev = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* value, cudaDeviceAttr, int) { *value = 148; return cudaSuccess; }      // (the SM count is all that is asked for)
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
static CUresult encode(...) { return CUDA_SUCCESS; }
cudaError_t cudaGetDriverEntryPoint(const char*, void** fn, unsigned long long, cudaDriverEntryPointQueryResult* found)
{
    *fn = reinterpret_cast<void*>(&encode);
    if (found) *found = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
}
