// A stand-in for the CUDA runtime that launches nothing: linked with libfr's
// objects in place of the real one, it lets the library's host code run on a
// machine without a GPU and keeps a list of the kernels it would have launched
// (mangled name, grid, block).  Memory is never touched; every query succeeds.
#include <cstring>
#include <map>
#include <string>

#include <cuda_runtime.h>

#define EXPORT extern "C" __attribute__((visibility("default")))

namespace {
std::map<const void *, std::string> &kernels()
{
    static std::map<const void *, std::string> m;
    return m;
}
std::string &record()
{
    static std::string s;
    return s;
}
struct Config {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
} g_config;
}  // namespace

// "name gridx blockx\n" of every launch since the last call with clear set
EXPORT const char *fake_launches(int clear)
{
    static std::string out;
    out = record();
    if (clear) record().clear();
    return out.c_str();
}

// the mangled names of all kernels of the library, one per line
EXPORT const char *fake_kernels(void)
{
    static std::string out;
    out.clear();
    for (const auto &k : kernels()) out += k.second + "\n";
    return out.c_str();
}

extern "C" {

void **__cudaRegisterFatBinary(void *)
{
    static void *handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *,
                            dim3 *, int *)
{
    kernels()[host] = name;
}

unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st *stream)
{
    g_config = {grid, block, smem, stream};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *stream)
{
    *grid = g_config.grid;
    *block = g_config.block;
    *smem = g_config.smem;
    std::memcpy(stream, &g_config.stream, sizeof g_config.stream);
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *kernel, const void *host)
{
    *kernel = (cudaKernel_t)const_cast<void *>(host);
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t kernel, dim3 grid, dim3 block, void **, size_t, cudaStream_t)
{
    record() += kernels()[(const void *)kernel] + " " + std::to_string(grid.x) + " " + std::to_string(block.x) + "\n";
    return cudaSuccess;
}

cudaError_t cudaGetDevice(int *dev)
{
    *dev = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *value, cudaDeviceAttr, int)
{
    *value = 152;  // asked for the number of SMs only
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *blocks, const void *, int, size_t, unsigned)
{
    *blocks = 2;
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return ""; }
cudaError_t cudaGetSymbolAddress(void **address, const void *symbol)
{
    *address = const_cast<void *>(symbol);
    return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *status)
{
    *status = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}

}  // extern "C"
