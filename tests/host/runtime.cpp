// A CUDA runtime for tests without a GPU: the library's own objects are linked against it instead of the real one, so that the
// host code runs as it is, planning and launches included, with addresses that nothing dereferences.  Launches and
// tensor maps go to launches.cu.
#include <cuda_runtime_api.h>

extern "C" {
void host_kernel(const void* host, const char* name);
void host_array(const void* host, size_t bytes);
void* host_array_address(const void* host);
void host_launch(const void* kernel, unsigned blocks, void** args);
void* host_encode();
bool host_refuses(const void* kernel);

void** __cudaRegisterFatBinary(void*) { static void* handle; return &handle; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) { host_kernel(host, name); }
void __cudaRegisterVar(void**, char* host, char*, const char*, int, size_t bytes, int, int) { host_array(host, bytes); }
static struct { dim3 grid, block; size_t smem; void* stream; } configured;
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st* stream) {
    configured.grid = grid; configured.block = block; configured.smem = smem; configured.stream = stream;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* stream) {
    *grid = configured.grid; *block = configured.block; *smem = configured.smem;
    *static_cast<void**>(stream) = configured.stream;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void* kernel, dim3 grid, dim3, void** args, size_t, cudaStream_t) {
    host_launch(kernel, grid.x * grid.y * grid.z, args);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* kernel, void** args) {
    host_launch(kernel, c->gridDim.x * c->gridDim.y * c->gridDim.z, args);
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int* device) { *device = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* value, cudaDeviceAttr, int) { *value = 148; return cudaSuccess; }      // asked for the SMs only
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* kernel, cudaFuncAttribute, int) { return host_refuses(kernel) ? cudaErrorInvalidValue : cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMemcpy(void*, const void*, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemset2DAsync(void*, size_t, int, size_t, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** address, const void* symbol) {
    *address = host_array_address(symbol);
    return *address ? cudaSuccess : cudaErrorInvalidSymbol;
}
cudaError_t cudaGetDriverEntryPoint(const char*, void** fn, unsigned long long, cudaDriverEntryPointQueryResult* found) {
    *fn = host_encode();
    if (found) *found = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
}
