// A fake CUDA runtime for host code: several devices, each of which keeps what it was
// told about each kernel.  Like the real one, it allows a kernel 48 KiB of dynamic
// shared memory on a device until cudaFuncSetAttribute raises it there.  Device 2 has no
// room for a block, device 3 refuses more than 100 KiB.
#include <map>
#include <utility>

#include <cuda_runtime_api.h>

int fake_device = 0, fake_launches = 0;
static std::map<std::pair<int, const void*>, int> allowed;
static int allowed_of(const void* f) {
    auto it = allowed.find({fake_device, f});
    return it == allowed.end() ? 48 * 1024 : it->second;
}

extern "C" {
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
    if (a != cudaFuncAttributeMaxDynamicSharedMemorySize || (fake_device == 3 && v > 100 * 1024))
        return cudaErrorInvalidValue;
    allowed[{fake_device, f}] = v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int,
                                                                   size_t smem, unsigned) {
    if (smem > (size_t)allowed_of(f)) return cudaErrorInvalidValue;
    *n = fake_device == 2 ? 0 : 1;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void* f, int t, size_t s) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(n, f, t, s, 0);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
    if (c->dynamicSmemBytes > (size_t)allowed_of(f)) return cudaErrorInvalidValue;
    ++fake_launches;
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
// what nvcc's host code refers to; nothing here launches by it
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t) {
    return cudaErrorUnknown;
}
unsigned __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return 1; }
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*,
                            dim3*, int*) {}
void __cudaUnregisterFatBinary(void**) {}
}

