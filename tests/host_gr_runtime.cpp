// Fake of the CUDA runtime calls of k_observe.cu: the limit of dynamic shared memory of every
// kernel, and what each launch asks for.  Linked in place of the runtime by
// tests/test_host_gr_launch.py.
#include <cuda_runtime_api.h>

#include <cstring>
#include <map>

static std::map<const void*, int> limit;
static int lowered = 0, beyond = 0, launches = 0;
static size_t asked = 0;

extern "C" {

// Times a kernel's limit was lowered, launches beyond it, launches.
void fake_gr(int* out) {
    out[0] = lowered;
    out[1] = beyond;
    out[2] = launches;
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int v) {
    if (limit.count(f) && v < limit[f]) ++lowered;
    limit[f] = v;
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { return std::memset(d, v, n), cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t bytes, cudaStream_t) { return asked = bytes, 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t* bytes, void*) { return *bytes = asked, cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { return *k = (cudaKernel_t)f, cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t bytes, cudaStream_t) {
    const auto it = limit.find((const void*)k);
    if ((int)bytes > (it == limit.end() ? 48 * 1024 : it->second)) ++beyond;
    ++launches;
    return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
char __cudaInitModule(void**) { return 0; }

}  // extern "C"
