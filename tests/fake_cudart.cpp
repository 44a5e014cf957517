// Stand-ins for the runtime calls of kernels_rebuild.cu's host code: a process with several devices,
// of which fake_device is current, that records the shared-memory limit set for each kernel on each
// device and runs nothing.
#include <cstddef>
#include <cstring>
#include <map>
#include <utility>

int fake_device = 0, fake_refuse = 0;
std::map<std::pair<int, const void*>, int> fake_limit;

extern "C" {
int cudaGetDevice(int* d) { *d = fake_device; return 0; }
int cudaDeviceGetAttribute(int* v, int, int) { *v = 232448; return 0; }
int cudaFuncGetAttributes(void* attr, const void*)
{
    const size_t static_smem = 64;
    std::memcpy(attr, &static_smem, sizeof(size_t));       // the struct's first member
    return 0;
}
int cudaFuncSetAttribute(const void* f, int, int bytes)
{
    if (fake_refuse) return 1;                             // cudaErrorInvalidValue
    fake_limit[{fake_device, f}] = bytes;
    return 0;
}
int cudaGetLastError() { return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = 1; return 0; }
int __cudaGetKernel(void**, const void*) { return 0; }
int __cudaLaunchKernel(...) { return 0; }
int __cudaPopCallConfiguration(...) { return 0; }
int __cudaPushCallConfiguration(...) { return 0; }
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
char __cudaInitModule(void**) { return 0; }
void __cudaRegisterFunction(...) {}
void __cudaUnregisterFatBinary(void**) {}
}
