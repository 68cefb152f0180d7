// A CUDA runtime without a GPU, for tests of the library's host code: allocations are addresses that
// nobody reads, copies to the host bring zeros, everything else succeeds.  Kernel launches of the step
// kernels are recorded by fake_launch.cu.
#include <cstddef>
#include <cstring>

extern "C" {

struct Attributes {  // cudaPointerAttributes
    int type, device;
    void *devicePointer, *hostPointer;
    long reserved[8];
};

void** __cudaRegisterFatBinary(void*) {
    static void* handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(...) { return 0; }
int __cudaPopCallConfiguration(...) { return 0; }
int __cudaGetKernel(void** k, const void* f) {
    *k = const_cast<void*>(f);
    return 0;
}
int __cudaLaunchKernel(...) { return 0; }
int cudaLaunchKernel(...) { return 0; }
int cudaLaunchKernelExC(...) { return 0; }

int cudaDeviceGetAttribute(int* v, int, int) {
    *v = 152;  // the SMs of a GB300: the only attribute that the library reads
    return 0;
}
int cudaGetDevice(int* d) {
    *d = 0;
    return 0;
}
int cudaPointerGetAttributes(void* out, const void*) {
    Attributes* a = static_cast<Attributes*>(out);
    a->type = 2;  // device memory
    a->device = 0;
    a->devicePointer = a->hostPointer = nullptr;
    return 0;
}
static int encode(...) { return 0; }
int cudaGetDriverEntryPointByVersion(const char*, void** p, unsigned, unsigned long long, int* q) {
    *p = reinterpret_cast<void*>(&encode);
    *q = 0;
    return 0;
}
int cudaGetSymbolAddress(void** p, const void*) {
    *p = nullptr;
    return 0;
}
const char* cudaGetErrorString(int) { return "an error of the fake"; }
int cudaGetLastError() { return 0; }
int cudaMemsetAsync(void*, int, size_t, void*) { return 0; }
int cudaMemcpyAsync(void* dst, const void*, size_t n, int kind, void*) {
    if (kind == 2) std::memset(dst, 0, n);
    return 0;
}
int cudaStreamSynchronize(void*) { return 0; }
int cudaStreamBeginCapture(void*, int) { return 0; }
int cudaStreamEndCapture(void*, void** g) {
    *g = nullptr;
    return 0;
}
int cudaGraphInstantiate(void** g, void*, unsigned long long) {
    *g = g;
    return 0;
}
int cudaGraphDestroy(void*) { return 0; }
int cudaGraphExecDestroy(void*) { return 0; }
int cudaGraphLaunch(void*, void*) { return 0; }
int cudaEventCreate(void** e) {
    *e = e;
    return 0;
}
int cudaEventCreateWithFlags(void** e, unsigned) {
    *e = e;
    return 0;
}
int cudaEventDestroy(void*) { return 0; }
int cudaEventRecord(void*, void*) { return 0; }
int cudaEventSynchronize(void*) { return 0; }
int cudaEventElapsedTime(float* ms, void*, void*) {
    *ms = 1.f;
    return 0;
}

}  // extern "C"
