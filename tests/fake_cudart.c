/* CUDA runtime stand-in for tests of the library's host logic without a GPU: device memory is host
 * memory, streams and events are empty handles, and launches do nothing (the library counts them
 * itself).  fake_fail_malloc(k) makes the k-th cudaMalloc from now fail, once. */
#include <stddef.h>
#include <stdint.h>
#include <stdlib.h>

#define API __attribute__((visibility("default")))

static long fail_in = 0, live = 0;
API void fake_fail_malloc(long k) { fail_in = k; }
API long fake_fail_left(void) { return fail_in; }
API long fake_live(void) { return live; }

static char handle;

API int cudaMalloc(void** p, size_t n) {
    if (fail_in > 0 && --fail_in == 0) return 2;   /* cudaErrorMemoryAllocation */
    *p = malloc(n ? n : 1);
    if (!*p) return 2;
    ++live;
    return 0;
}
API int cudaFree(void* p) {
    if (p) --live;
    free(p);
    return 0;
}
API int cudaMemcpy(void* d, const void* s, size_t n, int k) { return 0; }
API int cudaMemcpyAsync(void* d, const void* s, size_t n, int k, void* st) { return 0; }
API int cudaMemset(void* d, int v, size_t n) { return 0; }
API int cudaDeviceGetAttribute(int* v, int a, int dev) { *v = 152; return 0; }
API int cudaDeviceGetStreamPriorityRange(int* lo, int* hi) { *lo = 0; *hi = -5; return 0; }
API int cudaDeviceSynchronize(void) { return 0; }
API int cudaGetDevice(int* d) { *d = 0; return 0; }
API int cudaGetLastError(void) { return 0; }
API const char* cudaGetErrorString(int e) { return "fake"; }
API int cudaGetSymbolAddress(void** p, const void* s) { *p = &handle; return 0; }
API int cudaFuncSetAttribute(const void* f, int a, int v) { return 0; }
API int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int t, size_t sm, unsigned fl) {
    *n = 1;
    return 0;
}
API int cudaEventCreate(void** e) { *e = &handle; return 0; }
API int cudaEventCreateWithFlags(void** e, unsigned f) { *e = &handle; return 0; }
API int cudaEventDestroy(void* e) { return 0; }
API int cudaEventElapsedTime(float* ms, void* a, void* b) { *ms = 0.f; return 0; }
API int cudaEventRecord(void* e, void* s) { return 0; }
API int cudaEventSynchronize(void* e) { return 0; }
API int cudaStreamCreateWithFlags(void** s, unsigned f) { *s = &handle; return 0; }
API int cudaStreamCreateWithPriority(void** s, unsigned f, int p) { *s = &handle; return 0; }
API int cudaStreamDestroy(void* s) { return 0; }
API int cudaStreamSynchronize(void* s) { return 0; }
API int cudaStreamWaitEvent(void* s, void* e, unsigned f) { return 0; }
API int cudaStreamGetCaptureInfo(void* s, int* status, unsigned long long* id, void* g, void* d, void* e, size_t* n) {
    *status = 0;
    return 0;
}
API int cudaLaunchKernelExC(const void* cfg, const void* f, void** args) { return 0; }
API int __cudaLaunchKernel() { return 0; }
API int __cudaGetKernel(void** k, const void* f) { *k = &handle; return 0; }
API int __cudaPopCallConfiguration() { return 0; }
API void** __cudaRegisterFatBinary(void* f) {
    static void* h = &handle;
    return &h;
}
API void __cudaRegisterFatBinaryEnd(void** h) {}
API void __cudaRegisterFunction() {}
API void __cudaRegisterVar() {}
API void __cudaUnregisterFatBinary(void** h) {}
