// Stand-ins for the CUDA runtime calls that building a dense model makes, for a
// host program linked without the runtime: allocations are counted and can be
// refused, launches do nothing.
#include <stddef.h>
#include <stdio.h>
#include <stdlib.h>

#include <map>

static std::map<void *, size_t> live;
size_t held = 0;                          // bytes allocated
int allow = -1;                           // allocations that still succeed (-1: all)
bool capturing = false, relaxed = false;  // a capture under way; whether this thread's calls are relaxed

struct Dim3 { unsigned x, y, z; };
enum { kOk = 0, kNoMemory = 2, kCaptureUnsupported = 900, kGlobal = 0, kRelaxed = 2 };

extern "C" {
int cudaMalloc(void **p, size_t n) {
    if (capturing && !relaxed) return kCaptureUnsupported;
    if (allow == 0) return kNoMemory;
    if (allow > 0) allow--;
    *p = malloc(1);
    live[*p] = n;
    held += n;
    return kOk;
}
int cudaFree(void *p) {
    if (!p) return kOk;
    if (!live.count(p)) {
        printf("free of an address that is not held\n");
        exit(1);
    }
    held -= live[p];
    live.erase(p);
    free(p);
    return kOk;
}
int cudaThreadExchangeStreamCaptureMode(int *mode) {
    const int was = relaxed ? kRelaxed : kGlobal;
    relaxed = *mode == kRelaxed;
    *mode = was;
    return kOk;
}
int cudaMemcpy(void *, const void *, size_t, int) { return kOk; }
int cudaGetLastError() { return kOk; }
int cudaFuncSetAttribute(const void *, int, int) { return kOk; }
int cudaLaunchKernel(const void *, Dim3, Dim3, void **, size_t, void *) { return kOk; }
int __cudaLaunchKernel(void *, Dim3, Dim3, void **, size_t, void *) { return kOk; }
int __cudaGetKernel(void **kernel, const void *) {
    *kernel = nullptr;
    return kOk;
}
unsigned __cudaPushCallConfiguration(Dim3, Dim3, size_t, void *) { return 0; }
int __cudaPopCallConfiguration(Dim3 *, Dim3 *, size_t *, void *) { return kOk; }
void **__cudaRegisterFatBinary(void *) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *, void *, int *) {}
char __cudaInitModule(void **) { return 0; }
}
