/* A CUDA runtime that computes nothing, for the host paths of libls.so: preloaded, it takes the
 * place of the calls that set-up, factorisation and release make.  Device memory is host memory; the
 * allocation of number fail_at fails as the runtime's does, leaving its error to be read. */
#include <stdlib.h>
#include <string.h>

static int last, fail_at = -1, calls, live;

void fake_fail_at(int k) {
    fail_at = k;
    calls = 0;
}
int fake_live(void) { return live; }

int cudaGetLastError(void) {
    const int e = last;
    last = 0;
    return e;
}
int cudaPeekAtLastError(void) { return last; }
const char* cudaGetErrorString(int e) { return e == 2 ? "out of memory" : "error"; }

int cudaMalloc(void** p, size_t n) {
    if (calls++ == fail_at) return last = 2;
    *p = calloc(1, n ? n : 1);
    ++live;
    return 0;
}
int cudaHostAlloc(void** p, size_t n, unsigned flags) { return cudaMalloc(p, n); }
int cudaFree(void* p) {
    live -= p != NULL;
    free(p);
    return 0;
}
int cudaFreeHost(void* p) { return cudaFree(p); }

static int copy(void* d, const void* s, size_t n) {
    memcpy(d, s, n);
    return 0;
}
int cudaMemcpyAsync(void* d, const void* s, size_t n, int kind, void* st) { return copy(d, s, n); }
int cudaMemcpy(void* d, const void* s, size_t n, int kind) { return copy(d, s, n); }
int cudaMemsetAsync(void* d, int v, size_t n, void* st) {
    memset(d, v, n);
    return 0;
}

int cudaGetDevice(int* d) { return *d = 0; }
int cudaDeviceGetAttribute(int* v, int a, int d) {
    *v = 152;
    return 0;
}
int cudaFuncSetAttribute(const void* f, int a, int v) { return 0; }
int cudaStreamCreateWithFlags(void** s, unsigned f) {
    *s = NULL;
    return 0;
}
int cudaStreamDestroy(void* s) { return 0; }
int cudaStreamSynchronize(void* s) { return 0; }
int cudaEventCreate(void** e) {
    *e = NULL;
    return 0;
}
int cudaEventCreateWithFlags(void** e, unsigned f) { return cudaEventCreate(e); }
int cudaEventDestroy(void* e) { return 0; }

/* launches (grids, blocks and argument lists are not looked at) */
int cudaLaunchKernelExC(const void* cfg, const void* f, void** args) { return 0; }
int __cudaLaunchKernel(void* k, ...) { return 0; }
int __cudaGetKernel(void** k, const void* f) {
    *k = NULL;
    return 0;
}
unsigned __cudaPushCallConfiguration(void) { return 0; }
int __cudaPopCallConfiguration(void* g, void* b, size_t* s, void* st) { return 0; }
