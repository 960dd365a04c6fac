/* Preloaded into a child process by the tests: stands between the library and the CUDA
 * runtime.  SPI_SHIM_LIMIT: cudaMalloc fails (out of memory) once the live allocations would
 * exceed that many bytes, as on a device of that size; SPI_SHIM_REDZONE: so many bytes (a multiple
 * of 256) of NaN patterns before and behind every allocation, checked when it is freed;
 * SPI_SHIM_LOG: a file that receives the name of every kernel launched, a line per overwritten
 * red zone, and at exit the peak of the live allocations and the number of red zones checked. */
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdio.h>
#include <stdlib.h>

#define MAXP 65536
static void* ptr[MAXP];
static size_t len[MAXP];
static size_t live, peak, zones;

/* the runtime's own function (the library's dependency, loaded by then: not in the global scope) */
static void* runtime(const char* f) {
    void* h = dlopen("libcudart.so.13", RTLD_NOW | RTLD_NOLOAD);
    void* p = h ? dlsym(h, f) : 0;
    if (!p) {
        fprintf(stderr, "cuda_shim: no %s\n", f);
        exit(3);
    }
    return p;
}
static FILE* out(void) {
    static FILE* f;
    const char* p = getenv("SPI_SHIM_LOG");
    if (!f && p) f = fopen(p, "a");
    return f;
}
static size_t redzone(void) {
    const char* p = getenv("SPI_SHIM_REDZONE");
    return p ? (size_t)strtoull(p, 0, 10) : 0;
}
static int fill(void* p, size_t n) {
    static int (*set)(void*, int, size_t);
    if (!set) set = (int (*)(void*, int, size_t))runtime("cudaMemset");
    return n ? set(p, 0xff, n) : 0;
}
static void check(const char* side, const char* p, size_t n, size_t size) {
    static int (*copy)(void*, const void*, size_t, int);
    if (!copy) copy = (int (*)(void*, const void*, size_t, int))runtime("cudaMemcpy");
    unsigned char* h = malloc(n);
    if (copy(h, p, n, 2 /* device to host */) == 0) {
        ++zones;
        for (size_t i = 0; i < n; ++i)
            if (h[i] != 0xff) {
                if (out()) fprintf(out(), "overwritten %s %zu bytes at %zu\n", side, size, i);
                break;
            }
    }
    free(h);
}
int cudaMalloc(void** p, size_t n) {
    static int (*real)(void**, size_t);
    if (!real) real = (int (*)(void**, size_t))runtime("cudaMalloc");
    const char* lim = getenv("SPI_SHIM_LIMIT");
    const size_t z = redzone();
    if (lim && live + n > (size_t)strtoull(lim, 0, 10)) return 2; /* cudaErrorMemoryAllocation */
    int e = real(p, n + 2 * z);
    if (e == 0 && z) {
        e = fill(*p, z);
        if (e == 0) e = fill((char*)*p + z + n, z);
        *p = (char*)*p + z;
    }
    for (int i = 0; e == 0 && i < MAXP; ++i)
        if (!ptr[i]) {
            ptr[i] = *p;
            len[i] = n;
            live += n;
            if (live > peak) peak = live;
            break;
        }
    return e;
}
int cudaFree(void* p) {
    static int (*real)(void*);
    if (!real) real = (int (*)(void*))runtime("cudaFree");
    const size_t z = redzone();
    for (int i = 0; p && i < MAXP; ++i)
        if (ptr[i] == p) {
            ptr[i] = 0;
            live -= len[i];
            if (z) {
                check("before", (char*)p - z, z, len[i]);
                check("behind", (char*)p + len[i], z, len[i]);
                p = (char*)p - z;
            }
            break;
        }
    return real(p);
}
static void log_name(const char* name) {
    if (out() && name) fprintf(out(), "kernel %s\n", name);
}
typedef struct { unsigned x, y, z; } dim;
int __cudaLaunchKernel(void* k, dim g, dim b, void** a, size_t s, void* st) {
    static int (*real)(void*, dim, dim, void**, size_t, void*);
    static int (*name)(const char**, void*);
    const char* nm = 0;
    if (!real) real = (int (*)(void*, dim, dim, void**, size_t, void*))runtime("__cudaLaunchKernel");
    if (!name) {
        void* h = dlopen("libcuda.so.1", RTLD_NOW);
        name = h ? (int (*)(const char**, void*))dlsym(h, "cuKernelGetName") : 0;
    }
    if (name) name(&nm, k);
    log_name(nm);
    return real(k, g, b, a, s, st);
}
int cudaLaunchKernelExC(const void* cfg, const void* func, void** args) {
    static int (*real)(const void*, const void*, void**);
    static int (*name)(const char**, const void*);
    const char* nm = 0;
    if (!real) real = (int (*)(const void*, const void*, void**))runtime("cudaLaunchKernelExC");
    if (!name) name = (int (*)(const char**, const void*))runtime("cudaFuncGetName");
    if (name) name(&nm, func);
    log_name(nm);
    return real(cfg, func, args);
}
__attribute__((destructor)) static void report(void) {
    if (out()) {
        fprintf(out(), "peak %zu\nzones %zu\n", peak, zones);
        fflush(out());
    }
}
