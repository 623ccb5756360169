/* Fakes of CUDA runtime calls that fail, loaded ahead of the runtime (LD_PRELOAD); every other call passes through.
 * fake_malloc_limit: cudaMalloc answers out of memory above this many bytes. */
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>

size_t fake_malloc_limit = (size_t)-1;
int fake_refused = 0;

static void* next(const char* name) {
    void* h = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
    return h ? dlsym(h, name) : dlsym(RTLD_NEXT, name);
}

int cudaMalloc(void** p, size_t n) {
    static int (*real)(void**, size_t);
    if (!real) real = (int (*)(void**, size_t))next("cudaMalloc");
    if (n > fake_malloc_limit) {
        ++fake_refused;
        return 2; /* cudaErrorMemoryAllocation */
    }
    return real(p, n);
}
