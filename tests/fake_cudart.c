/* Fakes of CUDA runtime calls that fail, loaded ahead of the runtime (LD_PRELOAD); every other call passes through.
 * fake_malloc_limit: cudaMalloc answers out of memory above this many bytes.  fake_drop: kernels whose name holds
 * this text are not launched (the call reports success). */
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
#include <string.h>

size_t fake_malloc_limit = (size_t)-1;
int fake_refused = 0;
char fake_drop[64] = "";
int fake_dropped = 0;

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

int cudaLaunchKernelExC(const void* config, const void* func, void** args) {
    static int (*real)(const void*, const void*, void**);
    static int (*name_of)(const char**, const void*);
    if (!real) real = (int (*)(const void*, const void*, void**))next("cudaLaunchKernelExC");
    if (!name_of) name_of = (int (*)(const char**, const void*))next("cudaFuncGetName");
    const char* name = NULL;
    if (fake_drop[0] && name_of && name_of(&name, func) == 0 && name && strstr(name, fake_drop)) {
        ++fake_dropped;
        return 0;
    }
    return real(config, func, args);
}
