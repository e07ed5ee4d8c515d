/* Preloaded before the CUDA runtime library: passes cudaMalloc on, except that
 * once `allowed` requests have passed the next ones ask for 2^50 bytes, which
 * the runtime refuses.  allowed < 0: none is changed. */
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>

long allowed = -1;
long refused = 0;

int cudaMalloc(void** p, size_t bytes) {
    static int (*pass_on)(void**, size_t);
    if (!pass_on) { /* the runtime library the caller has loaded, whatever its scope */
        void* runtime = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
        if (runtime) pass_on = (int (*)(void**, size_t))dlsym(runtime, "cudaMalloc");
        if (!pass_on) return 999; /* cudaErrorUnknown */
    }
    if (allowed == 0) {
        ++refused;
        return pass_on(p, (size_t)1 << 50);
    }
    if (allowed > 0) --allowed;
    return pass_on(p, bytes);
}
