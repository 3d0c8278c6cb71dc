/* CUDA runtime calls that fail on request, for tests of error paths: preloaded
 * (LD_PRELOAD) into a child process, where the library's calls come here first.
 * fake_malloc: cudaMalloc answers "out of memory".  fake_group: launches of blocks that
 * wait for one another (cooperative, or one cluster) are refused as too large. */
#define _GNU_SOURCE
#include <cuda_runtime_api.h>
#include <dlfcn.h>

int fake_malloc, fake_group;

static void *real(const char *name) {
    void *lib = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
    return lib ? dlsym(lib, name) : 0;
}

/* (An impossible size: the runtime answers "out of memory" itself and keeps the error
 * for cudaGetLastError.) */
cudaError_t cudaMalloc(void **p, size_t n) {
    cudaError_t (*f)(void **, size_t) = real("cudaMalloc");
    return f(p, fake_malloc ? (size_t)1 << 60 : n);
}

cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *fn, void **args) {
    for (unsigned k = 0; fake_group && k < c->numAttrs; ++k)
        if (c->attrs[k].id == cudaLaunchAttributeCooperative ||
            c->attrs[k].id == cudaLaunchAttributeClusterDimension)
        {
            void *p;
            cudaError_t (*m)(void **, size_t) = real("cudaMalloc");
            m(&p, (size_t)1 << 60); /* leaves an error behind, as the launch would */
            return cudaErrorCooperativeLaunchTooLarge;
        }
    cudaError_t (*f)(const cudaLaunchConfig_t *, const void *, void **) = real("cudaLaunchKernelExC");
    return f(c, fn, args);
}
