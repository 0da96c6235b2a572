/* The CUDA runtime calls of libmwj's linear joins without a device, for tests that
 * preload this: allocations on the host, launches counted and not run.
 * FAKE_FITS: CTAs of the largest cluster the occupancy query finds room for;
 * FAKE_LAUNCHES: of the largest that a launch is not refused for. */
#include <cuda_runtime_api.h>
#include <stdlib.h>
#include <string.h>

static cudaError_t last = cudaSuccess;
static unsigned cluster[256], n_launches, refused;

static unsigned limit(const char *name) {
    const char *v = getenv(name);
    return v ? (unsigned)atoi(v) : 16u;
}
static unsigned cluster_of(const cudaLaunchConfig_t *c) {
    for (unsigned k = 0; k < c->numAttrs; ++k)
        if (c->attrs[k].id == cudaLaunchAttributeClusterDimension) return c->attrs[k].val.clusterDim.x;
    return 1;
}
/* clusters of the launches so far; returns how many were refused as well */
unsigned fake_launches(unsigned *sizes, unsigned *n) {
    memcpy(sizes, cluster, sizeof(unsigned) * n_launches);
    *n = n_launches;
    return refused;
}

cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **a) {
    const unsigned ctas = cluster_of(c);
    if (ctas > limit("FAKE_LAUNCHES")) {
        ++refused;
        return last = cudaErrorInvalidClusterSize;
    }
    cluster[n_launches++] = ctas;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *f, const cudaLaunchConfig_t *c) {
    *n = cluster_of(c) <= limit("FAKE_FITS");
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int d) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrComputeCapabilityMajor ? 10
         : a == cudaDevAttrComputeCapabilityMinor ? 3 : 232448;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) { *p = malloc(n); return cudaSuccess; }
cudaError_t cudaFree(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemset(void *p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t s) { return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, enum cudaMemcpyKind k) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute a, int v) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned f) { *s = 0; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned f) { *e = 0; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return cudaSuccess; }
