// Fakes of CUDA runtime (and libm) calls, linked in front of the library's objects with
// --wrap, for failures that no argument of the public entry points brings about:
//
//   fake_attribute_changes()  how often a kernel's shared-memory limit was set to
//                             another value than before
//   fake_copied_bytes()       bytes copied from host memory so far
//   fake_long_sines()         calls of the long double sine, cosine (or both) so far
//   fake_cluster_limit(c)     the device has no room for clusters of more than c
//                             CTAs: the query answers 0, a launch fails
//   fake_cluster_fails(on)    the launch of a cluster fails
#include <cuda_runtime.h>

#include <map>
#include <mutex>

namespace {
std::mutex lock;
std::map<const void*, int> limit;
size_t copied = 0, long_sines = 0;
int changes = 0, cluster_limit = 1 << 30, cluster_fails = 0;

int cluster_of(const cudaLaunchConfig_t* c) {
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension)
            return (int)c->attrs[i].val.clusterDim.x;
    return 0;
}
}  // namespace

extern "C" {
int fake_attribute_changes() {
    std::lock_guard<std::mutex> g(lock);
    return changes;
}
size_t fake_copied_bytes() {
    std::lock_guard<std::mutex> g(lock);
    return copied;
}
size_t fake_long_sines() { return long_sines; }
void fake_cluster_limit(int c) { cluster_limit = c; }
void fake_cluster_fails(int on) { cluster_fails = on; }

cudaError_t __real_cudaFuncSetAttribute(const void*, cudaFuncAttribute, int);
cudaError_t __wrap_cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
        std::lock_guard<std::mutex> g(lock);
        const auto it = limit.find(f);
        if (it != limit.end() && it->second != v) ++changes;
        limit[f] = v;
    }
    return __real_cudaFuncSetAttribute(f, a, v);
}

long double __real_sinl(long double);
long double __real_cosl(long double);
void __real_sincosl(long double, long double*, long double*);
long double __wrap_sinl(long double x) {
    ++long_sines;
    return __real_sinl(x);
}
long double __wrap_cosl(long double x) {
    ++long_sines;
    return __real_cosl(x);
}
void __wrap_sincosl(long double x, long double* s, long double* c) {
    ++long_sines;
    __real_sincosl(x, s, c);
}

cudaError_t __real_cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t);
cudaError_t __wrap_cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k,
                                   cudaStream_t st) {
    if (k == cudaMemcpyHostToDevice) {
        std::lock_guard<std::mutex> g(lock);
        copied += n;
    }
    return __real_cudaMemcpyAsync(d, s, n, k, st);
}

cudaError_t __real_cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**);
cudaError_t __wrap_cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
    const int n = cluster_of(c);
    if (n > cluster_limit || (n > 0 && cluster_fails)) return cudaErrorLaunchOutOfResources;
    return __real_cudaLaunchKernelExC(c, f, args);
}

cudaError_t __real_cudaOccupancyMaxActiveClusters(int*, const void*, const cudaLaunchConfig_t*);
cudaError_t __wrap_cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t* c) {
    if (cluster_of(c) > cluster_limit) {
        *n = 0;
        return cudaSuccess;
    }
    return __real_cudaOccupancyMaxActiveClusters(n, f, c);
}
}
