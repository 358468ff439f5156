// The host side of csrc/chol_cluster.cu against a stand-in for the CUDA
// runtime with three devices: the object that the library's build makes is
// linked with the functions below instead of libcudart and the rest of the
// library.  Like the runtime, the stand-in keeps function attributes per device
// and refuses a cluster of more than 8 CTAs on a device where the kernel's
// attribute was not set; device 2 places no 16-CTA cluster.  Prints one line per
// call: device, variant (16-byte rows or not), status, CTAs of the cluster.
#include "kernels.cuh"

#include <cstdarg>
#include <cstdio>
#include <set>
#include <utility>

static int g_device = 0, g_cluster = 0;
static std::set<std::pair<int, const void *>> g_allowed;

namespace realq {
realq_status_t fail(realq_status_t s, const char *, ...) { return s; }
realq_status_t check_launch(const char *) { return REALQ_OK; }
realq_status_t set_smem_limit(const void *, int) { return REALQ_OK; }
Launch::Launch(const char *n, cudaStream_t s) : name(n), stream(s), slot(-1) {}
Launch::~Launch() {}
}  // namespace realq

extern "C" {
// (registration of the object's kernels, which are never run)
void **__cudaRegisterFatBinary(void *) {
    static void *handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *, void *, int *) {}
unsigned __cudaPopCallConfiguration(void *, void *, void *, void *) { return 1; }
cudaError_t __cudaGetKernel(void **k, const void *f) {
    *k = const_cast<void *>(f);
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(void *, dim3, dim3, void **, size_t, cudaStream_t) { return cudaErrorNotSupported; }

cudaError_t cudaGetDevice(int *dev) {
    *dev = g_device;
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "stand-in"; }
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v) {
    if (a == cudaFuncAttributeNonPortableClusterSizeAllowed && v) g_allowed.insert({g_device, f});
    return cudaSuccess;
}
static int cluster_of(const cudaLaunchConfig_t *c) {
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) return (int)c->attrs[i].val.clusterDim.x;
    return 1;
}
static cudaError_t placed(const cudaLaunchConfig_t *c, const void *f) {
    if (cluster_of(c) > 8 && !g_allowed.count({g_device, f})) return cudaErrorInvalidClusterSize;
    if (cluster_of(c) > 8 && g_device == 2) return cudaErrorLaunchOutOfResources;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *f, const cudaLaunchConfig_t *c) {
    *n = placed(c, f) == cudaSuccess;
    return *n || g_device == 2 ? cudaSuccess : cudaErrorInvalidClusterSize;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) {
    g_cluster = cluster_of(c);
    return placed(c, f);
}
}

int main() {
    float *a = reinterpret_cast<float *>(4096);
    for (int pass = 0; pass < 2; ++pass)
        for (int dev = 0; dev < 3; ++dev)
            for (int vec = 0; vec < 2; ++vec) {
                g_device = dev;
                g_cluster = 0;
                const int st = realq::chol_inv_block(nullptr, vec ? 200 : 201, a, 200, 0, nullptr);
                std::printf("%d %d %d %d\n", dev, vec, st, g_cluster);
            }
    return 0;
}
