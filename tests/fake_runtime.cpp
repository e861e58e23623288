// A stand-in for the CUDA runtime that records launches, linked with the library's own
// objects by tests/test_launches.py: what the host side launches, where, and what
// it does when a device refuses, without a GPU.  Kernels do not run; device memory
// is host memory.
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <sstream>
#include <string>
#include <utility>

#include <cuda_runtime_api.h>

namespace {

int device = 0;
std::map<const void *, std::string> names;                // host stub -> mangled kernel name
std::set<std::pair<int, const void *>> clusters_allowed;  // (device, kernel): non-portable cluster sizes
std::ostringstream launches;
std::string text;

struct Pending {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
} pending;

void record(const void *f, dim3 grid, dim3 block, unsigned cluster) {
    launches << device << ' ' << names[f] << ' ' << grid.x * grid.y << ' ' << block.x << ' ' << cluster << '\n';
}

unsigned cluster_of(const cudaLaunchConfig_t *c) {
    for (unsigned i = 0; i < c->numAttrs; i++)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) return c->attrs[i].val.clusterDim.x;
    return 1;
}

bool refused(const void *f, unsigned cluster) { return cluster > 8 && !clusters_allowed.count({device, f}); }

}  // namespace

extern "C" {

void fake_device(int d) { device = d; }
const char *fake_launches() {  // "device kernel blocks threads cluster" a line, since the last call
    text = launches.str();
    launches.str("");
    return text.c_str();
}

void **__cudaRegisterFatBinary(void *) { return reinterpret_cast<void **>(&device); }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *f, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *) {
    names[f] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t stream) {
    pending = {grid, block, smem, stream};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *stream) {
    *grid = pending.grid;
    *block = pending.block;
    *smem = pending.smem;
    *static_cast<cudaStream_t *>(stream) = pending.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void *>(f));
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void **, size_t, cudaStream_t) {
    record(k, grid, block, 1);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void *f, dim3 grid, dim3 block, void **, size_t, cudaStream_t) {
    record(f, grid, block, 1);
    return cudaSuccess;
}
cudaError_t cudaLaunchCooperativeKernel(const void *f, dim3 grid, dim3 block, void **, size_t, cudaStream_t) {
    record(f, grid, block, 1);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) {
    const unsigned cluster = cluster_of(c);
    if (refused(f, cluster)) return cudaErrorInvalidClusterSize;
    record(f, c->gridDim, c->blockDim, cluster);
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *f, const cudaLaunchConfig_t *c) {
    *n = refused(f, cluster_of(c)) ? 0 : 1;
    return *n ? cudaSuccess : cudaErrorInvalidClusterSize;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v) {
    if (a == cudaFuncAttributeNonPortableClusterSizeAllowed && v) clusters_allowed.insert({device, f});
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) {
    std::memset(a, 0, sizeof(*a));
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) {
    *d = device;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 227 * 1024;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *) {
    static void *block = std::calloc(1, 16u << 20);
    *p = block;
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) {
    std::memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *to, const void *from, size_t n, cudaMemcpyKind, cudaStream_t) {
    std::memcpy(to, from, n);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }

}  // extern "C"
