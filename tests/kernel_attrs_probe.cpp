// Test harness: the library's shared-memory opt-in (ensure_kernel_attrs in qldpc_host.cpp) against fakes of the three CUDA
// calls it makes.  Prints one "set device bytes" line for each attribute set and one "rc value" line for each call.
#include <cuda_runtime.h>

#include <cstdio>

static int g_device = 0;
static cudaError_t fake_get_device(int *d)
{
    *d = g_device;
    return cudaSuccess;
}
static cudaError_t fake_get_attributes(cudaFuncAttributes *a, const void *)
{
    a->sharedSizeBytes = 1024;
    return cudaSuccess;
}
static cudaError_t fake_set_attribute(const void *, cudaFuncAttribute, int bytes)
{
    std::printf("set %d %d\n", g_device, bytes);
    return cudaSuccess;
}
#define cudaGetDevice fake_get_device
#define cudaFuncGetAttributes fake_get_attributes
#define cudaFuncSetAttribute fake_set_attribute
#define main layout_main
#include "host_layout_probe.cpp"
#undef main

int main()
{
    const int kernel = 0;
    const struct {
        int device;
        size_t bytes;
    } calls[] = {{0, 40000}, {0, 60000}, {0, 60000}, {1, 60000}, {1, 50000}, {0, 70000}, {1, 65000}, {0, 65000}, {1, 70000}};
    for (const auto &c : calls) {
        g_device = c.device;
        std::printf("rc %d\n", qldpc::detail::ensure_kernel_attrs(&kernel, c.bytes, 232448));
    }
    return 0;
}
