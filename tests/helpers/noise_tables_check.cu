// Test helper: the FP64 normals from the library's tables against those that the
// kernels form where there are no tables (flb_step64.cu, flb_device.cuh), over every
// radius and every angle; returns the number of pairs that differ in any bit, or
// -1 for a CUDA error or missing tables.
#include "../../paper_1204_6734_gb300/csrc/flb_step64.cu"

namespace {

__global__ void compare_kernel(flb::NoiseTables tab, int* differ) {
    const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x, m = (1u << 21) - 1u;
    // radii k, k + 1, k + 2 with angles that are permutations of k
    const uint32_t f[6] = {k, (k * 5u + 1u) & m, (k + 1u) & m, (k * 1664525u + 3u) & m, (k + 2u) & m, m - k};
    double a[6], b[6];
    flb::TableNoise::of(tab, f, a);
    flb::box_muller(f, b);
    for (int q = 0; q < 6; ++q)
        if (__double_as_longlong(a[q]) != __double_as_longlong(b[q])) atomicAdd(differ, 1);
}

}  // namespace

extern "C" long long noise_tables_differ() {
    int* d = nullptr;
    int n = -1;
    if (cudaMalloc(&d, sizeof(int)) != cudaSuccess) return -1;
    const flb::NoiseTables tab = flb::noise_tables();
    if (!tab.radius) return -1;
    if (cudaMemset(d, 0, sizeof(int)) != cudaSuccess) return -1;
    compare_kernel<<<(1 << 21) / 256, 256>>>(tab, d);
    if (cudaMemcpy(&n, d, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return -1;
    cudaFree(d);
    return n;
}
