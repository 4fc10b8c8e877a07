// flb_step64.cu -- the FP64 step of one lattice: one node per thread, one warp
// per block, pulled, sampled, collided and stored.
//
// Bound: the FP64 pipe (two lanes a cycle and SM). The collision and the sums
// are about 450 FP64 operations per node; the noise by functions, six divided
// square roots and the block's reduction by shuffles would be another 600; so:
//  * Normals by table. A draw has 21-bit fields: the radius sqrt(-2 ln u1) has
//    2^21 values, cosine and sine 2^19 up to signs and their exchange. Both come
//    from tables in L2 (16.8 and 8.4 MB; three 8-byte and three 16-byte reads
//    per node), computed once by the functions that would be called for every
//    node (bm_radius and bm_circle, flb_device.cuh: three logarithms, square
//    roots and sine-cosine pairs); without tables they are.
//  * 1 / sqrt(pivot) as rsqrt (flb_vec.cuh).
//  * The 54 sums of a warp by folding: in every round a lane keeps half of its
//    values and adds its partner's share of them, 62 additions in place of 270.
//  * One warp per block, so that a small lattice spreads over the SMs: 32 x 32
//    ran on 4 of 152 SMs as blocks of 256.
// f-norm, sampled, us per step before and after: 32 x 32 75.8 / 16.4, 400 x 300
// 282.7 / 131.9 (457 FP64 instructions per node, the pipe 83 % busy).
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>
#include <new>
#include <vector>

#include "flb_host.h"
#include "flb_step64.cuh"
#include "flb_tma.cuh"

namespace flb {

namespace {

// Entry k of the radius table is that of the field k; entry j of the circle that of
// the angle 2 pi j 2^-21.
__global__ void noise_tables_kernel(double* radius, double2* circle) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < kRadius) radius[k] = bm_radius(k);
    if (k < kQuarter) circle[k] = bm_circle(k);
}

// The warp's totals of s[0..53]: lane l gets sums 2 l and 2 l + 1.
__device__ __forceinline__ double2 fold_sums(const double (&s)[kSums]) {
    const int lane = threadIdx.x & 31;
    double v[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        const double hi = k + 32 < kSums ? s[k + 32 < kSums ? k + 32 : 0] : 0.0;
        const bool up = lane & 16;
        v[k] = (up ? hi : s[k]) + __shfl_xor_sync(0xffffffffu, up ? s[k] : hi, 16);
    }
#pragma unroll
    for (int h = 16, m = 8; h >= 2; h >>= 1, m >>= 1) {
        const bool up = lane & m;
#pragma unroll
        for (int k = 0; k < h; ++k) v[k] = (up ? v[k + h] : v[k]) + __shfl_xor_sync(0xffffffffu, up ? v[k] : v[k + h], m);
    }
    return make_double2(v[0], v[1]);
}

// acc[q] += the sum over blocks of partials[q][b], in a fixed order; one warp.
__device__ __forceinline__ void add_partials(const double* partials, int nblocks, double* acc, int q) {
    const double* p = partials + (size_t)q * nblocks;
    double v = 0.0;
#pragma unroll 8
    for (int b = threadIdx.x & 31; b < nblocks; b += 32) v += __ldcg(p + b);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) acc[q] += v;
}

// The sums of node g, added to s.
__device__ __forceinline__ void add_node(double (&s)[kSums], const double (&g)[9], const double (&ref)[9]) {
    double d[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) d[i] = g[i] - ref[i];
    int k = 9;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        s[i] += d[i];
#pragma unroll
        for (int j = i; j < 9; ++j) s[k++] += d[i] * d[j];
    }
}

// Blocks 0..a.blocks-1 step the nodes; when sampling, kSums further blocks add
// the previous step's partial sums (a.prev) to acc meanwhile, in place of a
// launch of their own after every step. SPLIT: a second warp of the block takes
// the sums of the nodes that the first one collides.
template <int BASIS, bool SAMPLE, bool TABLE, bool SPLIT>
__global__ void __launch_bounds__(SPLIT ? 64 : 32) step64_kernel(const Step64Args a, const CollideConst<double> cc) {
    allow_dependents();
    wait_dependency();
    if (SAMPLE && (int)blockIdx.x >= a.blocks) {
        if (a.prev && threadIdx.x < 32) add_partials(a.prev, a.blocks, a.acc, blockIdx.x - a.blocks);
        return;
    }
    const int Lx = a.geo.Lx, N = Lx * a.geo.Ly;   // N < 2^31 (checked at creation)
    const int lane = threadIdx.x & 31;
    const bool sums = SAMPLE && (!SPLIT || threadIdx.x >= 32), collides = !SPLIT || threadIdx.x < 32;
    double s[SAMPLE ? kSums : 1];
    if constexpr (SAMPLE) {
#pragma unroll
        for (int k = 0; k < kSums; ++k) s[k] = 0.0;
    }
    for (long long m = (long long)blockIdx.x * 32 + lane; m < N; m += (long long)a.blocks * 32) {
        const int n = (int)m, y = n / Lx, x = n - y * Lx;
        double g[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) g[i] = a.src[pull_at(a.geo, i, x, y)];
        if constexpr (SAMPLE) {
            if (sums) add_node(reinterpret_cast<double(&)[kSums]>(s), g, a.ref);
        }
        if (!collides) continue;
        double f[9];
        const uint32_t node = a.node0 + (uint32_t)n;
        auto again = [&](double* gg) {
#pragma unroll
            for (int i = 0; i < 9; ++i) gg[i] = g[i];
        };
        uint32_t st;
        if constexpr (TABLE)
            st = collide_basis<double, BASIS>(g, TableNoise{cc.key, node, a.step, a.noise}, again, a.lut, cc, f);
        else
            st = collide_basis<double, BASIS>(g, NodeNoise{cc.key, node, a.step}, again, a.lut, cc, f);
        if (st != kStatusOk) record_error(a.err, (int)(st & 0xFF), (long long)a.node0 + n, a.step);
        store_node(a.dst, a.geo, x, y, f);
    }
    if constexpr (SAMPLE) {
        if (!sums) return;
        const double2 t = fold_sums(reinterpret_cast<const double(&)[kSums]>(s));
        if (2 * lane < kSums) {
            a.partials[(size_t)(2 * lane) * a.blocks + blockIdx.x] = t.x;
            a.partials[(size_t)(2 * lane + 1) * a.blocks + blockIdx.x] = t.y;
        }
    }
}

// The last step's partial sums of a call.
__global__ void __launch_bounds__(32) add_partials_kernel(const double* partials, int nblocks, double* acc) {
    add_partials(partials, nblocks, acc, blockIdx.x);
}

std::mutex g_mutex;
struct ContextTables {
    unsigned long long ctx;
    NoiseTables tables;
};
std::vector<ContextTables> g_tables;

template <int BASIS, bool SAMPLE, bool SPLIT>
cudaError_t launch(const Step64Args& a, const CollideConst<double>& cc, cudaStream_t s) {
    const int grid = a.blocks + (SAMPLE ? kSums : 0), threads = SPLIT ? 64 : 32;
    const void* fn = a.noise.radius ? (const void*)step64_kernel<BASIS, SAMPLE, true, SPLIT>
                                    : (const void*)step64_kernel<BASIS, SAMPLE, false, SPLIT>;
    void* params[2] = {(void*)&a, (void*)&cc};
    return launch_dependent(fn, dim3(grid), dim3(threads), params, 0, s);
}

template <int BASIS>
cudaError_t launch(const Step64Args& a, const CollideConst<double>& cc, bool sample, bool split, cudaStream_t s) {
    return !sample ? launch<BASIS, false, false>(a, cc, s)
           : split ? launch<BASIS, true, true>(a, cc, s)
                   : launch<BASIS, true, false>(a, cc, s);
}

}  // namespace

NoiseTables noise_tables() {
    const unsigned long long ctx = context_id();
    if (!ctx) return NoiseTables();   // the kernel then forms the normals itself
    std::lock_guard<std::mutex> lock(g_mutex);
    for (const ContextTables& c : g_tables)
        if (c.ctx == ctx) return c.tables;
    NoiseTables t;
    void* p = nullptr;
    if (cudaMalloc(&p, sizeof(double) * kRadius + sizeof(double2) * kQuarter) != cudaSuccess) {
        cudaGetLastError();
        return NoiseTables();
    }
    double2* circle = (double2*)p;
    double* radius = (double*)(circle + kQuarter);
    // on a stream of its own, then waited for (once per context)
    cudaStream_t s;
    cudaError_t ce = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    if (ce == cudaSuccess) {
        noise_tables_kernel<<<kRadius / 128, 128, 0, s>>>(radius, circle);
        ce = cudaGetLastError();
        const cudaError_t e2 = cudaStreamSynchronize(s);
        if (ce == cudaSuccess) ce = e2;
        cudaStreamDestroy(s);
    }
    if (ce != cudaSuccess) {
        cudaGetLastError();
        cudaFree(p);
        return NoiseTables();
    }
    t.radius = radius;
    t.circle = circle;
    try {
        g_tables.push_back({ctx, t});
    } catch (const std::bad_alloc&) {
        cudaFree(p);
        return NoiseTables();
    }
    return t;
}

// About 16 blocks per SM, each with the same number of nodes per lane; fewer
// nodes than that: one per lane. (The reduction at a block's end costs a
// seventh of a node; with more blocks than about 12 per SM the last ones to
// finish leave SMs idle for less than a tenth of the step.)
int step64_blocks(long long nodes, int sms) {
    const long long warps = (nodes + 31) / 32, want = 16LL * (sms > 0 ? sms : 1);
    const long long per = std::max<long long>(1, (warps + want / 2) / want);
    return (int)std::max<long long>(1, (warps + per - 1) / per);
}

cudaError_t step64(const Step64Args& a, const CollideConst<double>& cc, int basis, bool sample, int sms,
                   cudaStream_t s) {
    // up to two blocks per SM the step takes as long as one warp's chain of
    // operations, which the sums then leave (32 x 32: 24.6 -> 16.4 us per step,
    // the launch that added the sums gone as well); with more blocks the FP64
    // pipe is busy either way (400 x 300: 83 %)
    const bool split = a.blocks <= 2 * sms;
    return basis == 0   ? launch<0>(a, cc, sample, split, s)
           : basis == 1 ? launch<1>(a, cc, sample, split, s)
                        : launch<2>(a, cc, sample, split, s);
}

cudaError_t step64_flush(const double* partials, int blocks, double* acc, cudaStream_t s) {
    add_partials_kernel<<<kSums, 32, 0, s>>>(partials, blocks, acc);
    return cudaGetLastError();
}

}  // namespace flb
