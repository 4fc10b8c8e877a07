// flb_step_fp16.cu -- the pipelined fused step with the FP16 deviation store.
//
// The state is kept as h_i = (f_i - c_i) / sqrt(kT) in FP16, with c = f^0(rho0,
// u0) in FP32: the thermal deviations are O(sqrt(kT f^0)), so h is O(1) and
// FP16's 11-bit significand resolves it to about 2.4e-4 of a standard
// deviation. A buffer then holds 18 bytes per node instead of 36 (36 bytes per
// node and step moved instead of 72). The collision itself is the FP32 one of
// flb_collide.cuh: each node decodes f = c + sqrt(kT) h, collides in packed
// FP32x2, and encodes h* = (f* - c) / sqrt(kT) with round-to-nearest.
//
// Structure as in flb_step_tma.cu: persistent CTAs, 128 x NW/2 tiles, 2D TMA
// boxes into a ring of shared-memory stages, NW = 16 (8 on small lattices)
// colliding warps with two nodes per thread, the last warp to release a stage
// refilling it. Boxes start 8 columns left of the tile (a TMA box of 16-bit
// elements must start at a multiple of 8 elements) and are 144 wide.
//
// Correlation sums with FP32 products by the colliding warps (flb_gram.cuh) of the
// deviations sqrt(kT) h, rounded to FP32. (Squares of h itself, exact in FP32, end in
// one of few bit patterns, and their sums rounded to nearest came out 3e-8 to 8e-8
// too small.) Sampler warps (4 beside 8 colliding warps) formed the same products in
// FP32 registers: 94.4 us per step at 2000 x 1500, f-norm, against 65.4 here; on the
// tensor cores they took 63.8, 4.7e-8 of <df df> lost to their cut-off.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "flb_collide.cuh"
#include "flb_gram.cuh"
#include "flb_host.h"
#include "flb_internal.h"
#include "flb_pipeline.cuh"
#include "flb_tma.cuh"

namespace flb {

namespace {

constexpr int kHBoxW = kTW + 16;   // x0 - 8 .. x0 + 135
constexpr int kHOff = 8;           // column of x0 in a box

// NW colliding warps, 128 x NW/2 tiles.
template <int NW>
struct HShape {
    static constexpr int TH = NW / 2;              // rows per tile
    static constexpr int SPLANE = TH * kHBoxW;     // halves per plane box
    static constexpr int STAGE = 9 * SPLANE;       // halves per stage (10.4 / 20.7 KB)
    static constexpr int STAGES = NW == 8 ? 16 : 9;
    static constexpr size_t smem_bytes() {
        return sizeof(__half) * (size_t)STAGES * STAGE + 2 * STAGES * sizeof(uint64_t) + sizeof(double) * 64 +
               sizeof(float) * (size_t)NW * kProdWarpFloats;
    }
    static_assert((SPLANE * sizeof(__half)) % 128 == 0, "plane boxes stay 128-byte aligned");
    static_assert((NW & (NW - 1)) == 0, "release counts wrap at 2^32");
};
static_assert(HShape<8>::smem_bytes() <= 227 * 1024 && HShape<16>::smem_bytes() <= 227 * 1024, "shared memory");

template <int NW>
__device__ __forceinline__ void issue_tile16(__half* smem, const CUtensorMap* map, const HArgs& a, int t, int s,
                                             uint64_t* full) {
    using HS = HShape<NW>;
    mbar_arrive_expect_tx(&full[s], 9u * HS::TH * kHBoxW * sizeof(__half));
    const int ty = t / a.tiles_x, x0 = (t - ty * a.tiles_x) * kTW, y0 = ty * HS::TH;
    __half* st = smem + s * HS::STAGE;
#pragma unroll
    for (int i = 0; i < 9; ++i)
        tma_load_2d(st + i * HS::SPLANE, map, x0 + kXO - kHOff, i * (a.geo.Ly + 2) + y0 + 1 - cvy(i), &full[s]);
}

template <int BASIS, bool SAMPLE, int NW>
__global__ void __launch_bounds__(NW * 32, 1)
step_fp16_kernel(const __grid_constant__ CUtensorMap map, const HArgs a, const CollideConst<float> cc) {
    using HS = HShape<NW>;
    constexpr int S = HS::STAGES, TH = HS::TH;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __half* smem = reinterpret_cast<__half*>(smem_raw);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + S * HS::STAGE);
    uint32_t* released = reinterpret_cast<uint32_t*>(full + S);   // releases of each stage
    double* red = reinterpret_cast<double*>(full + 2 * S);        // FP64 sums (kProdEntries)
    float* staged = reinterpret_cast<float*>(red + 64);

    const int c = threadIdx.x, warp = c >> 5, lane_id = c & 31;
    allow_dependents();
    if (c == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], 1);
            released[s] = 0u;
        }
        fence_mbar_init();
    }
    if constexpr (SAMPLE) {
        if (c < kProdEntries) red[c] = 0.0;
        prod_init(staged + warp * kProdWarpFloats);
    }
    __syncthreads();
    wait_dependency();
    const int Lx = a.geo.Lx, Ly = a.geo.Ly;

    // thread 0 issues the first tiles; after that the last warp to release a
    // stage refills it
    if (c == 0) {
        prefetch_tensormap(&map);
        for (int j = 0, t = blockIdx.x; j < S && t < a.ntiles; ++j, t += gridDim.x)
            issue_tile16<NW>(smem, &map, a, t, j, full);
    }
    const int ty = c >> 6, r = c & 63;
    const ProdLane gblk(SAMPLE ? smem_u32(staged + warp * kProdWarpFloats) : 0u);
    float gc[SAMPLE ? 8 : 1];
    if constexpr (SAMPLE) {
#pragma unroll
        for (int q = 0; q < 8; ++q) gc[q] = 0.f;
    }
    int k = 0, s = 0, n = 0, gtiles = 0;   // tile count, its stage and the stage's use
    bool timed_out = false;
    for (int t = blockIdx.x; t < a.ntiles; t += gridDim.x, ++k) {
        if (!mbar_wait(&full[s], n & 1)) {
            record_error(a.err, kStatusTimeout, -1, a.step);
            timed_out = true;
            break;
        }
        const __half* st = smem + s * HS::STAGE + ty * kHBoxW + kHOff + r;
        auto raw = [&](__half2* h) {   // this thread's nodes A and B, as stored
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const __half* p = st + i * HS::SPLANE - cvx(i);
                h[i] = __halves2half2(p[0], p[64]);
            }
        };
        f2 g[9];
        {
            __half2 h[9];
            raw(h);
#pragma unroll
            for (int i = 0; i < 9; ++i) g[i] = mad(f2(__half22float2(h[i])), f2(a.scale), f2(a.ref[i]));
        }
        const int tty = t / a.tiles_x, x0 = (t - tty * a.tiles_x) * kTW, y0 = tty * TH, y = y0 + ty;
        const int xA = x0 + r, xB = xA + 64;
        const bool inA = xA < Lx && y < Ly, inB = xB < Lx && y < Ly;
        const bool whole = x0 + kTW <= Lx && y0 + TH <= Ly;   // every node of the tile
        auto refetch = [&](f2* gg) {
            __half2 h[9];
            raw(h);
            f2 v[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                v[i] = f2(__half22float2(h[i]));
                gg[i] = mad(v[i], f2(a.scale), f2(a.ref[i]));
            }
            if constexpr (SAMPLE) {
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    v[i] = v[i] * f2(a.scale);
                    if (!whole) v[i] = f2(inA ? v[i].v.x : 0.f, inB ? v[i].v.y : 0.f);
                }
                prod_stage(gblk, v);
            }
        };
        const uint32_t nodeA = a.node0 + (uint32_t)xA + (uint32_t)Lx * (uint32_t)y;
        f2 f[9];
        const uint32_t stt = collide_basis<f2, BASIS>(g, PairNoise{cc.key, nodeA, nodeA + 64u, a.step}, refetch, a.lut,
                                                      cc, f);
        if constexpr (SAMPLE) {
            prod_sums(gblk, reinterpret_cast<float(&)[8]>(gc));
            if (++gtiles == kGramFlushTiles) {
                prod_flush(reinterpret_cast<float(&)[8]>(gc), red);
                gtiles = 0;
            }
        }
        // the NW-th release of this use of the stage refills it with the CTA's
        // tile S later
        __syncwarp();
        if (lane_id == 0 && ((release_count(&released[s]) + 1u) & (NW - 1)) == 0) {
            const int tn = t + S * gridDim.x;
            if (tn < a.ntiles) {
                fence_proxy_async_smem();
                issue_tile16<NW>(smem, &map, a, tn, s, full);
            }
        }
        if (stt) {
            if (inA && (stt & 0xFF)) record_error(a.err, (int)(stt & 0xFF), nodeA, a.step);
            if (inB && (stt >> 8)) record_error(a.err, (int)(stt >> 8), nodeA + 64u, a.step);
        }
        // h* = (f* - c) / sqrt(kT) = f* inv_scale + nref
        __half hA[9], hB[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const f2 h = mad(f[i], f2(a.inv_scale), f2(a.nref[i]));
            hA[i] = __float2half_rn(h.v.x);
            hB[i] = __float2half_rn(h.v.y);
        }
        __half* pa = a.dst + at(a.geo, 0, xA, y);
        if (x0 > 0 && y0 > 0 && x0 + kTW < Lx && y0 + TH < Ly) {
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                pa[i * a.geo.plane] = hA[i];
                pa[i * a.geo.plane + 64] = hB[i];
            }
        } else {
            if (inA) store_node_ghosts(pa, a.geo, xA, y, hA);
            if (inB) store_node_ghosts(pa + 64, a.geo, xB, y, hB);
        }
        if (++s == S) {
            s = 0;
            ++n;
        }
    }
    if (timed_out && lane_id == 0) {
        // copies this warp did not consume may still be in flight: wait (with
        // the bound of every wait) for the next S tiles
        for (int j = k; j < k + S && blockIdx.x + j * gridDim.x < a.ntiles; ++j)
            if (!mbar_wait(&full[j % S], (j / S) & 1)) break;
    }
    if constexpr (SAMPLE) {
        prod_flush(reinterpret_cast<float(&)[8]>(gc), red);
        __syncthreads();
        if (c < kSums) atomicAdd(&a.acc[c], prod_sum(red, c, 1.0));
    }
}

template <int NW>
const void* fp16_kernel(int basis, bool sample) {
    if (basis == 0)
        return sample ? (const void*)step_fp16_kernel<0, true, NW> : (const void*)step_fp16_kernel<0, false, NW>;
    if (basis == 1)
        return sample ? (const void*)step_fp16_kernel<1, true, NW> : (const void*)step_fp16_kernel<1, false, NW>;
    return sample ? (const void*)step_fp16_kernel<2, true, NW> : (const void*)step_fp16_kernel<2, false, NW>;
}

const void* fp16_kernel(int nw, int basis, bool sample) {
    return nw == 8 ? fp16_kernel<8>(basis, sample) : fp16_kernel<16>(basis, sample);
}

}  // namespace

cudaError_t fp16_plan(TmaPlan* plan, void* buf0, void* buf1, const Geometry& g) {
    plan->ready = false;
    int dev = 0, sms = 0;
    cudaError_t ce = cudaGetDevice(&dev);
    if (ce == cudaSuccess) ce = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (ce != cudaSuccess) return ce;
    // 16 warps where every SM gets several tiles of theirs, else 8
    const int tiles_x = (g.Lx + kTW - 1) / kTW;
    const int nw = (long long)tiles_x * ((g.Ly + 7) / 8) >= 4LL * sms ? 16 : 8, th = nw / 2;
    void* bufs[2] = {buf0, buf1};
    for (int b = 0; b < 2; ++b) {
        const cudaError_t e = tma_encode_planes(&plan->map[b], bufs[b], g, kHBoxW, th, 2);
        if (e != cudaSuccess) return e;
    }
    const size_t smem = nw == 8 ? HShape<8>::smem_bytes() : HShape<16>::smem_bytes();
    for (int basis = 0; basis < 3 && ce == cudaSuccess; ++basis)
        for (int smp = 0; smp < 2 && ce == cudaSuccess; ++smp)
            ce = allow_smem(fp16_kernel(nw, basis, smp), smem);
    if (ce != cudaSuccess) return ce;
    plan->nw = nw;
    plan->smem = smem;
    plan->tiles_x = tiles_x;
    plan->ntiles = tiles_x * ((g.Ly + th - 1) / th);
    plan->grid = sms < plan->ntiles ? sms : plan->ntiles;
    if (plan->grid < 1) plan->grid = 1;
    plan->ready = true;
    return cudaSuccess;
}

cudaError_t fp16_step(const TmaPlan& plan, int src, const HArgs& a, const CollideConst<float>& cc,
                      int basis, bool sample, cudaStream_t s) {
    if (!plan.ready) return cudaErrorInvalidValue;
    HArgs args = a;
    args.tiles_x = plan.tiles_x;
    args.ntiles = plan.ntiles;
    void* params[3] = {(void*)&plan.map[src], (void*)&args, (void*)&cc};
    return launch_dependent(fp16_kernel(plan.nw, basis, sample), dim3(plan.grid), dim3(plan.nw * 32), params, plan.smem,
                            s);
}

}  // namespace flb
