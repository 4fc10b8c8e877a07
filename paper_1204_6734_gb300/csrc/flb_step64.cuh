// flb_step64.cuh -- the FP64 step of one lattice (flb_step64.cu).
#pragma once

#include <cuda_runtime.h>

#include "flb_kernels.cuh"

namespace flb {

// Device tables of the FP64 noise on the current device, built on first use
// and kept until the process exits (25 MB): the Box-Muller radius of each of
// the 2^21 values of u1, and cosine and sine of the first quarter of the 2^21
// angles. Null where there is no memory for them (the kernels then form the same
// numbers themselves).
struct NoiseTables {
    const double* radius = nullptr;
    const double2* circle = nullptr;
};
NoiseTables noise_tables();

constexpr int kRadius = 1 << 21;

// A node's normals from the tables (unit normals of NodeNoise in FP64).
struct TableNoise {
    const NoiseKey& key;
    uint32_t node, step;
    NoiseTables tab;
    __device__ __forceinline__ void operator()(double n[6]) const {
        uint32_t k[6];
        node_fields(key, node, step, k);
        of(tab, k, n);
    }
    static __device__ __forceinline__ void of(const NoiseTables& tab, const uint32_t k[6], double n[6]) {
#pragma unroll
        for (int p = 0; p < 3; ++p)
            bm_pair(__ldg(tab.radius + k[2 * p]), __ldg(tab.circle + (k[2 * p + 1] & (kQuarter - 1))), k[2 * p + 1] >> 19,
                    n + 2 * p);
    }
};

struct Step64Args {
    const double* src;
    double* dst;
    Geometry geo;
    uint32_t step;
    uint32_t node0;     // noise counter of node (0, 0) (slabs: Lx y0)
    int blocks;         // step64_blocks
    double* partials;   // [kSums][blocks] when sampling
    const double* prev; // the previous sampled step's (null: none), added to acc
    double* acc;
    DevError* err;
    const double* lut;  // velocity table (look-up-table f-norm only)
    NoiseTables noise;
    double ref[9];      // c = f^0(rho0, u0), subtracted before sampling
};

// Blocks of the step (one warp each) of a lattice of `nodes` nodes.
int step64_blocks(long long nodes, int sms);
// One step; when sampling it leaves its blocks' partial sums in a.partials and
// adds a.prev to a.acc. step64_flush: a call's last partial sums.
cudaError_t step64(const Step64Args& a, const CollideConst<double>& cc, int basis, bool sample, int sms,
                   cudaStream_t s);
cudaError_t step64_flush(const double* partials, int blocks, double* acc, cudaStream_t s);

}  // namespace flb
