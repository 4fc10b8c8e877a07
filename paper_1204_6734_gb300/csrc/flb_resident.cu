// flb_resident.cu -- host side of the resident kernel for one lattice: how a
// lattice is cut into blocks, and the launch.
#include <cuda_runtime.h>

#include <algorithm>

#include "flb_host.h"
#include "flb_resident.cuh"

namespace flb {

namespace {

template <class Par, int SAMPLE>
const void* kernel_of(int basis, bool sample) {
    if (basis == 0)
        return sample ? (const void*)resident_kernel<0, SAMPLE, Par> : (const void*)resident_kernel<0, kResQuiet, Par>;
    if (basis == 1)
        return sample ? (const void*)resident_kernel<1, SAMPLE, Par> : (const void*)resident_kernel<1, kResQuiet, Par>;
    return sample ? (const void*)resident_kernel<2, SAMPLE, Par> : (const void*)resident_kernel<2, kResQuiet, Par>;
}

const void* kernel_of(int basis, bool half, bool sample) {
    return half ? kernel_of<LatticePar16, kResExact>(basis, sample) : kernel_of<LatticePar, kResStaged>(basis, sample);
}

}  // namespace

// Estimated microseconds of a step (f-norm, no sampling): wp warp passes of 64
// nodes on the four schedulers of an SM; blocks that exchange add their words'
// trip through L2 and the passes whose lanes move them (a row on the edge; a
// block of one row waits at both). A cut across x puts edge lanes into every
// row, and a warp waits at one edge after the other: blocks of five rows and more
// lose 9 us, and narrow ones 1.4 us in every pass of a scheduler that holds an edge.
// Measured: 21 x 21 in one block 1.6; 64 x 64 in 1 / 4 / 16 / 64 blocks 11.1 / 3.4 /
// 2.0 / 2.7; 300 x 130 in 26 / 44 / 65 / 130 blocks 5.2 / 3.7 / 3.4 / 4.1, in 2 x 65 4.7,
// 3 x 43 7.1; 626 x 62 in 1 x 62 4.7, 2 x 62 4.4, 2 x 31 5.5, 7 x 21 7.3; 4000 x 20 in
// 2 / 4 / 7 x 20 10.5 / 5.7 / 5.0; 512 x 512 in 128 blocks 6.5; 593 x 1269 in 141 15.1; 1000 x
// 750 in 150 15.0 (large blocks come out up to a tenth faster than estimated).
// Sampled, across x: 5000 x 100 in 152 x 1 28.9, 3000 x 150 in 75 x 2 23.4, 1648 x 176 in
// 50 x 3 17.3, 2923 x 132 in 38 x 4 16.0, 1147 x 319 in 36 x 4 22.3 and in 10 x 15 16.7 (one
// launch per step: 16.2, 14.6, 12.4, 14.4, 14.3).
double resident_step_us(int wp, int gx, int gy, int bw, int bh) {
    const int passes = (wp + 3) / 4;
    double t = std::max(1.75, 0.69 * passes + 0.3);
    if (gy > 1) t += 0.3 + 0.072 * bw / 32.0 + (bh == 1 ? 1.2 : 0.0);   // one row: two waits in a row
    if (gx > 1)
        t += std::max(bh == 1 ? 0.3 : bh == 2 ? 2.3 : bh < 5 ? 5.0 : 9.0, 1.4 * passes * std::min(1.0, 40.0 / bw));
    return t;
}

// us per step without / with sampling, this kernel and one launch per step: f-norm
// 21 x 21 1.6 / 2.1 and 4.0 / 6.7, 300 x 130 3.3 / 4.0 and 4.0 / 8.1, 400 x 300 4.0 / 4.8
// and 6.4 / 10.2, 512 x 512 6.5 / 7.7 and 8.5 / 12.2, 700 x 600 8.9 / 10.4 and 10.3 / 14.3,
// 1000 x 750 15.0 / 17.5 and 17.9 / 20.8, 900 x 900 16.3 / 19.0 and 19.4 / 22.9; the Hermite
// norm 300 x 130 2.6 / 3.1 and 2.8 / 7.3, 512 x 512 4.6 / 5.4 and 5.9 / 10.0, 900 x 900 10.9 /
// 13.0 and 14.4 / 17.0; the FP16 store 300 x 130 3.3 / 4.2 and 3.2 / 5.1, 512 x 512 6.6 / 9.1
// and 8.3 / 10.8, 700 x 600 9.0 / 11.8 and 10.8 / 14.4. Of 90 shapes drawn up to 1.15
// million nodes, in the f-norm and the Hermite norm, five took longer here: 1066 x 153,
// sampled, by 8 %, and four without sampling in the Hermite norm (about 3 us) by 2 to 17 %.
bool resident_pays(const ResidentPlan& p, double nodes, bool half, bool sample) {
    if (!p.gx || !p.smem[sample]) return false;
    const double us = half ? 1.05 * p.us : p.us, rest = nodes / 54e3;
    return sample ? 1.12 * us + 0.3 < (half ? 5.9 : 7.9) + rest : us + 0.6 < (half ? 3.4 : 4.0) + rest;
}

ResidentPlan resident_plan(int Lx, int Ly, int sms, bool cut, bool half) {
    ResidentPlan best;
    if (36LL * Lx * Ly > (long long)(cut ? sms : 1) * (long long)kResSmemMax) return best;
    double cost = 1e30;
    const int gxmax = cut ? std::min(Lx, sms) : 1;
    for (int gx = 1; gx <= gxmax; ++gx) {
        const int gymax = cut ? std::min(Ly, sms / gx) : 1;
        for (int gy = 1; gy <= gymax; ++gy) {
            const int bw = (Lx + gx - 1) / gx, bh = (Ly + gy - 1) / gy;
            const long long cells = (long long)bw * bh;
            if (cells > 16384 || (gx > 1 && bw < 32)) continue;   // narrow blocks: scattered loads
            const int wp = (int)(((cells + 1) / 2 + 31) / 32);   // warp passes per step
            const int warps = std::min(kResMaxWarps, wp);
            // sampling: three more warps, if there is room, for the reduction
            const int swarps = std::min(kResMaxWarps, wp + 3);
            const size_t q = res_smem_bytes((int)cells, kResQuiet, warps);
            const size_t t = res_smem_bytes((int)cells, half ? kResExact : kResStaged, swarps);
            if (q > kResSmemMax) continue;
            const double c = resident_step_us(wp, gx, gy, bw, bh);
            if (c >= cost) continue;
            cost = c;
            best.us = c;
            best.gx = gx;
            best.gy = gy;
            best.threads[0] = warps * 32;
            best.threads[1] = swarps * 32;
            best.smem[0] = q;
            best.smem[1] = t <= kResSmemMax ? t : 0;
            best.mail_words = res_mail_words(Lx, Ly, gx, gy);
        }
    }
    return best;
}

cudaError_t resident_prepare(const ResidentPlan& p, int basis, bool half) {
    cudaError_t ce = cudaSuccess;
    for (int smp = 0; smp < 2 && ce == cudaSuccess; ++smp)
        if (p.smem[smp])
            ce = allow_smem(kernel_of(basis, half, smp), kResSmemMax);
    return ce;
}

cudaError_t resident_step(const ResidentPlan& p, const ResidentArgs& a, const CollideConst<float>& cc, int basis,
                          bool half, bool sample, cudaStream_t s) {
    void* params[2] = {(void*)&a, (void*)&cc};
    const void* fn = kernel_of(basis, half, sample);
    const dim3 grid(p.gx * p.gy), block(p.threads[sample]);
    // blocks that wait for one another have to be on the GPU together
    if (p.gx * p.gy > 1) return cudaLaunchCooperativeKernel(fn, grid, block, params, p.smem[sample], s);
    return cudaLaunchKernel(fn, grid, block, params, p.smem[sample], s);
}

}  // namespace flb
