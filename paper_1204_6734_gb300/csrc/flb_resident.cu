// flb_resident.cu -- host side of the resident kernel for one lattice: how a
// lattice is cut into blocks, and the launch.
#include <cuda_runtime.h>

#include <algorithm>

#include "flb_resident.cuh"

namespace flb {

namespace {

const void* kernel_of(int basis, bool sample) {
    if (basis == 0) return sample ? (const void*)resident_kernel<0, kResStaged> : (const void*)resident_kernel<0, kResQuiet>;
    if (basis == 1) return sample ? (const void*)resident_kernel<1, kResStaged> : (const void*)resident_kernel<1, kResQuiet>;
    return sample ? (const void*)resident_kernel<2, kResStaged> : (const void*)resident_kernel<2, kResQuiet>;
}

// Estimated microseconds of a step (f-norm, no sampling): wp warp passes of 64
// nodes on the four schedulers of an SM; blocks that exchange add their words'
// trip through L2 and the passes whose lanes move them (a row on the edge; all
// rows are edges twice where a block has one; a cut across x puts two edge
// lanes into every row). Measured: 21 x 21 in one block 1.8, in two 2.1; 64 x 64
// in 1 / 4 / 16 / 64 blocks 11.1 / 3.4 / 2.0 / 2.7; 300 x 130 in 26 / 44 / 65 /
// 130 blocks 5.2 / 3.7 / 3.5 / 4.1; 512 x 512 in 128 x 1 7.0, 2 x 74 7.1, 8 x 19
// 7.9; 4000 x 20 in 1 / 2 / 4 / 7 x 20 20.0 / 10.5 / 5.7 / 4.9; 1000 x 750 in
// 150 x 1 16.4, 2 x 75 22.4. Sampling adds 0.4 (21 x 21) to 2.7 (1000 x 750).
}  // namespace

double resident_step_us(int wp, int gx, int gy, int bw, int bh) {
    double t = std::max(1.75, 0.69 * ((wp + 3) / 4) + 0.3);
    if (gy > 1) t += 0.3 + 0.072 * bw / 32.0 + (bh == 1 ? 1.2 : 0.0);   // one row: two waits in a row
    if (gx > 1) t += 1.0 + 0.08 * std::min(wp, bh);
    return t;
}

namespace {

// The same for one launch per step, from the measured 6.2 (up to 300 x 130),
// 8.2 (400 x 300), 10.3 (512 x 512), 19.8 (1000 x 750), 20.8 (900 x 900);
// sampled 2 to 4 more.
double one_step_us(double nodes) { return 6.2 + nodes / 55e3; }
}  // namespace

ResidentPlan resident_plan(int Lx, int Ly, int sms, bool cut) {
    ResidentPlan best;
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
            const size_t t = res_smem_bytes((int)cells, kResStaged, swarps);
            if (q > kResSmemMax) continue;
            const double c = resident_step_us(wp, gx, gy, bw, bh);
            if (c >= cost) continue;
            cost = c;
            best.gx = gx;
            best.gy = gy;
            best.threads[0] = warps * 32;
            best.threads[1] = swarps * 32;
            best.smem[0] = q;
            best.smem[1] = t <= kResSmemMax ? t : 0;
            best.mail_words = res_mail_words(Lx, Ly, gx, gy);
        }
    }
    if (cost > one_step_us((double)Lx * Ly)) best = ResidentPlan();
    return best;
}

cudaError_t resident_prepare(const ResidentPlan& p, int basis) {
    cudaError_t ce = cudaSuccess;
    for (int smp = 0; smp < 2 && ce == cudaSuccess; ++smp)
        if (p.smem[smp])
            ce = cudaFuncSetAttribute(kernel_of(basis, smp), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResSmemMax);
    return ce;
}

cudaError_t resident_step(const ResidentPlan& p, const ResidentArgs& a, const CollideConst<float>& cc, int basis,
                          bool sample, cudaStream_t s) {
    void* params[2] = {(void*)&a, (void*)&cc};
    const void* fn = kernel_of(basis, sample);
    const dim3 grid(p.gx * p.gy), block(p.threads[sample]);
    // blocks that wait for one another have to be on the GPU together
    if (p.gx * p.gy > 1) return cudaLaunchCooperativeKernel(fn, grid, block, params, p.smem[sample], s);
    return cudaLaunchKernel(fn, grid, block, params, p.smem[sample], s);
}

}  // namespace flb
