// flb_host.h -- host-side helpers shared by the C-ABI translation units:
// parameter validation, the reference equilibrium, the collision constants,
// grid sizing of the plain element-wise kernels and error-code mapping.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <cmath>
#include <mutex>
#include <vector>

#include "../../include/flb.h"
#include "flb_device.cuh"
#include "flb_kernels.cuh"

namespace flb {

// The current context's number, unique for the life of the program: what is set
// once per context is set again after a reset of the device. 0: unknown.
inline unsigned long long context_id() {
    using GetId = CUresult (*)(CUcontext, unsigned long long*);
    static const GetId get = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            p = nullptr;
        }
        return reinterpret_cast<GetId>(p);
    }();
    unsigned long long id = 0;
    return get && get(nullptr, &id) == CUDA_SUCCESS ? id : 0;
}

// Raise a kernel's dynamic shared memory limit in the current context to `bytes`,
// unless an earlier call has: creating a lattice asked the runtime two dozen
// times, about a third of the 230 us it took.
inline cudaError_t allow_smem(const void* fn, size_t bytes) {
    struct Done {
        unsigned long long ctx;
        const void* fn;
        size_t bytes;
    };
    static std::mutex mutex;
    static std::vector<Done> done;
    const unsigned long long ctx = context_id();
    if (!ctx) return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    std::lock_guard<std::mutex> lock(mutex);
    Done* mine = nullptr;
    for (Done& d : done)
        if (d.ctx == ctx && d.fn == fn) mine = &d;
    if (mine && mine->bytes >= bytes) return cudaSuccess;
    const cudaError_t ce = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (ce != cudaSuccess) return ce;
    try {
        if (mine)
            mine->bytes = bytes;
        else
            done.push_back({ctx, fn, bytes});
    } catch (const std::bad_alloc&) {   // asked again next time
    }
    return cudaSuccess;
}

// f_i^0(rho, u) of Eq. d2q9f0.
inline void feq_host(double rho, double ux, double uy, double f[9]) {
    const double usq = ux * ux + uy * uy;
    for (int i = 0; i < 9; ++i) {
        const double uv = ux * cvx(i) + uy * cvy(i);
        const double wi = i == 0 ? 4.0 / 9.0 : (i <= 4 ? 1.0 / 9.0 : 1.0 / 36.0);
        f[i] = rho * wi * (1.0 + 3.0 * uv + 4.5 * uv * uv - 1.5 * usq);
    }
}

// 1 if p describes a lattice flb_create accepts.
inline int valid_params(const flb_params* p) {
    if (!p) return 0;
    if (p->Lx < 1 || p->Ly < 1) return 0;
    if ((long long)p->Lx * p->Ly >= (1LL << 31)) return 0;
    if (!(p->rho0 > 0) || !std::isfinite(p->rho0)) return 0;
    if (!(p->kT >= 0) || !std::isfinite(p->kT)) return 0;
    if (!std::isfinite(p->ux0) || !std::isfinite(p->uy0)) return 0;
    for (int a = 3; a < 9; ++a)
        if (!(p->omega[a] > 0 && p->omega[a] < 2)) return 0;
    if (p->basis != FLB_BASIS_STANDARD && p->basis != FLB_BASIS_LOCAL &&
        p->basis != FLB_BASIS_LOCAL_LUT)
        return 0;
    if (p->precision != FLB_FP64 && p->precision != FLB_FP32 && p->precision != FLB_FP16_DEV)
        return 0;
    if (p->precision == FLB_FP16_DEV && !(p->kT > 0)) return 0;   // the store scale is sqrt(kT)
    if (p->reserved != 0) return 0;
    // the mean velocity must leave every f_i^0(1,u0) > 0 (Fig. 11)
    const double usq = p->ux0 * p->ux0 + p->uy0 * p->uy0;
    for (int i = 0; i < 9; ++i) {
        const double uv = p->ux0 * cvx(i) + p->uy0 * cvy(i);
        if (!(1.0 + 3.0 * uv + 4.5 * uv * uv - 1.5 * usq > 0.0)) return 0;
    }
    return 1;
}

// -omega_a and the noise amplitudes sqrt(kT omega_a (2 - omega_a)), a = 3..8.
template <class T>
CollideConst<T> collide_const(const flb_params* p) {
    CollideConst<T> cc;
    for (int a = 0; a < 6; ++a) {
        const double om = p->omega[3 + a];
        cc.nomega[a] = (T)(-om);
        const double v = p->kT * om * (2.0 - om);
        cc.amp[a] = (T)(v > 0 ? std::sqrt(v) : 0.0);
    }
    cc.key = make_noise_key(p->seed, p->replica);
    return cc;
}

// Scale s of the tensor-core correlation sums (the nodes are staged as
// (f - f^0(rho0, u0)) / s in FP16): s = sqrt(kT rho0) makes the thermal
// fluctuations of order one. Used only where a deviation as large as a few
// rho0 stays far inside FP16's range (|d| / s <= 4 sqrt(rho0 / kT) <= 16000);
// otherwise, and at kT = 0, the sums are taken with FP32 products.
inline bool tensor_sampling_ok(const flb_params* p) {
    return p->kT > 0 && std::sqrt(p->rho0 / p->kT) <= 4000.0;
}
inline double gram_scale(const flb_params* p) { return std::sqrt(p->kT * p->rho0); }

// Allocate need + extra bytes or, where they cannot be had, need; *got_extra tells
// which. alloc(&p, bytes): cudaMalloc.
template <class Alloc>
cudaError_t alloc_with_extra(Alloc&& alloc, void** p, size_t need, size_t extra, bool* got_extra) {
    *p = nullptr;
    *got_extra = true;
    cudaError_t ce = alloc(p, need + extra);
    if (ce != cudaSuccess && extra > 0) {
        *p = nullptr;
        *got_extra = false;
        ce = alloc(p, need);
    }
    return ce;
}
// cudaMalloc, its error not left behind.
inline cudaError_t device_alloc(void** p, size_t bytes) {
    const cudaError_t ce = cudaMalloc(p, bytes);
    if (ce != cudaSuccess) cudaGetLastError();
    return ce;
}

// Steps of [ta, tb) that the schedule (warmup, every) samples. No sum of times
// passes tb or warmup, so any `every` up to 2^63 - 1 will do.
inline int64_t count_sampled(int64_t ta, int64_t tb, int64_t warmup, int64_t every) {
    if (every <= 0) return 0;
    const int64_t lo = ta > warmup ? ta : warmup;
    if (lo >= tb) return 0;
    const int64_t past = (lo - warmup) % every, skip = past ? every - past : 0;
    return skip < tb - lo ? (tb - 1 - lo - skip) / every + 1 : 0;
}

// The device address of page-locked host memory, or null for other memory:
// the state I/O kernels then read or write the caller's host array themselves
// (one pass over the host link, no device staging buffer).
inline double* pinned_view(const void* host) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, host) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return a.type == cudaMemoryTypeHost ? static_cast<double*>(a.devicePointer) : nullptr;
}

inline int grid_for(long long n) {
    long long b = (n + 255) / 256;
    if (b > 4096) b = 4096;
    return (int)(b < 1 ? 1 : b);
}

inline int map_status(int code) {
    if (code == kStatusInvalidVelocity) return FLB_ERR_INVALID_VELOCITY;
    if (code == kStatusNonfinite) return FLB_ERR_NONFINITE;
    if (code == kStatusTimeout) return FLB_ERR_TIMEOUT;
    return code ? FLB_ERR_STATE : FLB_OK;
}

}  // namespace flb
