// flb_basis.cuh -- the weights of the f-norm at a velocity, in FP64: f_i^0(1, u),
// used where the velocity table of the look-up-table f-norm is built.
#pragma once

#include "flb_collide.cuh"

namespace flb {

__device__ __forceinline__ void feq_unit_fp64(double ux, double uy, double W[9]) {
    const double usq = ux * ux + uy * uy;
    for (int i = 0; i < 9; ++i) {
        const double uv = ux * cvx(i) + uy * cvy(i);
        const double wi = i == 0 ? 4.0 / 9.0 : (i <= 4 ? 1.0 / 9.0 : 1.0 / 36.0);
        W[i] = wi * (1.0 + 3.0 * uv + 4.5 * uv * uv - 1.5 * usq);
    }
}

}  // namespace flb
