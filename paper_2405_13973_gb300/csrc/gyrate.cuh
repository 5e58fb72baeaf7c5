// gyrate.cuh -- the exact gyration U0(h) (Eq. U0, B along +z: clockwise
// velocity rotation) as a literal sequence of IEEE operations: the rounded
// intrinsics keep it free of contraction in every translation unit.
#pragma once
#include "internal.h"

namespace pt {

__device__ __forceinline__ void gyrate(const PushParams& pp, double& x, double& y, double& z,
                                       double& vx, double& vy, double vz) {
    const double ux = vx, uy = vy, c1 = __dsub_rn(1.0, pp.C);
    x = __dadd_rn(x, __ddiv_rn(__dadd_rn(__dmul_rn(ux, pp.S), __dmul_rn(uy, c1)), pp.wc));
    y = __dadd_rn(y, __ddiv_rn(__dsub_rn(__dmul_rn(uy, pp.S), __dmul_rn(ux, c1)), pp.wc));
    z = __dadd_rn(z, __dmul_rn(vz, pp.h));
    vx = __dadd_rn(__dmul_rn(ux, pp.C), __dmul_rn(uy, pp.S));
    vy = __dadd_rn(__dmul_rn(-ux, pp.S), __dmul_rn(uy, pp.C));
}

}  // namespace pt
