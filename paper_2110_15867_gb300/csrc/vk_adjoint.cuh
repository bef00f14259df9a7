// vk_adjoint.cuh -- the limited curvature with its partials, for the reverse sweeps (adjoint.cu,
// adjoint_tile.cu).
#pragma once

#include "vk_common.cuh"

namespace vk {

// minmod of (4 d0 - d1, 4 d1 - d0, d0, d1) with its partials ka = dr/dd0 and kb = dr/dd1 (the
// selected argument's; 0 where the minmod is 0)
template <typename C> __device__ __forceinline__ C dm4_coef(C d0, C d1, C &ka, C &kb)
{
    const C a = C(4) * d0 - d1, b = C(4) * d1 - d0;
    const C lo = mn2(mn3(a, b, d0), d1), hi = mx2(mx3(a, b, d0), d1);
    const C r = mn2(mx2(lo, C(0)), hi);
    const bool z = r == C(0), ia = r == a, ib = r == b, i0 = r == d0;
    ka = z ? C(0) : ia ? C(4) : ib ? C(-1) : i0 ? C(1) : C(0);
    kb = z ? C(0) : ia ? C(-1) : ib ? C(4) : i0 ? C(0) : C(1);
    return r;
}

} // namespace vk
