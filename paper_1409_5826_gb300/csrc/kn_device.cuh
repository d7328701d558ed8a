// kn_device.cuh -- device helpers shared by the integrator kernels: timers and
// approximate exponentials, TwoSum, the FP32 pieces of the QSS update.
#pragma once

#include "kn_internal.h"

namespace kn {

__device__ __forceinline__ long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return (long long)t;
}

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Knuth's TwoSum (TAOCP vol. 2, 4.2.2): s = fl(a + b) and the exact rounding
// error e = (a + b) - s, for any a, b (no ordering condition).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bv = __fsub_rn(s, a);
    const float av = __fsub_rn(s, bv);
    e = __fadd_rn(__fsub_rn(a, av), __fsub_rn(b, bv));
}

// Warps of a group that hold species (species i goes to lane i mod G): a warp
// whose first lane is at or past N has none, skips the update and its
// reductions, and is left out of the combine.
__device__ __forceinline__ int species_warps(const PlanDev& P) { return (min(P.G, P.N) + 31) >> 5; }

// FP32 versions for the mixed form.  In powers of r = 1/x above x = 1 the
// c1 h f term is written (c1 / r) (f / k), since h r = 1/k: nothing then
// overflows or underflows before the result does (x up to FLT_MAX).  The
// denominators d and c2 lie in [1, 685], so the approximate division
// __fdividef (2 ulp) is exact enough; f / k and 1/x use the correctly rounded
// division and reciprocal.
__device__ __forceinline__ void qss_weights32(float x, float& a, float& b) {
    float n, d, dn;
    if (x <= 1.f) {
        n = fmaf(fmaf(x + 11.f, x, 60.f), x, 180.f);
        d = fmaf(fmaf(x + 12.f, x, 60.f), x, 360.f);
        dn = fmaf(x, x, 180.f);
    } else {
        const float r = __frcp_rn(x);
        n = fmaf(fmaf(fmaf(180.f, r, 60.f), r, 11.f), r, 1.f);
        d = fmaf(fmaf(fmaf(360.f, r, 60.f), r, 12.f), r, 1.f);
        dn = r * fmaf(180.f * r, r, 1.f);
    }
    a = __fdividef(n, d);
    b = __fdividef(dn, d);
}

__device__ __forceinline__ float qss_update1_32(float y, float f, float k, float h) {
    const float x = __fmul_rn(k, h);
    if (x <= 1.f) {
        const float c0 = fmaf(fmaf(12.f, x, -120.f), x, 360.f);
        const float c1 = fmaf(fmaf(x + 12.f, x, 60.f), x, 360.f);
        const float c2 = fmaf(fmaf(fmaf(x + 12.f, x, 72.f), x, 240.f), x, 360.f);
        return __fdividef(fmaf(c0, y, c1 * __fmul_rn(h, f)), c2);
    }
    const float r = __frcp_rn(x);
    const float c0 = fmaf(fmaf(360.f, r, -120.f), r, 12.f) * __fmul_rn(r, r);
    const float c1r = fmaf(fmaf(fmaf(360.f, r, 60.f), r, 12.f), r, 1.f);  // c1 / r
    const float c2 = fmaf(fmaf(fmaf(fmaf(360.f, r, 240.f), r, 72.f), r, 12.f), r, 1.f);
    return __fdividef(fmaf(c0, y, c1r * __fdiv_rn(f, k)), c2);
}

}  // namespace kn
