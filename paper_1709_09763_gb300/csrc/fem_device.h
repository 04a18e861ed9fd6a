// Device arithmetic shared by the forward-solve kernels (fem_solve.cu, fem_tile.cu).
#pragma once

#include <cuda_runtime.h>

namespace mls2mc {

// 1 / x rounded to nearest (the same value as the IEEE division 1 / x)
__device__ __forceinline__ float recip(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double recip(double x) { return __drcp_rn(x); }
// The smoother's inverse diagonals on the coarse levels: the approximate reciprocal of the special
// function unit (one instruction, relative error below 2^-22) on the FP32 path. They only shape the
// multigrid preconditioner -- the CG operator and the refinement residual use the edge weights --
// and the preconditioner stays symmetric because every sweep uses the same value at a node.
__device__ __forceinline__ float recip_coarse(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ double recip_coarse(double x) { return __drcp_rn(x); }

// ---- error-free transformations (Knuth TwoSum, Dekker), double-float accumulation ----
template <typename Real>
__device__ __forceinline__ void two_sum(Real a, Real b, Real& s, Real& e) {
    s = a + b;
    const Real bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// (ah, al) += (bh, bl), result renormalised so that |al| <= ulp(ah)/2
template <typename Real>
__device__ __forceinline__ void df_add(Real& ah, Real& al, Real bh, Real bl) {
    Real s, e;
    two_sum(ah, bh, s, e);
    e += al + bl;
    ah = s + e;
    al = e - (ah - s);
}

}  // namespace mls2mc
