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
__host__ __device__ __forceinline__ void two_sum(Real a, Real b, Real& s, Real& e) {
    s = a + b;
    const Real bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// (ah, al) += (bh, bl), result renormalised so that |al| <= ulp(ah)/2
template <typename Real>
__host__ __device__ __forceinline__ void df_add(Real& ah, Real& al, Real bh, Real bl) {
    Real s, e;
    two_sum(ah, bh, s, e);
    e += al + bl;
    ah = s + e;
    al = e - (ah - s);
}

// The refinement's (rh, rl) -= (eh, el) + (wh, wl) + (nh, nl) + (sh, sl), the fluxes of a node's four edges: the
// sum renormalised after every edge (the first on its own is df_add onto 0), then subtracted. Gathering the low
// parts in one number instead is 1 - 3 % faster on a whole solve (4000 particles on 1/32 182.4 against 187.9 us,
// on 1/64 806 against 816; 8000 on 1/128 13.36 against 13.49 ms) and leaves 1.3 - 2 times the rounding error.
template <typename Real>
__host__ __device__ __forceinline__ void df_residual(Real& rh, Real& rl, Real eh, Real el, Real wh, Real wl, Real nh,
                                                     Real nl, Real sh, Real sl) {
    Real ah = eh + el, al = el - (ah - eh);
    df_add(ah, al, wh, wl);
    df_add(ah, al, nh, nl);
    df_add(ah, al, sh, sl);
    df_add(rh, rl, -ah, -al);
}

}  // namespace mls2mc
