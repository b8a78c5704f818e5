// The alpha-step of the decomposition: the ridge solve of a group-row from its sums.
#pragma once
#include <cuda_runtime.h>

namespace ptqtp {

constexpr double kLambda0 = 1e-8, kLambdaMax = 1.0, kKappaThr = 1e6;

// a / b for two numerators that are finite and not negative zero, far from the ends of the range, correctly rounded: with y = RN(1 / b)
// and q within one unit of the quotient, q + y (a - b q) rounded once is RN(a / b) (P. Markstein, "Computation of elementary functions
// on the IBM RISC System/6000 processor", 1990).  The first correction brings a y there, the second is the theorem's.
__device__ __forceinline__ double quotient(double a, double b, double y) {
    double q = __dmul_rn(a, y);
    q = __fma_rn(__fma_rn(-b, q, a), y, q);
    return __fma_rn(__fma_rn(-b, q, a), y, q);
}
// The alpha-step from the sums: new lambda and scales (Eq. 3-6, Algorithm 2, Appendix B and C).  FINITE: the sums are.
static __device__ __noinline__ double enlarged_lambda(double fro, double det, double lam) {
    const double kappa = __ddiv_rn(fro, fabs(det));
    if (kappa >= kKappaThr) lam = fmin(__dmul_rn(lam, __dsqrt_rn(__ddiv_rn(kappa, kKappaThr))), kLambdaMax);
    return fmax(lam, kLambda0);
}
template <bool FINITE>
__device__ __forceinline__ void solve_scales(double n11, double n22, double n12, double b1, double b2, double& lam, double& a1,
                                             double& a2) {
    double A11 = __dadd_rn(n11, lam), A22 = __dadd_rn(n22, lam);
    const double n12sq = __dmul_rn(n12, n12);
    double det = __dsub_rn(__dmul_rn(A11, A22), n12sq);
    const double fro = __dadd_rn(__dadd_rn(__dmul_rn(A11, A11), __dmul_rn(A22, A22)), __dmul_rn(__dmul_rn(2.0, n12), n12));
    // kappa = fro / |det|: the division is left out where its result cannot reach the threshold; lambda, never below kLambda0, stays
    if (!(fro < 0.5 * kKappaThr * fabs(det))) {
        lam = enlarged_lambda(fro, det, lam);
        A11 = __dadd_rn(n11, lam);
        A22 = __dadd_rn(n22, lam);
        det = __dsub_rn(__dmul_rn(A11, A22), n12sq);
    }
    const double p1 = __dsub_rn(__dmul_rn(A22, b1), __dmul_rn(n12, b2)), p2 = __dsub_rn(__dmul_rn(A11, b2), __dmul_rn(n12, b1));
    if (FINITE) {
        const double y = __drcp_rn(det);
        a1 = quotient(p1, det, y);
        a2 = quotient(p2, det, y);
    } else {
        a1 = __ddiv_rn(p1, det);
        a2 = __ddiv_rn(p2, det);
    }
}

}  // namespace ptqtp
