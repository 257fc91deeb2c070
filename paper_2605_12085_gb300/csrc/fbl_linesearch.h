// The sufficient-decrease test (2.3) in FP64, formed in one place for the host loop,
// the decision kernels and the limit of a trial's objective: the same operations
// with the same roundings (none contracted into an FMA), so that all of them agree
// to the last bit on which trials fail.
#pragma once

#include <math.h>

#ifdef __CUDACC__
#define FBL_HD __host__ __device__ __forceinline__
#else
#define FBL_HD inline
#endif

namespace fbl {

FBL_HD double ls_mul(double a, double b) {
#ifdef __CUDA_ARCH__
    return __dmul_rn(a, b);
#else
    return a * b;  // (the host code is compiled without contraction)
#endif
}
FBL_HD double ls_add(double a, double b) {
#ifdef __CUDA_ARCH__
    return __dadd_rn(a, b);
#else
    return a + b;
#endif
}
FBL_HD double ls_div(double a, double b) {
#ifdef __CUDA_ARCH__
    return __ddiv_rn(a, b);
#else
    return a / b;
#endif
}

// f_N = scale/2 rho, rho the sum of squares.
FBL_HD double ls_objective(double scale, double rho) { return ls_mul(ls_mul(0.5, scale), rho); }

// The right-hand side f_N(x) + g^T d + ||d||^2 / (2 alpha).
FBL_HD double ls_rhs(double scale, double rho0, double gTd, double dd, double alpha) {
    return ls_add(ls_add(ls_objective(scale, rho0), gTd), ls_div(dd, ls_mul(2.0, alpha)));
}

// A partial sum of rho1's squares above this settles that (2.3) fails with the right-hand
// side rhs, whatever the rest of them and the order of the sum: two FP64 sums of the
// same n squares differ by at most 2 n 2^-53 of either, 4.8e-7 for 2^31 blocks.
FBL_HD double ls_limit(double scale, double rhs) {
    return ls_mul(ls_div(rhs > 0.0 ? rhs : 0.0, ls_mul(0.5, scale)), 1.0 + 1e-6);
}

}  // namespace fbl
