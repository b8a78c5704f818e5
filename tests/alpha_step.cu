// The solve of dec_solve.h with its shared reciprocal against the one with IEEE divisions, for tests.
#include "dec_solve.h"

__global__ void compare(const double* __restrict__ in, int n, double* out, int* differ) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double* v = in + (size_t)6 * i;                // n11, n22, n12, b1, b2, lambda
    double lam = v[5], a1, a2, lam_div = v[5], d1, d2;
    ptqtp::solve_scales<true>(v[0], v[1], v[2], v[3], v[4], lam, a1, a2);
    ptqtp::solve_scales<false>(v[0], v[1], v[2], v[3], v[4], lam_div, d1, d2);
    out[3 * (size_t)i] = a1;
    out[3 * (size_t)i + 1] = a2;
    out[3 * (size_t)i + 2] = lam;
    if (__double_as_longlong(a1) != __double_as_longlong(d1) || __double_as_longlong(a2) != __double_as_longlong(d2) ||
        __double_as_longlong(lam) != __double_as_longlong(lam_div))
        atomicAdd(differ, 1);
}

extern "C" __attribute__((visibility("default"))) int run_compare(const double* in, int n, double* out, int* differ, void* stream) {
    compare<<<(n + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(in, n, out, differ);
    return (int)cudaGetLastError();
}
