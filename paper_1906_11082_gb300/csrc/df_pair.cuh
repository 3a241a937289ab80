// Pair distances of direct sums in double-float, for the reference gravity
// and the self-gravitation sums.
//
// The FP64 pipe (2 operations per clock and SM) is 1/64 of the float pipe, so
// a double-float pair of about 60 float operations beats one of ten FP64
// operations. A pair errs by about 2^-45 relative, unbiased; a sum over N
// pairs by that over sqrt(N), below the rounding of an FP64 sum.
//
// Coordinates are scaled by a power of two to [-1, 1] and cut into three
// floats on the grids 2^-22, 2^-45 and the rest, so that differences of the
// first two limbs are exact.
#pragma once

#include <cuda_runtime.h>
#include <cstdint>

namespace nm {

constexpr int kLimbs = 9;   // three limbs of three coordinates, [limb][coordinate]

// limbs[i * kLimbs + 3 l + d] of the points x[stride i + d], scaled by inv.
static __global__ void split_points_kernel(int64_t n, int stride, const double* x, double inv, float* limbs) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < 3 * n; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / 3;
        const int d = (int)(t - 3 * i);
        const double v = x[stride * i + d] * inv;
        const double h = rint(v * 0x1p22) * 0x1p-22, r = v - h, m = rint(r * 0x1p45) * 0x1p-45;
        float* o = limbs + i * kLimbs + d;
        o[0] = (float)h;
        o[3] = (float)m;
        o[6] = (float)(r - m);
    }
}

// (h, l) = a - b of one coordinate given as three limbs each. The first
// difference is zero or at least the grid step, the second at most that step.
__device__ __forceinline__ void limb_diff(float ah, float am, float al, float bh, float bm, float bl, float& h, float& l) {
    const float d1 = __fadd_rn(ah, -bh), d2 = __fadd_rn(am, -bm), d3 = __fadd_rn(al, -bl);
    h = __fadd_rn(d1, d2);
    l = __fadd_rn(__fadd_rn(d2, -__fadd_rn(h, -d1)), d3);
}

// (s, e) = a + b exactly.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float z = __fadd_rn(s, -a);
    e = __fadd_rn(__fadd_rn(a, -__fadd_rn(s, -z)), __fadd_rn(b, -z));
}

// y ~ 1/r (a float) and e = 1 - r^2 y^2 of the vector d = (h, l): 1/r = y (1 +
// e/2 + 3/8 e^2) and 1/r^3 = y^3 (1 + 3/2 e + 15/8 e^2) up to e^3 ~ 2^-65.
// q + ql = y^2.
__device__ __forceinline__ void inv_dist_df(const float (&h)[3], const float (&l)[3], float& y, float& e, float& q, float& ql) {
    float p[3], r[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        p[d] = __fmul_rn(h[d], h[d]);
        r[d] = __fmaf_rn(__fadd_rn(h[d], h[d]), l[d], __fmaf_rn(h[d], h[d], -p[d]));
    }
    float s, s2, e1, e2;
    two_sum(p[0], p[1], s, e1);
    two_sum(s, p[2], s2, e2);
    const float lo = __fadd_rn(__fadd_rn(__fadd_rn(r[0], r[1]), r[2]), __fadd_rn(e1, e2));
    asm("rsqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(s2));
    q = __fmul_rn(y, y);
    ql = __fmaf_rn(y, y, -q);
    e = __fmaf_rn(-lo, q, __fmaf_rn(-s2, ql, __fmaf_rn(-s2, q, 1.f)));
}

// (a, b) += (wh + wl)(xh + xl): the sum in a, its errors in b.
__device__ __forceinline__ void df_add(float& a, float& b, float wh, float wl, float xh, float xl) {
    const float p = __fmul_rn(wh, xh);
    const float t = __fmaf_rn(wl, xh, __fmaf_rn(wh, xl, __fmaf_rn(wh, xh, -p)));
    float s, e;
    two_sum(a, p, s, e);
    a = s;
    b = __fadd_rn(b, __fadd_rn(e, t));
}

}  // namespace nm
