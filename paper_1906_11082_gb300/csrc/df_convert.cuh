// Conversions between double and (pairs of) floats for the device code.
#pragma once

#include <cuda_runtime.h>

namespace nm {

// Conversions between double and float on the integer units: an FP64
// instruction (conversions are) takes 16 cycles of an SM, an integer one
// half a cycle. Values outside the normal ranges go the plain way.
__device__ __forceinline__ double widen(float f) {
    const unsigned u = __float_as_uint(f), a = u & 0x7FFFFFFFu;
    if (a - 0x00800000u >= 0x7F000000u) return (double)f;
    return __hiloint2double((int)((u & 0x80000000u) | ((a >> 3) + 0x38000000u)), (int)(u << 29));
}
// h = float(d), l = float(d - h), both rounded to nearest even.
__device__ __forceinline__ void split_pair(double d, float& h, float& l) {
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const unsigned a = hi & 0x7FFFFFFFu, e = a >> 20;
    if (e - 949u >= 1149u - 949u) {
        h = __double2float_rn(d);
        l = __double2float_rn(d - (double)h);
        return;
    }
    unsigned u = ((a - 0x38000000u) << 3) | (lo >> 29);
    const unsigned r = lo & 0x1FFFFFFFu;
    const unsigned up = r > 0x10000000u || (r == 0x10000000u && (u & 1u));
    u += up;
    const int rem = (int)r - (up ? 0x20000000 : 0);   // d - h in units of 2^(e - 1075)
    const unsigned sg = hi & 0x80000000u;
    h = __uint_as_float(u | sg);
    l = __int_as_float(__float_as_int((float)rem * __uint_as_float((e - 948u) << 23)) ^ sg);
}

}  // namespace nm
