// dfloat.cuh -- a value as an unevaluated sum of two floats (48 significant bits), for arithmetic
// that starts from FP64 inputs and ends in FP32 or 16-bit storage.
//
// A GB300 SM finishes 2 FP64 operations a clock against 128 FP32 ones, so a sum or a product of two
// such pairs (8 and 4 FP32 instructions) takes about a tenth of the time of the FP64 instruction.
// The sums and products rest on Dekker's and Knuth's error-free transformations (T. J. Dekker, "A
// floating-point technique for extending the available precision", Numer. Math. 18, 1971).  The pair is
// not normalised after each operation: l stays within a few last places of h, so an operation is
// exact to about 2^-44 of its operands' magnitude, 2^-20 of the last place of the float that is
// stored in the end (normalising took 3 more instructions an operation: lbm_init of a 192^3 FP32 box 15%
// longer).  Infinities and values beyond the FP32 range become NaN here, and values below about 2^-100 lose the last
// bits of their low part; callers redo both in FP64.
#pragma once

#include <stdint.h>

namespace lbm {

struct DF {
    float h, l;
    DF() = default;
    __host__ __device__ constexpr DF(float a) : h(a), l(0.0f) {}
    __host__ __device__ constexpr DF(float a, float b) : h(a), l(b) {}
    // 47 leading bits of x by integer operations (the conversions between float and double run at the
    // FP64 rate): the float of the 24 leading bits, and the next 23 as the difference of two floats
    // one binade apart.  Outside 2^-103 <= |x| < 2^128 by conversion.
    __device__ __forceinline__ explicit DF(double x) {
        const uint32_t w1 = (uint32_t)__double2hiint(x), w0 = (uint32_t)__double2loint(x);
        const uint32_t s = w1 & 0x80000000u, e = (w1 >> 20) & 0x7ffu;
        if (e - 920u <= 1150u - 920u) {
            h = __uint_as_float(s | ((e - 896u) << 23) | ((w1 & 0xfffffu) << 3) | (w0 >> 29));
            const uint32_t b = s | ((e - 919u) << 23);
            l = __uint_as_float(b | ((w0 >> 6) & 0x7fffffu)) - __uint_as_float(b);
        } else if ((w1 << 1 | w0) == 0u) {
            h = __uint_as_float(s);
            l = 0.0f;
        } else {
            h = (float)x;
            l = (float)(x - (double)h);
        }
    }
};

#ifdef __CUDACC__
// a + b: exact
__device__ __forceinline__ DF df_two(float a, float b) {
    const float s = a + b, t = s - a;
    return DF(s, (a - (s - t)) + (b - t));
}
__device__ __forceinline__ DF operator+(DF a, DF b) {
    const DF s = df_two(a.h, b.h);
    return DF(s.h, s.l + (a.l + b.l));
}
__device__ __forceinline__ DF operator-(DF a) { return DF(-a.h, -a.l); }
__device__ __forceinline__ DF operator-(DF a, DF b) { return a + (-b); }
__device__ __forceinline__ DF operator*(DF a, DF b) {
    const float p = __fmul_rn(a.h, b.h);
    return DF(p, fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -p))));
}
__device__ __forceinline__ DF& operator+=(DF& a, DF b) { return a = a + b; }
__device__ __forceinline__ DF& operator-=(DF& a, DF b) { return a = a - b; }
__device__ __forceinline__ DF fma(DF a, DF b, DF c) { return a * b + c; }
// one Newton step from the FP32 value
__device__ __forceinline__ DF df_sqrt(DF a) {
    if (!(a.h > 0.0f)) return DF(sqrtf(a.h));
    const float s = sqrtf(a.h);
    const DF d = a - DF(s) * DF(s);
    return DF(s, (d.h + d.l) / (2.0f * s));
}
__device__ __forceinline__ float df_value(DF a) { return a.h + a.l; }
__device__ __forceinline__ double df_double(DF a) { return (double)a.h + (double)a.l; }
#endif

}  // namespace lbm
