// Conversions between FP64 and FP32 or float-float by integer instructions, bit for bit the values
// of the casts.
//
// GB300 runs the FP64 unit, which also does the FP64 <-> FP32 conversions, at 1/64 of the FP32 rate:
// a conversion holds an SM's unit for 16 clocks per warp, and the 24 conversions (FP32) or 72 to 96
// FP64 instructions (float-float) per site took longer than the memory traffic of the layout kernels
// (64 x 32^3, FP32: 181 us in and 121 us out, 88% of the FP64 unit's rate, at 44% and 73% of the
// copy bandwidth). Rounding a mantissa takes 8 integer instructions, 4 to 6 clocks per warp. Values
// outside the normal range of both formats (and, for float-float, below 2^-70, where the low word's
// scale factor would leave FP32) take the casts.
#pragma once
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define OVL_HD __host__ __device__ __forceinline__
#else
#include <math.h>
#define OVL_HD inline
#endif

namespace ovl {

OVL_HD uint32_t conv_f_bits(float x) {
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    uint32_t u;
    memcpy(&u, &x, 4);
    return u;
#endif
}
OVL_HD float conv_f_of(uint32_t u) {
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float x;
    memcpy(&x, &u, 4);
    return x;
#endif
}
OVL_HD void conv_d_words(double x, uint32_t &hi, uint32_t &lo) {
#ifdef __CUDA_ARCH__
    hi = (uint32_t)__double2hiint(x);
    lo = (uint32_t)__double2loint(x);
#else
    uint64_t u;
    memcpy(&u, &x, 8);
    hi = (uint32_t)(u >> 32);
    lo = (uint32_t)u;
#endif
}
OVL_HD double conv_d_of(uint32_t hi, uint32_t lo) {
#ifdef __CUDA_ARCH__
    return __hiloint2double((int)hi, (int)lo);
#else
    const uint64_t u = (uint64_t)hi << 32 | lo;
    double x;
    memcpy(&x, &u, 8);
    return x;
#endif
}
OVL_HD int conv_f2i_rn(float x) {
#ifdef __CUDA_ARCH__
    return __float2int_rn(x);
#else
    return (int)lrintf(x);
#endif
}

OVL_HD bool finite_bits(double x) {
    uint32_t hi, lo;
    conv_d_words(x, hi, lo);
    return (hi & 0x7fffffffu) < 0x7ff00000u;
}

// The exponent and upper 23 mantissa bits of a double whose exponent is in the normal FP32 range,
// as FP32 bits without the sign, and whether the 29 bits below round them up (to nearest even).
OVL_HD uint32_t conv_trunc(uint32_t hi, uint32_t lo, uint32_t &up) {
    const uint32_t f = (hi << 3 | lo >> 29) + 0x40000000u;   // exponent - 896
    up = ((lo & 0x1fffffffu) + 0x0fffffffu + (f & 1u)) >> 29;
    return f;
}

// (float)x
OVL_HD float d2f(double x) {
    uint32_t hi, lo, up;
    conv_d_words(x, hi, lo);
    const uint32_t a = hi & 0x7fffffffu, sign = hi & 0x80000000u;
    if (a - (897u << 20) < (254u << 20)) {
        const uint32_t f = conv_trunc(hi, lo, up);
        return conv_f_of(sign | (f + up));
    }
    return (a | lo) == 0 ? conv_f_of(sign) : (float)x;
}
// (double)x
OVL_HD double f2d(float x) {
    const uint32_t b = conv_f_bits(x), a = b & 0x7fffffffu, sign = b & 0x80000000u;
    if (a - 0x00800000u < 0x7f000000u) return conv_d_of(sign | ((a >> 3) + (896u << 20)), b << 29);
    return a == 0 ? conv_d_of(sign, 0u) : (double)x;
}
// h = (float)x, l = (float)(x - h)
OVL_HD void d2ff(double x, float &h, float &l) {
    uint32_t hi, lo, up;
    conv_d_words(x, hi, lo);
    const uint32_t a = hi & 0x7fffffffu, sign = hi & 0x80000000u;
    if (a - (953u << 20) < (197u << 20)) {   // 2^-70 <= |x| < 2^127
        const uint32_t f = conv_trunc(hi, lo, up);
        h = conv_f_of(sign | (f + up));
        const int rem = (int)(lo & 0x1fffffffu) - (int)(up << 29);   // (|x| - |h|) / 2^(e - 52)
        l = (float)(sign ? -rem : rem) * conv_f_of(((a >> 20) - 948u) << 23);
    } else if ((a | lo) == 0) {
        h = conv_f_of(sign);
        l = 0.f;
    } else {
        h = (float)x;
        l = (float)(x - (double)h);
    }
}
// (double)h + (double)l for |l| <= ulp(h) (others by the casts)
OVL_HD double ff2d(float h, float l) {
    const uint32_t b = conv_f_bits(h), a = b & 0x7fffffffu, sign = b & 0x80000000u, c = conv_f_bits(l);
    // h normal, at least 2^-70, and no power of two (the sum could be in the binade below)
    if (a - (57u << 23) < (198u << 23) && (a & 0x7fffffu)) {
        const float s = l * conv_f_of((306u - (a >> 23)) << 23);   // in units of the sum's last place
        if (s < 536870912.f && s > -536870912.f) {   // 2^29: less than h's last mantissa bit; false for NaN
            const int n = conv_f2i_rn(s), m = sign ? -n : n;
            const uint32_t w = b << 29, v = w + (uint32_t)m;
            // carry or borrow out of the low word
            const int carry = m < 0 ? -(int)(v > w) : (int)(v < w);
            return conv_d_of((sign | ((a >> 3) + (896u << 20))) + (uint32_t)carry, v);
        }
    }
    if (((b | c) & 0x7fffffffu) == 0) return conv_d_of(b & c, 0u);
    return (double)h + (double)l;
}

}  // namespace ovl
