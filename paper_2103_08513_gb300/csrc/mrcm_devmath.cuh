// Device arithmetic helpers shared by the libmrcm kernels: FP64 <-> FP32
// conversions, an FP64 reciprocal and maxima that stay off the FP64 unit.
#pragma once
#include <cuda_runtime.h>

namespace mrcm {

// FP64 <-> FP32 conversions on the integer pipe.  On this GPU a conversion
// instruction occupies the FP64 unit as long as an FMA does, and the local
// solve is bound by that unit, so the refinement loop converts with bit
// operations instead: FP64 -> FP32 truncates the significand (round toward
// zero; the FP32 value only feeds the low-precision correction solve),
// flushes magnitudes below the FP32 normal range to zero and saturates to
// infinity above it; FP32 -> FP64 is exact for normal numbers (FP32
// subnormals, which the correction never needs, become zero).
__device__ __forceinline__ float f64_to_f32_rz(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned int sign = (unsigned int)(b >> 32) & 0x80000000u;
    const int e = (int)((b >> 52) & 0x7FF) - 1023 + 127;
    unsigned int f;
    if (e <= 0) f = sign;
    else if (e >= 255) f = sign | 0x7F800000u;
    else f = sign | ((unsigned int)e << 23) | (unsigned int)((b >> 29) & 0x7FFFFFu);
    return __uint_as_float(f);
}
__device__ __forceinline__ double f32_to_f64(float x) {
    const unsigned int f = __float_as_uint(x);
    const unsigned long long sign = (unsigned long long)(f & 0x80000000u) << 32;
    const int e = (int)((f >> 23) & 0xFF);
    unsigned long long b;
    if (e == 0) b = sign;
    else if (e == 255) b = sign | 0x7FF0000000000000ull | ((unsigned long long)(f & 0x7FFFFFu) << 29);
    else b = sign | ((unsigned long long)(e - 127 + 1023) << 52) | ((unsigned long long)(f & 0x7FFFFFu) << 29);
    return __longlong_as_double((long long)b);
}

// 1 / d with integer operations: the FP32 reciprocal Y 2^-24 of the significand M 2^-52, its
// error e = 1 - M Y 2^-76 exactly (below 2^-22, so 64 bits hold it), then Y (1 + e + e^2)
// rounded to 53 bits: within 0.5 ulp over 4e7 random d (1 ulp at d = 2 - ulp).  An FP64 warp
// instruction takes 16 cycles of an SM here and 66 of a dependent chain, so the four FMAs of
// two Newton steps cost a per-cell kernel 64 cycles and a pivot chain 270; these ~30 integer
// instructions cost 8 and 130.  Zero, subnormal, infinite and NaN d, and d whose reciprocal is
// subnormal, take the division.
__device__ __forceinline__ double rcp64(double d) {
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const unsigned ex = (hi >> 20) & 0x7FFu;
    if (ex - 1u > 2042u) return 1.0 / d;
    float yf;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(__uint_as_float(0x3F800000u | (hi & 0xFFFFFu) << 3 | lo >> 29)));
    const unsigned fy = __float_as_uint(yf);                  // in [1/2, 1]
    const unsigned Y = ((fy & 0x7FFFFFu) | 0x800000u) << ((fy >> 23) - 126u);
    const long long E = -(long long)((unsigned long long)lo * Y + ((unsigned long long)(((hi & 0xFFFFFu) | 0x100000u) * Y) << 32));
    const int Eh = (int)(E >> 32);
    const long long c1 = (long long)(int)Y * Eh + (long long)__umulhi(Y, (unsigned)E);            // Y e, in 2^-68
    const unsigned t = (unsigned)(((long long)Eh * Eh) >> 20);                                     // e^2
    const long long R = ((long long)Y << 38) + ((c1 + (long long)(((unsigned long long)Y * t) >> 24)) >> 6);
    const unsigned long long mant = (unsigned long long)(R + 256) >> 9;
    return __longlong_as_double((long long)((((unsigned long long)(2044u - ex) << 52) + mant) |
                                            (unsigned long long)(hi & 0x80000000u) << 32));
}

// n / d from r = 1 / d by one correction step (the quotient's residual is exact in an FMA):
// three FP64 operations
__device__ __forceinline__ double div64(double n, double d, double r) {
    const double q = n * r;
    const double e = fma(-q, d, n);
    return fma(e, r, q);
}

// Maximum of |x| as bits of a non-negative double (integer operations: an FP64 comparison
// occupies the FP64 unit like an FMA); a NaN counts as infinity.
__device__ __forceinline__ unsigned long long abs_bits(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
    return b > 0x7FF0000000000000ull ? 0x7FF0000000000000ull : b;
}

}  // namespace mrcm
