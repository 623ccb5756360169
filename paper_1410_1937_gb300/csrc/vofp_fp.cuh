// FP64 arithmetic in fewer FP64 instructions than the plain operators take, with the same results.
#pragma once
#include <cstdint>

namespace vofp {

__device__ __forceinline__ long long bits_of(double a) { return __double_as_longlong(a); }

// r = sqrt(d) and 1 / r.  An approximation y of d^-1/2 to 45 bits comes from FP32 arithmetic (a step of third
// order from rsqrtf, its residual 1 - d y^2 formed without cancellation by fused products, in the manner of
// Dekker's double-length arithmetic), then one FP64 Newton step each for the root and for its reciprocal:
// r = g + (d - g g) y / 2 with g = d y, and 1 / r = y + (1 - r y) y.  Both are within 2^-37 of a half unit in the
// last place, so correctly rounded but for one value in some 2^36.  Five FP64 instructions instead of the
// twelve of sqrt and the division.  Those are taken by values that are not normal numbers of moderate size, and by the two
// below each power of 4, whose root's significand is all ones: the step for its reciprocal ends on a tie there
// (Markstein 1990).
__device__ __forceinline__ void sqrt_and_inverse(double d, double& r, double& inv) {
    const unsigned long long b = (unsigned long long)bits_of(d);
    const unsigned int e = (unsigned int)(b >> 52);   // sign and exponent
    if (e - 200u >= 1600u || (b & 0x1ffffffffffffeull) == 0xffffffffffffeull) {
        r = sqrt(d);
        inv = 1.0 / r;
        return;
    }
    // d = 4^h m, m in [1, 4): m = mh + ml with mh its leading 24 bits
    const unsigned int odd = (e + 1u) & 1u;                  // e = 1023: even power
    const int h = ((int)e - 1023 - (int)odd) / 2;            // exact: e - 1023 - odd is even
    const float mh = __uint_as_float(((127u + odd) << 23) | (unsigned int)((b >> 29) & 0x7fffffu));
    const float ml = (float)(int)(b & 0x1fffffffu) * __uint_as_float((127u - 52u + odd) << 23);
    const float y = fminf(fmaxf(rsqrtf(mh), 0.5f), 1.0f);
    const float p = __fmul_rn(y, y), pe = __fmaf_rn(y, y, -p);
    const float t = __fmul_rn(mh, p), te = __fmaf_rn(mh, p, -t);
    const float res = __fsub_rn(__fsub_rn(1.0f, t), __fmaf_rn(ml, p, __fmaf_rn(mh, pe, te)));
    const float cy = __fmul_rn(y, __fmul_rn(res, __fmaf_rn(0.375f, res, 0.5f)));
    // y + cy in units of 2^-53 (y in [1/2, 1]; |cy| < 2^-21), scaled by 2^-h
    const unsigned int yb = __float_as_uint(y);
    long long yd = ((long long)(yb >> 23) - 127 + 1023 - h) << 52 | (long long)(yb & 0x7fffffu) << 29;
    yd += __float2int_rn(cy * 9007199254740992.0f);
    const double yy = __longlong_as_double(yd), hy = __longlong_as_double(yd - (1ll << 52));
    const double g = __dmul_rn(d, yy);
    r = __fma_rn(__fma_rn(-g, g, d), hy, g);
    inv = __fma_rn(__fma_rn(-r, yy, 1.0), yy, yy);
}

// (float)a for a >= 0, by integer arithmetic where the result is a normal number: the conversion instruction
// takes as long as an FP64 operation.
__device__ __forceinline__ float to_float(double a) {
    const unsigned long long b = (unsigned long long)bits_of(a);
    if ((unsigned int)(b >> 52) - 897u < 252u) {
        const unsigned long long v = b - (896ull << 52);
        return __uint_as_float((unsigned int)((v + 0x0fffffffull + ((v >> 29) & 1ull)) >> 29));
    }
    if (b == 0ull) return 0.0f;
    float f;
    asm volatile("cvt.rn.f32.f64 %0, %1;" : "=f"(f) : "d"(a));   // (volatile: not ahead of the branch)
    return f;
}

}  // namespace vofp
