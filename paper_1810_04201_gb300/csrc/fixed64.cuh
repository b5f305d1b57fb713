// FP64 links and half spinors as 58-bit fixed-point numbers, and their products on the
// integer multiply-add pipe (sm_103a).
//
// GB300 issues 2 FP64 operations per SM and clock (conversions between doubles and integers
// included), so the 840 operations a site takes bound the FP64 operator at 420 clocks per site
// and SM, ten times its HBM time.  The integer pipes are wider: a 32 x 32-bit multiply-add onto
// a 64-bit sum costs four cycles of a scheduler where an FP64 multiply-add costs 64.  A link
// entry is at most one in modulus, so it is kept as u = (H 2^29 + L) 2^-58 with
// -2^28 <= L < 2^28, and a half spinor as (H 2^29 + L) 2^-57 in units of the power of two above
// the largest component that the lane has met.  A real product is then three integer
// multiply-adds,
//   H H' 2^58 + (H L' + L H') 2^29   (L L' is dropped: about a unit of 2^-57 per hop),
// a complex one nine (three real products), and the sums are exact: one rounding per link
// product and one when the sum of the eight hops becomes a double.  FP64 arithmetic rounds each
// partial sum to 2^-53 of itself, so the result is as close to the exact operator as before:
// 1.5e-16 relative on Haar links and Gaussian spinors for both (64-bit reference summed in
// another order; the rounding of the result itself).
// Measured, one Dslash with L2 flushed: 32^3 x 64 3090 -> 903 us, 16^4 107 -> 36 us; with
// recon-12 links 5066 -> 1400 us.
//
// Bounds.  Spinor components (a sum of two doubles) have |H| < 2^29, |L| < 2^30; links
// |H| <= 2^29 (1 + 2^-11), |L| <= 2^28 and rows and columns of norm at most 1 + 2^-10.  The
// largest sum, the middle one of (ur + ui)(x + y), is below
// sqrt(2) 2^29 sqrt(3) 2^31 + 3 2^29 2^30 < 2^62.2; a hop is below sqrt(3) 2^58.6 < 2^59.4
// and eight hops below 2^62.4.
#pragma once
#include <cuda_runtime.h>

namespace wd {

constexpr int kFxBits = 29;                      // bits of a low limb
constexpr double kFxLinkScale = 0x1p58;          // a link entry of one
constexpr int kFxSpinorBits = 57;                // a spinor component of one unit
// Exponents (biased) of the units this arithmetic takes: below, a scaled result could be
// subnormal; above, the sum of eight hops could overflow.  Other fields go through FP64.
constexpr int kFxMinExp = 128, kFxMaxExp = 2030;

// link entry -> limbs
__device__ __forceinline__ int2 fx_link(double u) {
    const long long f = __double2ll_rn(u * kFxLinkScale);
    const int h = (int)((f + (1ll << (kFxBits - 1))) >> kFxBits);
    return make_int2(h, (int)(f - ((long long)h << kFxBits)));
}
__device__ __forceinline__ double fx_link_value(int h, int l) {
    return fma((double)h, 0x1p-29, (double)l * 0x1p-58);
}

// the larger of m and the |hi words| of two doubles, as float bits; NaN for words from
// 0x7f800001 on (doubles of 2^1017 and above, infinities and NaN)
__device__ __forceinline__ float fx_max(float m, double a, double b) {
    float r;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;"
        : "=f"(r) : "f"(m), "f"(__int_as_float(__double2hiint(a))), "f"(__int_as_float(__double2hiint(b))));
    return r;
}

// |d| in units 2^(E - 1022 - 57), E >= the exponent of d: high limb (28 bits) and low limb
// (29 bits), truncated; c = ((E + 4) << 21) | 0x1fffff
__device__ __forceinline__ void fx_limbs(double d, unsigned c, int &h, int &l) {
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const unsigned n = (c - 2u * hi) >> 21;  // E + 4 - (exponent of d); the sign drops out
    const unsigned a = __funnelshift_l(lo, hi, 11) | 0x80000000u, b = lo << 11;
    unsigned gl, gh;
    asm("{\n\t.reg .b64 t;\n\tmov.b64 t, {%2, %3};\n\tshr.u64 t, t, %4;\n\tmov.b64 {%0, %1}, t;\n\t}"
        : "=r"(gl), "=r"(gh) : "r"(b), "r"(a), "r"(n));
    h = (int)gh;
    l = (int)(gl >> 3);
}

// limbs of (-1)^ma |a| + (-1)^mb |b| with ma, mb = 0 or -1, times the signs of a and b
__device__ __forceinline__ void fx_sum(double a, int ma, double b, int mb, unsigned c, int &h, int &l) {
    int ha, la, hb, lb;
    fx_limbs(a, c, ha, la);
    fx_limbs(b, c, hb, lb);
    ma ^= __double2hiint(a) >> 31;
    mb ^= __double2hiint(b) >> 31;
    const int k = -ma - mb;
    h = (ha ^ ma) + (hb ^ mb) + k;
    l = (la ^ ma) + (lb ^ mb) + k;
}

__device__ __forceinline__ long long fx_mac(int a, int b, long long s) { return (long long)a * b + s; }

// s x 2^(e), e = (exponent of the unit) - 1022 - 57: the double nearest to the integer s,
// moved by the exponent (kFxMinExp..kFxMaxExp keep it normal)
__device__ __forceinline__ double fx_value(long long s, int e) {
    const double d = (double)s;
    return s == 0 ? 0.0 : __hiloint2double(__double2hiint(d) + (e << 20), __double2loint(d));
}

}  // namespace wd
