// FP64 links and half spinors as integer and float limbs, and their products off the FP64 pipe
// (sm_103a).
//
// GB300 issues 2 FP64 operations per SM and clock (conversions between doubles and integers
// included), so the 840 operations a site takes bound the FP64 operator at 420 clocks per site
// and SM, ten times its HBM time.  A 32 x 32-bit multiply-add onto a 64-bit sum costs four cycles
// of a scheduler, an FP32 one one, an FP64 one 64.  So a link entry, at most one in modulus, is
// kept as u = H 2^-30 + L 2^-62, H an integer and L a float, and a half spinor likewise in units
// of the power of two above the largest component that the lane has met.  A real product is
//   H H' 2^-60   exact, summed in 64-bit integers, and
//   (H L' + L H') 2^-92   in FP32,
// and the sum of the eight hops, an integer in 2^-57 units, becomes a double with one rounding.
// FP64 arithmetic rounds each partial sum to 2^-53 of itself; here the FP32 products are off by 2^-24
// of 2^-30 units, spinors by 2^-62 and links by 2^-56.  In norm the result is closer to the exact
// operator than with FP64 arithmetic (relative error against 128-bit arithmetic, Haar links, Gaussian
// spinors: kappa 0.12 8.2e-17 -> 6.2e-17, kappa 1 1.57e-16 -> 1.01e-16, recon-12 at kappa 0.12
// 1.06e-16 -> 9.1e-17).  A component far below the unit is not: what that could lose goes through
// FP64 arithmetic (kFxSmallBits below).
// Measured, one Dslash with L2 flushed: 32^3 x 64 3090 -> 838 us (256-thread blocks; 64: 857),
// 16^4 107 -> 37 us; with recon-12 links 5066 -> 978 us.  (Three integer products of 29-bit limbs per
// real product, the first form: 882-888, 36.5 and 1400 us.)  What bounds it now is the latency of its
// integer and FP64 results with 16 warps per SM: on 32^3 x 64 the integer, multiply-add and FP64 pipes
// are busy 48, 40 and 39 % of the cycles, the XU pipe 2 %, DRAM 32 %, issue slots 51 %.
//
// Bounds.  A spinor component is a sum of two doubles, each below (1 - 2^-21) units, so H fits 32
// bits; |L| <= 2^31 (a rebuilt row's 2^31 + 2^10); links |H| <= 2^30 (1 + 2^-11) with rows and columns of
// norm at most 1 + 2^-10.  By Cauchy and Schwarz a sum of six products H H' is below sqrt(6) 2^61
// (1 + 2^-10) < 2^62.3, the small ones, in units of the sums, below 2^30, one hop below sqrt(6) 2^58
// and eight hops below 2^62.3.
#pragma once
#include <cuda_runtime.h>
#include <cmath>
#include <cstring>

namespace wd {

constexpr double kFxLinkScale = 0x1p30;          // H of a link entry of one
constexpr int kFxAccBits = 57, kFxAccShift = 3;  // products come in units 2^-60, sums in 2^-57
constexpr long long kFxHalfAcc = 1ll << (kFxAccShift - 1);
constexpr float kFxSmallToAcc = 0x1p-35f;        // small products come in units 2^-92
// Exponents (biased) of the units this arithmetic takes: below, a scaled result could be
// subnormal; above, the sum of eight hops could overflow.  Other fields go through FP64.
constexpr int kFxMinExp = 128, kFxMaxExp = 2030;

// A site with a complex sum whose parts are both below 2^-kFxSmallBits units is redone in FP64 where
// one colour of all spinors that a spin of its sums takes is below 2^-kFxSpreadBits units and not zero,
// unless every colour is below 2^-kFxNoiseBits, as rounding leaves it where a projection cancels (around
// a point source half of the sums are such: with them redone a 24^3 x 48 FP64 solve took 40.4 ms for 33.6).
// On Gaussian fields one warp in two million gets as far as looking at the spinors; with the real and
// imaginary parts of a sum each by itself one in a hundred did, and 16^4 took 71 us for 32.
constexpr int kFxSmallBits = 14, kFxSpreadBits = 12, kFxNoiseBits = 45;
constexpr int kFxSmallHi = 1 << (kFxAccBits - kFxSmallBits - 32);  // that sum's high word

// a float of given bits and a float's bits, on either side (the arithmetic of a link is also compiled
// for the host, where tests look at the limbs)
__host__ __device__ __forceinline__ float fx_float(int b) {
#ifdef __CUDA_ARCH__
    return __int_as_float(b);
#else
    float f;
    memcpy(&f, &b, sizeof f);
    return f;
#endif
}
__host__ __device__ __forceinline__ int fx_bits(float f) {
#ifdef __CUDA_ARCH__
    return __float_as_int(f);
#else
    int b;
    memcpy(&b, &f, sizeof b);
    return b;
#endif
}
// link entry -> (H, bits of the float L): u = H 2^-30 + L 2^-62
__host__ __device__ __forceinline__ int2 fx_link(double u) {
    const int h = (int)rint(u * kFxLinkScale);
    return make_int2(h, fx_bits((float)(fma((double)h, -0x1p-30, u) * 0x1p62)));
}
__host__ __device__ __forceinline__ double fx_link_value(int h, int l) {
    return fma((double)h, 0x1p-30, (double)fx_float(l) * 0x1p-62);
}

// the larger of m and the |hi words| of two doubles, as float bits; NaN for words from
// 0x7f800001 on (doubles of 2^1017 and above, infinities and NaN)
__device__ __forceinline__ float fx_max(float m, double a, double b) {
    float r;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;"
        : "=f"(r) : "f"(m), "f"(__int_as_float(__double2hiint(a))), "f"(__int_as_float(__double2hiint(b))));
    return r;
}

// |d| in units 2^(E - 1022 - 62), truncated; E + 1 above the exponent of d;
// c = ((E + 2) << 21) | 0x1fffff
__device__ __forceinline__ unsigned long long fx_fixed(double d, unsigned c) {
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const unsigned n = (c - 2u * hi) >> 21;  // E + 2 - (exponent of d); the sign drops out
    const unsigned a = __funnelshift_l(lo, hi, 11) | 0x80000000u, b = lo << 11;
    unsigned long long t;
    asm("{\n\t.reg .b64 t;\n\tmov.b64 t, {%1, %2};\n\tshr.u64 %0, t, %3;\n\t}" : "=l"(t) : "r"(b), "r"(a), "r"(n));
    return t;
}
// s 2^-62 units as H 2^-30 + L 2^-62, |L| <= 2^31
__device__ __forceinline__ void fx_split(long long s, int &h, float &l) {
    const int lo = (int)s;
    h = (int)(s >> 32) + (int)((unsigned)lo >> 31);
    l = (float)lo;
}
// limbs of (-1)^m d (m = 0 or -1)
__device__ __forceinline__ void fx_limbs(double d, int m, unsigned c, int &h, float &l) {
    m ^= __double2hiint(d) >> 31;
    fx_split((long long)(fx_fixed(d, c) ^ (unsigned long long)(long long)m) - m, h, l);
}
// limbs of (-1)^ma a + (-1)^mb b
__device__ __forceinline__ void fx_sum(double a, int ma, double b, int mb, unsigned c, int &h, float &l) {
    ma ^= __double2hiint(a) >> 31;
    mb ^= __double2hiint(b) >> 31;
    fx_split((long long)(fx_fixed(a, c) ^ (unsigned long long)(long long)ma) +
             (long long)(fx_fixed(b, c) ^ (unsigned long long)(long long)mb) - (ma + mb), h, l);
}

// a magnitude, given as twice a high word, in units of exponent E: 0 zero (or below 2^-1042), 1 below
// 2^-kFxNoiseBits, 2 below 2^-kFxSpreadBits, 3 larger
__device__ __forceinline__ unsigned fx_class(unsigned hi2, int E) {
    const int e = (int)(hi2 >> 21);
    return hi2 == 0 ? 0u : e <= E - kFxNoiseBits ? 1u : e <= E - kFxSpreadBits ? 2u : 3u;
}

__host__ __device__ __forceinline__ long long fx_mac(int a, int b, long long s) { return (long long)a * b + s; }

// (hr, hi, fr, fi) += u z (ADJ: conj(u) z) for a link entry u and z = x + iy with limbs
// (x, xf = float(x), xl) and likewise y; mre, mim: the factors of u's imaginary limb in the
// real and the imaginary part (ADJ ? y : -y, ADJ ? -x : x).  hr, hi: exact products of the high
// limbs; fr, fi: the cross products in FP32, in units 2^-32 of those.
template <bool ADJ>
__host__ __device__ __forceinline__ void fx_cmac(int4 u, int x, int mre, int y, int mim, float xf, float yf, float xl, float yl,
                                        long long &hr, long long &hi, float &fr, float &fi) {
    const float rf = (float)u.x, rl = fx_float(u.y), jf = ADJ ? -(float)u.z : (float)u.z,
                jl = ADJ ? -fx_float(u.w) : fx_float(u.w);
    hr = fx_mac(u.z, mre, fx_mac(u.x, x, hr));
    hi = fx_mac(u.z, mim, fx_mac(u.x, y, hi));
    fr = fmaf(-jl, yf, fmaf(-jf, yl, fmaf(rl, xf, fmaf(rf, xl, fr))));
    fi = fmaf(jl, xf, fmaf(jf, xl, fmaf(rl, yf, fmaf(rf, yl, fi))));
}

// The link entry of the value h 2^-60 + f 2^-92.  The cross sums f of a rebuilt entry (up to 2^63)
// take L past 2^31 several times over; what is over is carried to H, so that |L| <= 2^31 + 2^10, as of
// a stored entry but for rounding.  Rounded by a magic addition: conversions of f to an integer and
// back cost 2 % of a recon-12 operator.
__host__ __device__ __forceinline__ int2 fx_link_of(long long h, float f) {
    constexpr float magic = 0x1.8p23f;
    const int q = (int)((h + (1ll << 29)) >> 30);
    const int r = (int)(h - ((long long)q << 30));
    const float l = fmaf((float)r, 4.f, f * 0x1p-30f), m = fmaf(l, 0x1p-32f, magic);
    return make_int2(q + (fx_bits(m) - fx_bits(magic)), fx_bits(fmaf(m - magic, -0x1p32f, l)));
}

// Row 2 = conj(row0 x row1) of a recon-12 link in the same arithmetic.
__host__ __device__ __forceinline__ void fx_row2(int4 (&u)[9]) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        // conj(a b - c d) with a = u[i], b = u[3 + j], c = u[j], d = u[3 + i]
        const int i = (k + 1) % 3, j = (k + 2) % 3;
        const int4 a = u[i], b = u[3 + j], c = u[j], d = u[3 + i];
        long long hr = 0, hi = 0;
        float fr = 0.f, fi = 0.f;
        fx_cmac<false>(a, b.x, -b.z, b.z, b.x, (float)b.x, (float)b.z, fx_float(b.y), fx_float(b.w), hr, hi, fr, fi);
        long long gr = 0, gi = 0;
        float er = 0.f, ei = 0.f;
        fx_cmac<false>(c, d.x, -d.z, d.z, d.x, (float)d.x, (float)d.z, fx_float(d.y), fx_float(d.w), gr, gi, er, ei);
        const int2 re = fx_link_of(hr - gr, fr - er), im = fx_link_of(gi - hi, ei - fi);
        u[6 + k] = make_int4(re.x, re.y, im.x, im.y);
    }
}

// v 2^e as a double, rounded once; e = (exponent of the unit) - 1022 - kFxAccBits
__device__ __forceinline__ double fx_value(long long v, int e) {
    const double d = (double)v;
    return v == 0 ? 0.0 : __hiloint2double(__double2hiint(d) + (e << 20), __double2loint(d));
}

}  // namespace wd
