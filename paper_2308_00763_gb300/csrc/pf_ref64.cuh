// pf_ref64.cuh -- the elementary functions of the FP64 filter, from tables.
//
// This part issues 1.7 FP64 operations per clock and SM (profiles/cuda_core_peaks.json, DFMA)
// against 125 FP32 and 64 integer multiplications, so the FP64 step is bound by the count of
// its FP64 operations, two thirds of which were the math library's log, sqrt, sincospi and exp.
// Table-driven forms (P. T. P. Tang, "Table-driven implementation of the exponential function
// in IEEE floating-point arithmetic", ACM TOMS 15, 1989, and "... of the logarithm function",
// ACM TOMS 16, 1990; angle addition for sine and cosine) need 21 FP64 operations a Box-Muller
// pair and 9 an exponential; field extraction, scaling by powers of two and the conversions to
// and from FP32 (which run at the FP64 rate) are integer operations on the words.
// The tables (104 KB) hold correctly rounded values, written by the build (ref64_tables.py) and
// compiled in as initialised data: every context that loads the library has them, with no upload
// to order against a launch and no record of who has made one.  The argument of the logarithm and
// the angle have 24 bits (the generator's uniforms), which the splits below use.
// Largest errors in ulp of the value (and their root mean square), over all 2^23 uniforms, and
// over 2^22 arguments of the exponential in [-30, 0], CUDA's functions -> these:
//   radius        0.852 (0.3254) -> 0.852 (0.3254)
//   sine, cosine  1.476 (0.3610) -> 1.093 (0.2888)
//   exponential   0.888 (0.3017) -> 0.501 (0.2887)
// Measured us a frame when they came in, library functions -> tables: 2^20 particles 375 -> 227, 200003
// 231 -> 134 (the sine and cosine as accurate as above: 2 % of the step now).
#pragma once
#include <stdint.h>

namespace pfk {

struct Ref64Tables {
    double2 turn_hi[1024];   // (cos, sin)(2 pi i / 2^13): an octant's top 10 bits
    float2 turn_rest[1024];  // ... their rounding errors
    double2 turn_lo[2048];   // (cos - 1, sin)(2 pi i / 2^24): its low 11 bits
    double2 ex[2048];        // 2^(i / 2048) and its rounding error
    // per mantissa interval of [1, 2): c ~ 1 / centre with 24 bits, and -ln c (from interval
    // kLnUpper on -ln 2c: the mantissa is halved) as a multiple of 2^-42 and the rest
    struct Ln { float c, lo; double hi; } ln[1024];
    struct Ln eln2[32];      // -i ln 2 likewise (c unused)
};
constexpr int kLnUpper = 424;   // first interval whose centre is above sqrt 2

__device__ const Ref64Tables g_ref64 = {
#include "ref64_tables.inc"
};

// Exact conversions of normal values by their words.
__device__ __forceinline__ double widen_bits(float f) {
    const uint32_t b = __float_as_uint(f);
    return __hiloint2double(static_cast<int>((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)),
                            static_cast<int>(b << 29));
}
// (the top 20 mantissa bits)
__device__ __forceinline__ float narrow_bits(double d) {
    const uint32_t h = static_cast<uint32_t>(__double2hiint(d));
    return __uint_as_float((h & 0x80000000u) | (((h & 0x7fffffffu) - 0x38000000u) << 3));
}
__device__ __forceinline__ double scale_bits(double d, int e) {   // d * 2^e, both normal
    return __hiloint2double(__double2hiint(d) + e * 0x00100000, __double2loint(d));
}
__device__ __forceinline__ double flip_bits(double d, uint32_t sign) {
    return __hiloint2double(static_cast<int>(static_cast<uint32_t>(__double2hiint(d)) ^ sign), __double2loint(d));
}

// Two N(0,1) draws from the uniforms of two words: r = sqrt(-2 ln u_a) times (cos, sin)(2 pi u_b).
__device__ __forceinline__ void box_muller_table(uint32_t wa, uint32_t wb, double &nx, double &ny) {
    // u_a = m / 2^24, m odd with 24 bits: m = 2^k z, z in [1, 2)
    const uint32_t m = (wa >> 8) | 1u;
    const int lz = __clz(static_cast<int>(m));            // 8 .. 31, k = 31 - lz
    const uint32_t f = (m << lz) << 1;                    // the fraction, left aligned
    const double z = __hiloint2double(static_cast<int>(0x3ff00000u | (f >> 12)), static_cast<int>(f << 20));
    const int j = static_cast<int>(f >> 22);
    const Ref64Tables::Ln e = g_ref64.ln[j], w = g_ref64.eln2[lz - 7 - (j >= kLnUpper ? 1 : 0)];
    const double base = w.hi + e.hi;                      // exact
    const double r = fma(z, widen_bits(e.c), -1.0);       // exact; |r| <= 2^-11
    // ln(1 + r) = r + r^2 (-1/2 + r (1/3 + r (-1/4 + r/5))); the last bracket in FP32
    const double q = fma(r, widen_bits(fmaf(0.2f, narrow_bits(r), -0.25f)), 1.0 / 3.0);
    const double l = base + (fma(r * r, fma(r, q, -0.5), r) + widen_bits(w.lo + e.lo));
    // y = -2 ln u in (1e-7, 34); its root by two Newton steps from the FP32 reciprocal root
    const double y = scale_bits(flip_bits(l, 0x80000000u), 1);
    const double g = widen_bits(rsqrtf(narrow_bits(y)));
    const double h = scale_bits(g, -1);
    double s = y * g;
    s = fma(fma(-s, s, y), h, s);
    s = fma(fma(-s, s, y), h, s);
    // u_b = v / 2^24, v odd: quadrant, the angle's distance to the nearer axis (below an octant, so
    // that neither value is a difference of larger ones), and that angle's two halves
    const uint32_t v = (wb >> 8) | 1u, rem = v & 0x3fffffu, quad = v >> 22;
    const bool far = rem > 0x200000u;
    const uint32_t o = far ? 0x400000u - rem : rem;
    const double2 a = __ldg(&g_ref64.turn_hi[o >> 11]), b = __ldg(&g_ref64.turn_lo[o & 2047u]);
    const float2 t = __ldg(&g_ref64.turn_rest[o >> 11]);
    // cos(a + b) = cos a + (rest + cos a (cos b - 1) - sin a sin b), the sine likewise
    const double ca = s * (a.x + fma(a.x, b.x, fma(-a.y, b.y, widen_bits(t.x))));
    const double sa = s * (a.y + fma(a.y, b.x, fma(a.x, b.y, widen_bits(t.y))));
    const bool swap = far != ((quad & 1u) != 0u);
    nx = flip_bits(swap ? sa : ca, (quad == 1u || quad == 2u) ? 0x80000000u : 0u);
    ny = flip_bits(swap ? ca : sa, quad >= 2u ? 0x80000000u : 0u);
}

// exp(d) for |d| < 700 (the caller's test is on the high word): 2^(k + i/2048) (1 + p(r)).
__device__ __forceinline__ bool exp_table_takes(double d) {
    return (static_cast<uint32_t>(__double2hiint(d)) & 0x7fffffffu) < 0x4085e000u;
}
__device__ __forceinline__ double exp_table(double d) {
    const double magic = 6755399441055744.0;              // 1.5 * 2^52
    const double t = fma(d, 2954.639443740597, magic);   // 2048 / ln 2
    const int i = __double2loint(t);
    const double kd = t - magic;
    // ln 2 / 2048 in two parts, the first with 33 bits (kd has at most 21: the product is exact)
    const double r = fma(kd, 2.0512280628325608e-14, fma(kd, -0.0003384507717782981, d));
    // p = e^r - 1 = r + r^2 (1/2 + r (1/6 + r/24)), the last bracket in FP32
    const double p = fma(r * r, fma(r, widen_bits(fmaf(narrow_bits(r), 1.0f / 24.0f, 1.0f / 6.0f)), 0.5), r);
    const double2 v = __ldg(&g_ref64.ex[i & 2047]);
    return scale_bits(v.x + fma(v.x, p, v.y), i >> 11);
}

}  // namespace pfk
