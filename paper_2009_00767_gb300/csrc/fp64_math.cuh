// fp64_math.cuh -- FP64 log, reciprocal and reciprocal square root for the FP64 near fields.
//
// GB300 issues about one FP64 warp instruction per SM every 19 clocks (1.05 TFLOP/s measured with
// fmm_probe_peak) beside four FP32 / integer ones per clock, so a near field in FP64 is bound by its
// count of FP64 instructions and little else.  These functions keep that count low: 5 for log, 3 for
// 1 / x, 5 for 1 / sqrt(x); exponents, table indices and every term far below the result's last bit
// are formed with integer and FP32 instructions.  Results are within 3 units in the last place (log: 2.7
// at 1.001, at most 1.7 elsewhere over 8e7 values of all exponents against quadruple precision; the other
// two below 2), log(1) is 0.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

// Table of the logarithm.  Its intervals are the values of the top bits of x above kFmmLogLow, 2^kFmmLogBits to
// a power of two; kFmmLogLow (0.7065) puts 1 at the centre of one, so that x near 1 has exponent 0, c = 1 and
// log c = 0 and nothing cancels there.  c_j = fl(1 / z_j) for the centre z_j of an interval, and -log(c_j).
constexpr int kFmmLogBits = 9;
constexpr int kFmmLogEntries = 1 << kFmmLogBits;
constexpr int kFmmLogStep = 1 << (20 - kFmmLogBits);   // of the high word
constexpr int kFmmLogLow = 0x3ff00000 - 300 * kFmmLogStep - kFmmLogStep / 2;

__host__ __device__ inline double2 fmm_log_entry(int j) {
    const int h = kFmmLogLow + j * kFmmLogStep + kFmmLogStep / 2;   // the centre's high word, the low one is 0
    const double scale = h < 0x3ff00000 ? 0.5 : 1.0;
    const double c = 1.0 / (scale * (1.0 + (double)(h & 0xfffff) / 1048576.0));
    return make_double2(c, -log(c));
}

__device__ __noinline__ static double fmm_log_rare(double x) { return x > 0.0 ? log(x) : 0.0; }

// log(x) for x >= 0, with 0 for x = 0 (a coincident pair's term).  Table-driven (Tang, "Table-driven
// implementation of the logarithm function in IEEE floating-point arithmetic", ACM TOMS 16, 1990): with
// x = 2^e z and the entry of z's interval, r = z c - 1 (one rounding by FMA, |r| <= 2^-10) and
//     log x = e ln 2 - log c + r (1 + r (-1/2 + r K)),   K = 1/3 + d,  d = r (-1/4 + r (1/5 - r/6)).
// |d| < 2^-12 comes from FP32 (off by 2^-35) and goes into K's bits as a whole multiple of 2^-34, so K's error
// is below 2^-54 of the result also where that is r itself; the next term of the series is below 2^-62 of it.
__device__ __forceinline__ double fmm_log(double x, const double2* __restrict__ tab) {
    const int hi = __double2hiint(x), lo = __double2loint(x);
    if ((unsigned)hi - 0x00100000u >= 0x7fe00000u) return fmm_log_rare(x);   // zero, subnormal or infinite
    const int at = hi - kFmmLogLow;   // e and the interval
    const double2 t = tab[(at >> (20 - kFmmLogBits)) & (kFmmLogEntries - 1)];
    const double r = fma(__hiloint2double(hi - (at & 0xfff00000), lo), t.x, -1.0);
    // r in FP32, truncated, by its bits (r is 0 or at least 2^-106 in magnitude; 0 gives a K that r^2 cancels)
    const int rh = __double2hiint(r);
    const float rf = __uint_as_float((rh & 0x80000000u) |
                                     ((__funnelshift_l(__double2loint(r), rh, 3) - (384u << 23)) & 0x7fffffffu));
    const float d = rf * fmaf(rf, fmaf(rf, -1.f / 6.f, 0.2f), -0.25f);
    const long long di = (int)(__float_as_uint(fmaf(d, 0x1p34f, 12582912.f)) - 0x4b400000u);   // d 2^34, rounded
    const double kd = __longlong_as_double(0x3fd5555555555555ll + di * (1ll << 20));   // K's spacing is 2^-54
    // e as a double, by way of an exact FP32 integer
    const uint32_t e = __float_as_uint(__int_as_float(0x4b400000 + (at >> 20)) - 12582912.f);
    const double ed = __hiloint2double(e == 0u ? 0 : (int)((e & 0x80000000u) | (((e & 0x7fffffffu) >> 3) + (896u << 20))), 0);
    const double s = fma(r, fma(r, kd, -0.5), 1.0);
    return fma(r, s, fma(ed, 0.69314718055994530942, t.y));
}

// 1 / x for a normal x below 2^1022 (the MUFU flushes a subnormal result): the MUFU's start y0, good to about 20
// bits, then y0 (1 + e + e^2) with e = 1 - x y0, the series of 1 / (1 - e) up to a remainder of e^3 < 2^-57.
__device__ __forceinline__ bool fmm_rcp_range(double x) { return (unsigned)__double2hiint(x) - 0x00100000u < 0x7fc00000u; }
__device__ __forceinline__ double fmm_rcp(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// 1 / sqrt(x) for a normal x: the MUFU's start y0, then y0 (1 + e/2 + 3 e^2 / 8) with e = 1 - x y0^2, the series of
// 1 / sqrt(1 - e) up to a remainder of 5 e^3 / 16 < 2^-57.
__device__ __forceinline__ double fmm_rsqrt(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-(x * y), y, 1.0);
    return fma(y * e, fma(e, 0.375, 0.5), y);
}

// The interaction-list offsets as orbits of quarter turns (fp64.cu): a representative of each.
constexpr int kFmmOrbits = 10;
__host__ __device__ constexpr int fmm_orbit_x(int o) { return o < 3 ? 2 : (o == 3 ? 1 : 3); }
__host__ __device__ constexpr int fmm_orbit_y(int o) { return o < 3 ? o : (o == 3 ? 2 : (o < 9 ? o - 6 : 3)); }
// Doubles of the far field's tables for p1 = p + 1 coefficients: R[k][l] and C(m, j) (each padded to an
// even count), then d^-k of every orbit.
__host__ __device__ inline size_t fmm_far_table_doubles(int p1) {
    return 2 * (size_t)((p1 * p1 + 1) & ~1) + 2 * (size_t)kFmmOrbits * p1;
}
