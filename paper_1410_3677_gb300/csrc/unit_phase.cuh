// Unit phases: in FP64 from a table, for the FP64 form's kernels, and in FP32 by Taylor series.
#pragma once

#include <cuda_runtime.h>

namespace fstat {

// cos and sin of 2 pi (q / 4 + r), |r| <= 1/8, by Taylor series (first terms left out:
// 2 pi r ^11/11! and ^10/10!, below 2.5e-8); only the low two bits of q count.
__device__ __forceinline__ void unit_f(int q, float r, float &cs, float &sn) {
    const float r2 = r * r;
    constexpr double T = 6.283185307179586476925286766559, T2 = T * T;
    const float s = r * fmaf(r2, fmaf(r2, fmaf(r2, fmaf(r2, (float)(T * T2 * T2 * T2 * T2 / 362880.0),
                                                        (float)(-T * T2 * T2 * T2 / 5040.0)),
                                               (float)(T * T2 * T2 / 120.0)), (float)(-T * T2 / 6.0)), (float)T);
    const float k = fmaf(r2, fmaf(r2, fmaf(r2, fmaf(r2, (float)(T2 * T2 * T2 * T2 / 40320.0),
                                                    (float)(-T2 * T2 * T2 / 720.0)),
                                           (float)(T2 * T2 / 24.0)), (float)(-T2 / 2.0)), 1.f);
    const bool odd = q & 1;
    const float a = odd ? s : k, b = odd ? k : s;
    cs = __int_as_float(__float_as_int(a) ^ (((q + 1) & 2) << 30));
    sn = __int_as_float(__float_as_int(b) ^ ((q & 2) << 30));
}

namespace p64 {

constexpr int kUnitTab = 2048;     // entries e^{-2 pi i m / 2048}

// Adding and taking off 1.5 2^52 rounds |x| < 2^51 to an integer, whose low 32 bits are those
// of the sum: two FP64 instructions, against a conversion each way that the pipe takes no
// faster (0.6 % slower passes and 1 % slower geometry).
constexpr double kMagic = 6755399441055744.0;

// floor(x) as double and its low 32 bits, |x| < 2^51.
__device__ __forceinline__ double floor_int(double x, int &i) {
    const double m = __dadd_rd(x, kMagic);
    i = __double2loint(m);
    return __dsub_rn(m, kMagic);
}

// e^{-2 pi i cyc}: the nearest table entry e^{-2 pi i m / 2048} times e^{-i d},
// |d| <= pi / 2048, by its Taylor series (the first terms left out are d^7/5040
// and d^6/720, below 2e-20): 13 FP64 operations.  cyc need not be reduced; from 2^38
// cycles on, where the rounding above ends, it is.
__device__ __forceinline__ double2 unit_phase(const double2 *__restrict__ tab, double cyc) {
    if ((__double2hiint(cyc) & 0x7fffffff) >= 0x42500000) cyc -= floor(cyc);   // also infinities and NaN
    const double x = fma(cyc, (double)kUnitTab, kMagic);
    const int m = __double2loint(x);
    const double e = fma(cyc, (double)kUnitTab, -(x - kMagic));   // exact, |e| <= 1/2
    constexpr double h = 6.283185307179586476925286766559 / kUnitTab;   // d = h e
    const double q = e * e;
    const double s = e * fma(q, fma(q, h * h * h * h * h / 120.0, -h * h * h / 6.0), h);
    const double c = fma(q, fma(q, h * h * h * h / 24.0, -h * h / 2.0), 1.0);
    const double2 t = __ldg(tab + (m & (kUnitTab - 1)));
    return make_double2(fma(t.x, c, t.y * s), fma(t.y, c, -(t.x * s)));
}

}  // namespace p64
}  // namespace fstat
