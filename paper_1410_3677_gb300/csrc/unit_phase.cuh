// Unit phases in FP64 from a table, for the FP64 form's kernels.
#pragma once

#include <cuda_runtime.h>

namespace fstat {
namespace p64 {

constexpr int kUnitTab = 2048;     // entries e^{-2 pi i m / 2048}

// e^{-2 pi i fr}: the nearest table entry e^{-2 pi i m / 2048} times e^{-i d},
// |d| <= pi / 2048, by its Taylor series (the first terms left out are d^7/5040
// and d^6/720, below 2e-20): 14 FP64 operations.
__device__ __forceinline__ double2 unit_phase(const double2 *__restrict__ tab, double fr) {
    const double x = fr * (double)kUnitTab;
    const int m = __double2int_rn(x);
    const double d = (x - (double)m) * (6.283185307179586476925286766559 / kUnitTab);
    const double d2 = d * d;
    const double s = d * fma(d2, fma(d2, 1.0 / 120.0, -1.0 / 6.0), 1.0);
    const double c = fma(d2, fma(d2, 1.0 / 24.0, -0.5), 1.0);
    const double2 e = __ldg(tab + (m & (kUnitTab - 1)));
    return make_double2(fma(e.x, c, e.y * s), fma(e.y, c, -(e.x * s)));
}

}  // namespace p64
}  // namespace fstat
