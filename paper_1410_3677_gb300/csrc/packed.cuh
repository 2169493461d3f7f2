// Packed FP32 arithmetic for the search passes: two independent complex values
// per "PC" (their real parts in one float2, their imaginary parts in another),
// computed with the paired single-precision instructions of sm_100-class GPUs
// (add/sub/mul/fma .f32x2).  A paired instruction occupies the FP32 pipe for
// as long as two scalar ones but takes one issue slot, and the FFT passes are
// bound by instruction issue, so two transforms of the same shape (two jobs of
// a stage, or the two halves of a decimation-in-frequency split) run for the
// issue cost of one.  The DFT codelets on arrays of PC are in fft_codelets.cuh.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace fstat {
namespace pk {

__device__ __forceinline__ unsigned long long as_u64(float2 a) {
    return *reinterpret_cast<unsigned long long *>(&a);
}
__device__ __forceinline__ float2 as_f2(unsigned long long u) { return *reinterpret_cast<float2 *>(&u); }

__device__ __forceinline__ float2 padd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 psub(float2 a, float2 b) {
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(as_u64(a)), "l"(as_u64(b)));
    return as_f2(r);
}
__device__ __forceinline__ float2 pmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 bc(float v) { return make_float2(v, v); }

struct PC {
    float2 re, im;
};

__device__ __forceinline__ PC add(const PC &a, const PC &b) { return {padd(a.re, b.re), padd(a.im, b.im)}; }
__device__ __forceinline__ PC sub(const PC &a, const PC &b) { return {psub(a.re, b.re), psub(a.im, b.im)}; }
// a + i^K b (K mod 4): a quarter turn costs no instruction, only a choice of
// add or subtract per component
template <int K>
__device__ __forceinline__ PC add_rot(const PC &a, const PC &b) {
    constexpr int k = ((K % 4) + 4) % 4;
    if constexpr (k == 0) return add(a, b);
    else if constexpr (k == 2) return sub(a, b);
    else if constexpr (k == 1) return {psub(a.re, b.im), padd(a.im, b.re)};
    else return {padd(a.re, b.im), psub(a.im, b.re)};
}

__device__ __forceinline__ float2 pneg(float2 a) { return make_float2(-a.x, -a.y); }
// x w for run-time twiddles w (one per lane of the pair); the negation is an
// operand modifier of the paired multiply, not an instruction
__device__ __forceinline__ PC cmul(const PC &x, const PC &w) {
    return {pfma(x.re, w.re, pmul(x.im, pneg(w.im))), pfma(x.re, w.im, pmul(x.im, w.re))};
}

}  // namespace pk
}  // namespace fstat
