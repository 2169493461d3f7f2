// Forward DFT codelets of 4 to 32 points on registers, for scalars (float, double) and for
// packed pairs (packed.cuh), natural order in and out.
//
// A twiddle multiply before a butterfly is written W = i^k c (1 - i t), c = cos, t = tan of an
// angle within 45 degrees: the factor (1 - i t) costs two multiply-adds, the quarter turn
// nothing, and c goes into the butterfly's additions, which become multiply-adds (the
// radix-4 form of Linzer and Feig, "Implementation of efficient FFT algorithms on fused
// multiply-add architectures", 1993).  A twiddled radix-4 butterfly takes 22 instructions
// instead of 28, a 16-point DFT 144 instead of 160, the 32-point one 376 instead of 432.
#pragma once

#include <cuda_runtime.h>

#include "packed.cuh"

namespace fstat {
namespace cod {

// cos(pi m / 16), |m| <= 8
__host__ __device__ constexpr double cos16(int m) {
    const int a = m < 0 ? -m : m;
    return a == 0 ? 1.0 : a == 1 ? 0.98078528040323044913 : a == 2 ? 0.92387953251128675613
         : a == 3 ? 0.83146961230254523708 : a == 4 ? 0.70710678118654752440
         : a == 5 ? 0.55557023301960222474 : a == 6 ? 0.38268343236508977173
         : a == 7 ? 0.19509032201612826785 : 0.0;
}
__host__ __device__ constexpr double tan16(int m) { return m < 0 ? -tan16(-m) : cos16(8 - m) / cos16(m); }
// W_32^e = i^turn (1 - i tan16(dev)) cos16(dev), |dev| <= 4
__host__ __device__ constexpr int quarters(int e) { return (e + 4) / 8; }
__host__ __device__ constexpr int turn(int e) { return (4 - quarters(e) % 4) % 4; }
__host__ __device__ constexpr int dev(int e) { return e - 8 * quarters(e); }

// ------------------------------------------------------------------ operations
template <typename T>
struct SC {
    T re, im;
    using real = T;
};
__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }

// a + i^K b
template <int K, typename T>
__device__ __forceinline__ SC<T> add_rot(const SC<T> &a, const SC<T> &b) {
    constexpr int k = ((K % 4) + 4) % 4;
    if constexpr (k == 0) return {a.re + b.re, a.im + b.im};
    else if constexpr (k == 1) return {a.re - b.im, a.im + b.re};
    else if constexpr (k == 2) return {a.re - b.re, a.im - b.im};
    else return {a.re + b.im, a.im - b.re};
}
// a + g i^K b
template <int K, typename T>
__device__ __forceinline__ SC<T> mad_rot(const SC<T> &a, double g, const SC<T> &b) {
    constexpr int k = ((K % 4) + 4) % 4;
    const T c = (T)g;
    if constexpr (k == 0) return {fma_(b.re, c, a.re), fma_(b.im, c, a.im)};
    else if constexpr (k == 1) return {fma_(b.im, -c, a.re), fma_(b.re, c, a.im)};
    else if constexpr (k == 2) return {fma_(b.re, -c, a.re), fma_(b.im, -c, a.im)};
    else return {fma_(b.im, c, a.re), fma_(b.re, -c, a.im)};
}
// x (1 - i t)
template <typename T>
__device__ __forceinline__ SC<T> twist(const SC<T> &x, double t) {
    const T c = (T)t;
    return {fma_(x.im, c, x.re), fma_(x.re, -c, x.im)};
}

using pk::PC;   // a + i^K b: pk::add_rot
template <int K>
__device__ __forceinline__ PC mad_rot(const PC &a, double g, const PC &b) {
    constexpr int k = ((K % 4) + 4) % 4;
    const float2 c = pk::bc((float)g);   // negated operands are modifiers: one constant serves both signs
    if constexpr (k == 0) return {pk::pfma(b.re, c, a.re), pk::pfma(b.im, c, a.im)};
    else if constexpr (k == 1) return {pk::pfma(pk::pneg(b.im), c, a.re), pk::pfma(b.re, c, a.im)};
    else if constexpr (k == 2) return {pk::pfma(pk::pneg(b.re), c, a.re), pk::pfma(pk::pneg(b.im), c, a.im)};
    else return {pk::pfma(b.im, c, a.re), pk::pfma(pk::pneg(b.re), c, a.im)};
}
__device__ __forceinline__ PC twist(const PC &x, double t) {
    const float2 c = pk::bc((float)(t < 0 ? -t : t));
    return t < 0 ? PC{pk::pfma(pk::pneg(x.im), c, x.re), pk::pfma(x.re, c, x.im)}
                 : PC{pk::pfma(x.im, c, x.re), pk::pfma(pk::pneg(x.re), c, x.im)};
}

// The factor 1 - i t of W_32^E.
template <int E, class V>
__device__ __forceinline__ V unscaled(const V &x) {
    constexpr int d = dev(E);
    if constexpr (d == 0) return x;
    else if constexpr (d == 4) return add_rot<3>(x, x);
    else if constexpr (d == -4) return add_rot<1>(x, x);
    else return twist(x, tan16(d));
}
// a + i^K c_E b, c_E the cosine of W_32^E's remaining angle
template <int E, int K, class V>
__device__ __forceinline__ V mad_cos(const V &a, const V &b) {
    if constexpr (dev(E) == 0) return add_rot<K>(a, b);
    else return mad_rot<K>(a, cos16(dev(E)), b);
}

// ------------------------------------------------------------------ butterflies
// (x0, x1) <- x0 +- W_32^E x1
template <int E, class V>
__device__ __forceinline__ void comb2(V &x0, V &x1) {
    const V u = unscaled<E>(x1), a = x0;
    x0 = mad_cos<E, turn(E)>(a, u);
    x1 = mad_cos<E, turn(E) + 2>(a, u);
}

// 4-point DFT of x0, W_32^E1 x1, W_32^E2 x2, W_32^E3 x3.  NZ: inputs from NZ on are zero
// (not read); HALF: only the outputs 0 and 1.
template <int E1, int E2, int E3, int NZ = 4, bool HALF = false, class V>
__device__ __forceinline__ void comb4(V &x0, V &x1, V &x2, V &x3) {
    static_assert(NZ >= 1 && NZ <= 4, "non-zero inputs");
    constexpr int K1 = turn(E1), K2 = turn(E2), K3 = turn(E3);
    const V a = x0;
    if constexpr (NZ == 1) {
        x1 = x2 = x3 = a;
    } else {
        const V u1 = unscaled<E1>(x1);
        V t0 = a, t1 = a, t2 = u1, t3 = u1;   // t2, t3 still to be scaled by i^K1 c_E1
        if constexpr (NZ >= 3) {
            const V u2 = unscaled<E2>(x2);
            t0 = mad_cos<E2, K2>(a, u2);
            t1 = mad_cos<E2, K2 + 2>(a, u2);
        }
        if constexpr (NZ == 4) {
            const V u3 = unscaled<E3>(x3);
            constexpr int d1 = dev(E1) < 0 ? -dev(E1) : dev(E1), d3 = dev(E3) < 0 ? -dev(E3) : dev(E3);
            if constexpr (d1 == d3) {
                t2 = add_rot<K3 - K1>(u1, u3);
                t3 = add_rot<K3 - K1 + 2>(u1, u3);
            } else {
                constexpr double rho = cos16(d3) / cos16(d1);
                t2 = mad_rot<K3 - K1>(u1, rho, u3);
                t3 = mad_rot<K3 - K1 + 2>(u1, rho, u3);
            }
        }
        x0 = mad_cos<E1, K1>(t0, t2);
        x1 = mad_cos<E1, K1 + 3>(t1, t3);
        if constexpr (!HALF) {
            x2 = mad_cos<E1, K1 + 2>(t0, t2);
            x3 = mad_cos<E1, K1 + 1>(t1, t3);
        }
    }
}

template <int NZ = 8, bool LOWER = false, class V>
__device__ __forceinline__ void dft8(V *x) {
    static_assert(NZ >= 2 && NZ <= 8, "each half keeps an input");
    comb4<0, 0, 0, (NZ + 1) / 2>(x[0], x[2], x[4], x[6]);
    comb4<0, 0, 0, NZ / 2>(x[1], x[3], x[5], x[7]);
    V y[8] = {x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7]};   // E_k at 2k, O_k at 2k + 1
    comb2<0>(y[0], y[1]);
    comb2<4>(y[2], y[3]);
    comb2<8>(y[4], y[5]);
    comb2<12>(y[6], y[7]);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        x[k] = y[2 * k];
        if constexpr (!LOWER) x[k + 4] = y[2 * k + 1];
    }
}

// 16-point DFT of x_m W_32^{m S}, S = 0, or S = 1 (the odd outputs of a 32-point DFT whose
// upper half of inputs is zero: there the first layer takes W_8^{m'}, the second
// W_32^{q (1 + 2k)}).  Inputs from NZ on are zero; LOWER: only the outputs 0 .. 7.
template <int S, int NZ = 16, bool LOWER = false, class V>
__device__ __forceinline__ void dft16s(V *x) {
    static_assert(NZ >= 4 && NZ <= 16, "each sub-DFT keeps an input");
    comb4<4 * S, 8 * S, 12 * S, (NZ + 3) / 4>(x[0], x[4], x[8], x[12]);
    comb4<4 * S, 8 * S, 12 * S, (NZ + 2) / 4>(x[1], x[5], x[9], x[13]);
    comb4<4 * S, 8 * S, 12 * S, (NZ + 1) / 4>(x[2], x[6], x[10], x[14]);
    comb4<4 * S, 8 * S, 12 * S, NZ / 4>(x[3], x[7], x[11], x[15]);
    // output k of sub-DFT q sits at x[4 k + q]; outputs k + 4 p of the whole
    comb4<S, 2 * S, 3 * S, 4, LOWER>(x[0], x[1], x[2], x[3]);
    comb4<S + 2, 2 * S + 4, 3 * S + 6, 4, LOWER>(x[4], x[5], x[6], x[7]);
    comb4<S + 4, 2 * S + 8, 3 * S + 12, 4, LOWER>(x[8], x[9], x[10], x[11]);
    comb4<S + 6, 2 * S + 12, 3 * S + 18, 4, LOWER>(x[12], x[13], x[14], x[15]);
    V y[16];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int p = 0; p < (LOWER ? 2 : 4); ++p) y[k + 4 * p] = x[4 * k + p];
#pragma unroll
    for (int k = 0; k < (LOWER ? 8 : 16); ++k) x[k] = y[k];
}
template <int NZ = 16, bool LOWER = false, class V>
__device__ __forceinline__ void dft16(V *x) { dft16s<0, NZ, LOWER>(x); }

// 32-point DFT: 8-point DFTs of x[4m + q], then for each k the twiddles W_32^{qk} and a
// 4-point DFT across q.  NZ = 32 or 24 (the last quarter zero).
template <int K, class V>
__device__ __forceinline__ void dft32_layer(V (&s)[4][8], V *x) {
    if constexpr (K < 8) {
        comb4<K, 2 * K, 3 * K>(s[0][K], s[1][K], s[2][K], s[3][K]);
#pragma unroll
        for (int p = 0; p < 4; ++p) x[K + 8 * p] = s[p][K];
        dft32_layer<K + 1>(s, x);
    }
}
template <int NZ = 32, class V>
__device__ __forceinline__ void dft32(V *x) {
    static_assert(NZ == 32 || NZ == 24, "known-zero inputs");
    V s[4][8];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
#pragma unroll
        for (int m = 0; m < NZ / 4; ++m) s[q][m] = x[4 * m + q];
        dft8<NZ / 4>(s[q]);
    }
    dft32_layer<0>(s, x);
}

// 32-point DFT whose inputs from NZ <= 16 on are zero: the even outputs are the 16-point DFT
// of x, the odd ones that of x_m W_32^m.
template <int NZ, class V>
__device__ __forceinline__ void dft32_half(V *x) {
    V e[16], o[16];
#pragma unroll
    for (int m = 0; m < NZ; ++m) e[m] = o[m] = x[m];
    dft16s<0, NZ>(e);
    dft16s<1, NZ>(o);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        x[2 * k] = e[k];
        x[2 * k + 1] = o[k];
    }
}

// R-point DFT, R = 4, 8, 16 or 32, of x[0 .. NZ) (the rest zero); LOWER: the first half of the
// outputs only (R <= 16).
template <int R, int NZ = R, bool LOWER = false, class V>
__device__ __forceinline__ void dft(V *x) {
    if constexpr (R == 4) comb4<0, 0, 0, NZ, LOWER>(x[0], x[1], x[2], x[3]);
    else if constexpr (R == 8) dft8<NZ, LOWER>(x);
    else if constexpr (R == 16) dft16<NZ, LOWER>(x);
    else if constexpr (NZ <= 16) dft32_half<NZ>(x);
    else dft32<NZ>(x);
}

}  // namespace cod
}  // namespace fstat
