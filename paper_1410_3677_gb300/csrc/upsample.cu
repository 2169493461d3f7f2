// Per-band steps of a search: the noise variance's partial sums, the FP32 form's
// ephemeris split, and the U-fold FFT upsample of the narrow-band series
// ("resampling ... using the FFT and splines", Sect. 2).
//
// The upsampled series is x itself at sub-phase 0 and, at sub-phase s of U, the
// band-limited interpolant at k + s/U: a circular convolution of x with the
// periodic sinc d(t), t = k + s/U,
//   n odd   d(t) = sin(pi t) / (n sin(pi t / n)),
//   n even  d(t) = sin(pi t) cos(pi t / n) / (n sin(pi t / n))  (Nyquist bin split).
// Its transform depends on n and U alone, so the plan holds it and a search does
// one forward and one inverse real transform per sub-phase in FP64, of length
// M = n when n is a power of two, else of the power of two M >= 2n - 1 (the linear
// convolution that holds the circular one).  A real transform of length M is a
// complex one of H = M/2 points on z[m] = x[2m] + i x[2m + 1]; the even/odd
// untangling, the product with the kernel's transform K and the tangling back are
// linear in Z[k] and conj(Z[H - k]) and collapse to
//   Z'[k] = alpha_k Z[k] + beta_k conj(Z[H - k]),
//   alpha = (K_k + K_{k+H})/2 - sin(pi k/H)/2 (K_k - K_{k+H}),
//   beta  = i cos(pi k/H)/2 (K_k - K_{k+H})            (both divided by H).
// Three launches, H = N1 N2: columns (k2 -> l2); pairs of rows (l2, N2 - l2), which
// hold each other's partners: k1 -> l1, the product, and straight back l1 -> k1;
// columns (l2 -> k2) and the interleaved store.
// The FP64 units (1/64 of the FP32 rate) bound the three.
// Measured on GB300 for a band of a search (with BandInputs), U = 2, against a
// Bluestein transform each way (23 launches): n = 86 164 390 -> 54 us, n = 344 656
// 1521 -> 186 us, n = 4096 113 -> 26 us.
#include <math.h>

#include <algorithm>

#include "dfloat.cuh"
#include "fstat_internal.h"
#include "reduce64.cuh"

namespace fstat {

namespace {

constexpr int kTS = 128;           // target threads per CTA
constexpr int kMinLogH = kMinLogN - 1, kMaxLogH = kMaxLogN - 1;

// Sequences of length M on M / 4 threads each, 4 elements per thread: 2^17 points make a
// thousand warps, enough for the FP64 units of all SM quarters (16 elements per thread
// made 256 warps and left half of the units idle).
template <int LOGH, int PASS>      // PASS 1: columns (length N2), 2: rows (length N1)
struct CfgU {
    static constexpr int N1 = 1 << (LOGH / 2), N2 = 1 << (LOGH - LOGH / 2), H = 1 << LOGH;
    static constexpr int M = PASS == 1 ? N2 : N1;
    static constexpr int TPS = M / 4;                                    // threads per sequence
    static constexpr int COUNT = PASS == 1 ? N1 : N2;                    // sequences
    static constexpr int F0 = kTS / TPS, F1 = F0 < COUNT ? F0 : COUNT;
    static constexpr int F = F1 < PASS ? PASS : F1;                      // sequences per CTA (rows: pairs)
    static constexpr int THREADS = F * TPS;
    static constexpr int TILES = COUNT / F;
    static constexpr int LD = M + M / 8;                                 // exchange row
    static constexpr size_t SMEM = (size_t)F * (LD + (PASS == 2 ? M : 0)) * sizeof(double2);
    static_assert(M >= 8 && THREADS <= 1024, "tile shape");
};

__device__ __forceinline__ int padu(int i) { return i + (i >> 3); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 conj_if(bool c, double2 a) { return c ? make_double2(a.x, -a.y) : a; }

// DFT of one sequence (direction DIR), Stockham radix 4 and a last radix 2 for odd log2 M:
// ld(i) gives element i, st(i, v) takes output i; thread j < M / 4; w[k] = e^{-2 pi i k / M};
// ex is the sequence's exchange row.  HALF: the upper half of the inputs is zero (not read).
template <int M, int DIR, class LD, class ST>
__device__ __forceinline__ void dft_seq(int j, const double2 *__restrict__ w, double2 *ex, bool half, LD ld, ST st) {
    constexpr int Q = M / 4;
    double2 x[4];
    x[0] = ld(j);
    x[1] = ld(j + Q);
    if (half) {
        const double2 t = DIR < 0 ? make_double2(x[1].y, -x[1].x) : make_double2(-x[1].y, x[1].x);   // DIR i x1
        const double2 a = x[0], b = x[1];
        x[0] = cadd(a, b);
        x[1] = cadd(a, t);
        x[2] = csub(a, b);
        x[3] = csub(a, t);
    } else {
        x[2] = ld(j + 2 * Q);
        x[3] = ld(j + 3 * Q);
    }
#pragma unroll
    for (int Ns = 1; Ns <= Q; Ns *= 4) {
        const int k = j & (Ns - 1);
        if (Ns > 1) {
#pragma unroll
            for (int r = 0; r < 4; ++r) x[r] = ex[padu(j + r * Q)];
            __syncthreads();
#pragma unroll
            for (int r = 1; r < 4; ++r) x[r] = cmul(x[r], conj_if(DIR > 0, __ldg(w + k * r * (Q / Ns))));
        }
        if (Ns > 1 || !half) {
            const double2 t0 = cadd(x[0], x[2]), t1 = csub(x[0], x[2]), t2 = cadd(x[1], x[3]), d = csub(x[1], x[3]);
            const double2 t3 = DIR < 0 ? make_double2(d.y, -d.x) : make_double2(-d.y, d.x);
            x[0] = cadd(t0, t2);
            x[1] = cadd(t1, t3);
            x[2] = csub(t0, t2);
            x[3] = csub(t1, t3);
        }
        const int o = (j - k) * 4 + k;
        if (Ns * 4 == M) {
#pragma unroll
            for (int r = 0; r < 4; ++r) st(o + r * Ns, x[r]);
            return;
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) ex[padu(o + r * Ns)] = x[r];
        __syncthreads();
    }
    // last stage of radix 2 (Ns = M / 2): butterflies j and j + M / 4
    double2 y[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int k = j + h * Q;
        const double2 a = ex[padu(k)], b = cmul(ex[padu(k + 2 * Q)], conj_if(DIR > 0, __ldg(w + k)));
        y[h] = csub(a, b);
        x[h] = cadd(a, b);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        st(j + h * Q, x[h]);
        st(j + h * Q + 2 * Q, y[h]);
    }
}

// The band's other inputs, by kSigmaParts blocks beside the first upsample kernel's (or alone
// when U = 1; a launch of their own took 5 us): part `part` of the sum of x^2 (compensated)
// and of the ephemeris split into double-float pairs (r2 null in the FP64 form).
struct BandInputs {
    const double *x;
    int64_t n;
    double *parts;
    const double *r;
    DF *r2;
    __device__ __forceinline__ void run(int part) const {
        __shared__ double sh[32];
        const int T = (int)blockDim.x;
        const int64_t first = (int64_t)part * T + threadIdx.x, step = (int64_t)kSigmaParts * T;
        if (r2)
            for (int64_t i = first; i < n; i += step)
#pragma unroll
                for (int c = 0; c < 3; ++c) r2[c * n + i] = df_from_double(r[3 * i + c]);
        KahanD k;
        for (int64_t i = first; i < n; i += step) k.add(x[i] * x[i]);
        const double v = warp_sum(k.s - k.c);
        if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int w = 0; w < (T + 31) / 32; ++w) t += sh[w];
            parts[part] = t;
        }
    }
};

template <typename TO>
__global__ void k_copy_series(BandInputs in, TO *__restrict__ xu) {
    in.run(blockIdx.x);
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < in.n; k += (int64_t)gridDim.x * blockDim.x)
        xu[k] = (TO)in.x[k];
}

__device__ __forceinline__ double2 *up_smem() {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    return reinterpret_cast<double2 *>(smem_raw);
}

// Columns c of z[m] = x[2m] + i x[2m + 1] (zero beyond n), times W_H^{c l2}, to A[l2][c].
template <int LOGH>
__global__ void __launch_bounds__(CfgU<LOGH, 1>::THREADS)
k_up_columns(const double *__restrict__ x, int64_t n, double2 *__restrict__ A, const double2 *__restrict__ tw,
             const double2 *__restrict__ w, BandInputs in) {
    using C = CfgU<LOGH, 1>;
    if (blockIdx.x >= C::TILES) return in.run(blockIdx.x - C::TILES);
    const int f = (int)threadIdx.x % C::F, j = (int)threadIdx.x / C::F;   // consecutive threads: adjacent columns
    const int c = blockIdx.x * C::F + f;
    auto ld = [&](int i) {
        const int64_t m = c + (int64_t)C::N1 * i;
        if (2 * m + 1 < n) return __ldg(reinterpret_cast<const double2 *>(x) + m);
        return make_double2(2 * m < n ? __ldg(x + 2 * m) : 0.0, 0.0);
    };
    auto st = [&](int i, double2 v) {
        const int64_t q = (int64_t)i * C::N1 + c;
        A[q] = cmul(v, __ldg(tw + q));
    };
    // z[m] = 0 from m = H / 2 on when n <= M / 2 (M = 2 H)
    dft_seq<C::M, -1>(j, w, up_smem() + f * C::LD, n <= C::H, ld, st);
}

// Rows: a CTA holds pairs p of rows, p and N2 - p, or the two that are their own partners, 0
// and N2 / 2; sequence 2 q is the first row of its q-th pair, 2 q + 1 the second.
template <class C>
__device__ __forceinline__ int row_of(int tile, int f) {
    const int p = tile * (C::F / 2) + (f >> 1);
    return (f & 1) == 0 ? p : p == 0 ? C::N2 / 2 : C::N2 - p;
}

// k1 -> l1 of the pairs, alpha Z + beta conj(Z[H - k]), l1 -> k1 times conj(W_H^{k1 l2}).
// With k = N2 l1 + l2 the partner of (l2, l1) is (N2 - l2, N1 - 1 - l1), or (0, -l1 mod N1)
// in row 0.  grid.z: sub-phases; A is read by every one, B holds one region each.
template <int LOGH>
__global__ void __launch_bounds__(CfgU<LOGH, 2>::THREADS)
k_up_rows(const double2 *__restrict__ A, double2 *__restrict__ B, const double2 *__restrict__ ab,
          const double2 *__restrict__ tw, const double2 *__restrict__ w) {
    using C = CfgU<LOGH, 2>;
    const int f = (int)threadIdx.x / C::TPS, j = (int)threadIdx.x % C::TPS;
    const int l2 = row_of<C>(blockIdx.x, f);
    double2 *ex = up_smem() + f * C::LD, *Z = up_smem() + C::F * C::LD;   // Z: [f][N1]
    const int64_t row = (int64_t)l2 * C::N1;
    dft_seq<C::M, -1>(j, w, ex, false, [&](int i) { return A[row + i]; }, [&](int i, double2 v) { Z[f * C::N1 + i] = v; });
    __syncthreads();
    const bool self = l2 == 0 || l2 == C::N2 / 2;
    const double2 *mine = Z + f * C::N1, *other = self ? mine : Z + (f ^ 1) * C::N1;
    const double2 *t = ab + 2 * ((int64_t)C::H * blockIdx.z + row);
    auto ld = [&](int i) {
        const double2 z = mine[i], q = other[l2 == 0 ? (C::N1 - i) & (C::N1 - 1) : C::N1 - 1 - i];
        const double2 al = __ldg(t + 2 * i), be = __ldg(t + 2 * i + 1);
        return make_double2(al.x * z.x - al.y * z.y + be.x * q.x + be.y * q.y,
                            al.x * z.y + al.y * z.x + be.y * q.x - be.x * q.y);
    };
    double2 *out = B + (int64_t)C::H * blockIdx.z + row;
    dft_seq<C::M, 1>(j, w, ex, false, ld, [&](int i, double2 v) {
        const double2 e = __ldg(tw + row + i);
        out[i] = make_double2(v.x * e.x + v.y * e.y, v.y * e.x - v.x * e.y);
    });
}

// Plan time: the kernel's transform in the rows' order.
template <int LOGH>
__global__ void __launch_bounds__(CfgU<LOGH, 2>::THREADS)
k_up_rows_forward(const double2 *__restrict__ A, double2 *__restrict__ Z, const double2 *__restrict__ w) {
    using C = CfgU<LOGH, 2>;
    const int f = (int)threadIdx.x / C::TPS, j = (int)threadIdx.x % C::TPS;
    const int64_t row = (int64_t)row_of<C>(blockIdx.x, f) * C::N1;
    dft_seq<C::M, -1>(j, w, up_smem() + f * C::LD, false, [&](int i) { return A[row + i]; },
                      [&](int i, double2 v) { Z[row + i] = v; });
}

// l2 -> k2 of the columns and the interleaved store xu[U k + s]; the launch's sub-phase 1
// also stores sub-phase 0, x itself.
template <int LOGH, typename TO>
__global__ void __launch_bounds__(CfgU<LOGH, 1>::THREADS)
k_up_output(const double2 *__restrict__ B, const double *__restrict__ x, TO *__restrict__ xu, int64_t n, int U,
            const double2 *__restrict__ w) {
    using C = CfgU<LOGH, 1>;
    const int f = (int)threadIdx.x % C::F, j = (int)threadIdx.x / C::F;
    const int c = blockIdx.x * C::F + f, s = (int)blockIdx.z + 1;
    const double2 *in = B + (int64_t)C::H * blockIdx.z + c;
    auto st = [&](int i, double2 y) {
        const int64_t m = c + (int64_t)C::N1 * i, k = 2 * m;
        if (k >= n) return;
        const bool odd = k + 1 < n;
        if (U == 2 && odd) {   // four neighbours of the upsampled series
            const double2 v = __ldg(reinterpret_cast<const double2 *>(x) + m);
            if constexpr (sizeof(TO) == 4) {
                reinterpret_cast<float4 *>(xu)[m] = make_float4((float)v.x, (float)y.x, (float)v.y, (float)y.y);
            } else {
                reinterpret_cast<double2 *>(xu)[2 * m] = make_double2(v.x, y.x);
                reinterpret_cast<double2 *>(xu)[2 * m + 1] = make_double2(v.y, y.y);
            }
            return;
        }
        xu[U * k + s] = (TO)y.x;
        if (odd) xu[U * (k + 1) + s] = (TO)y.y;
        if (s == 1) {
            xu[U * k] = (TO)__ldg(x + k);
            if (odd) xu[U * (k + 1)] = (TO)__ldg(x + k + 1);
        }
    };
    dft_seq<C::M, 1>(j, w, up_smem() + f * C::LD, false, [&](int i) { return in[(int64_t)i * C::N1]; }, st);
}

// The convolution kernel d(m + s/U) on the M-point circle: h[m], m < n, and (linear
// convolution, M > n) h[M - m] for the negative lags.  |m + s/U| <= n/2 by the
// periodicity of d, so that sin(pi t / n) keeps its relative precision.
__global__ void k_up_kernel(double *__restrict__ h, int64_t n, int64_t M, int U, int s) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= M) return;
    double v = 0.0;
    if (i < n || i > M - n) {
        int64_t m = i < n ? i : i - M;      // lag
        if (2 * m > n) m -= n;
        if (2 * m < -n) m += n;
        const double a = (double)((int64_t)U * m + s) / (double)((int64_t)U * n);   // t / n
        double sn, cs;
        sincospi(a, &sn, &cs);
        v = sinpi((double)s / (double)U) / ((double)n * sn);
        if (m & 1) v = -v;
        if (n % 2 == 0) v *= cs;
    }
    h[i] = v;
}

__global__ void k_up_alpha_beta(const double2 *__restrict__ Z, double2 *__restrict__ ab, int logh) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t H = int64_t(1) << logh, N1 = int64_t(1) << (logh / 2), N2 = H / N1;
    if (i >= H) return;
    const int64_t l2 = i / N1, l1 = i % N1, k = N2 * l1 + l2, kp = (H - k) & (H - 1);
    const double2 z = Z[i], zp = Z[(kp % N2) * N1 + kp / N2];
    const double2 q = make_double2(zp.x, -zp.y);
    double sn, cs;
    sincospi((double)k / (double)H, &sn, &cs);
    // p = (1 - i W)/2, p' = (1 + i W)/2, W = e^{-i pi k/H}: K_k = p Z + p' Q, K_{k+H} = p' Z + p Q
    const double2 p = make_double2(0.5 * (1.0 - sn), -0.5 * cs), pp = make_double2(0.5 * (1.0 + sn), 0.5 * cs);
    auto mul = [](double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); };
    const double2 pz = mul(p, z), ppq = mul(pp, q), ppz = mul(pp, z), pq = mul(p, q);
    const double2 K0 = make_double2(pz.x + ppq.x, pz.y + ppq.y), K1 = make_double2(ppz.x + pq.x, ppz.y + pq.y);
    const double2 S = make_double2(K0.x + K1.x, K0.y + K1.y), D = make_double2(K0.x - K1.x, K0.y - K1.y);
    const double g = 0.5 / (double)H;
    ab[2 * i] = make_double2(g * (S.x - sn * D.x), g * (S.y - sn * D.y));
    ab[2 * i + 1] = make_double2(-g * cs * D.y, g * cs * D.x);
}

// W_H^{k1 l2}, [l2][k1]
__global__ void k_up_twiddle(double2 *__restrict__ t, int logh) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t H = int64_t(1) << logh, N1 = int64_t(1) << (logh / 2);
    if (i >= H) return;
    double s, c;
    sincospi(2.0 * (double)((i % N1) * (i / N1)) / (double)H, &s, &c);
    t[i] = make_double2(c, -s);
}

inline unsigned blocks(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

template <class K>
void smem_limit(K k, size_t bytes) {
    if (bytes > 48 * 1024) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int LOGH>
void forward_columns(const double *x, int64_t n, double2 *A, const UpsampleTables &t, const BandInputs *in,
                     cudaStream_t s) {
    using C1 = CfgU<LOGH, 1>;
    auto k1 = k_up_columns<LOGH>;
    smem_limit(k1, C1::SMEM);
    k1<<<C1::TILES + (in ? kSigmaParts : 0), C1::THREADS, C1::SMEM, s>>>(x, n, A, t.tw, t.w_cols, in ? *in : BandInputs{});
}

template <int LOGH>
int run_t(const BandDev &b, int U, void *xu, bool fp32, const UpsampleTables &t, double2 *scratch,
          const BandInputs &in, cudaStream_t s) {
    using C1 = CfgU<LOGH, 1>;
    using C2 = CfgU<LOGH, 2>;
    double2 *A = scratch, *B = scratch + C1::H;
    forward_columns<LOGH>(b.x, b.n, A, t, &in, s);
    auto k2 = k_up_rows<LOGH>;
    smem_limit(k2, C2::SMEM);
    k2<<<dim3(C2::TILES, 1, (unsigned)(U - 1)), C2::THREADS, C2::SMEM, s>>>(A, B, t.ab, t.tw, t.w_rows);
    const dim3 grid(C1::TILES, 1, (unsigned)(U - 1));
    if (fp32) {
        auto k3 = k_up_output<LOGH, float>;
        smem_limit(k3, C1::SMEM);
        k3<<<grid, C1::THREADS, C1::SMEM, s>>>(B, b.x, (float *)xu, b.n, U, t.w_cols);
    } else {
        auto k3 = k_up_output<LOGH, double>;
        smem_limit(k3, C1::SMEM);
        k3<<<grid, C1::THREADS, C1::SMEM, s>>>(B, b.x, (double *)xu, b.n, U, t.w_cols);
    }
    return 3;
}

template <int LOGH>
int tables_t(int64_t n, int U, UpsampleTables &t, double2 *ab, double2 *tw, double2 *scratch, cudaStream_t s) {
    using C2 = CfgU<LOGH, 2>;
    constexpr int64_t H = C2::H;
    double2 *A = scratch, *Z = scratch + 2 * H;
    double *h = reinterpret_cast<double *>(scratch + H);   // M = 2H doubles
    k_up_twiddle<<<blocks(H, 256), 256, 0, s>>>(tw, LOGH);
    t.tw = tw;
    t.ab = ab;
    auto k2 = k_up_rows_forward<LOGH>;
    smem_limit(k2, C2::SMEM);
    for (int sub = 1; sub < U; ++sub) {
        k_up_kernel<<<blocks(2 * H, 256), 256, 0, s>>>(h, n, 2 * H, U, sub);
        forward_columns<LOGH>(h, 2 * H, A, t, nullptr, s);
        k2<<<C2::TILES, C2::THREADS, C2::SMEM, s>>>(A, Z, t.w_rows);
        k_up_alpha_beta<<<blocks(H, 256), 256, 0, s>>>(Z, ab + 2 * H * (sub - 1), LOGH);
    }
    return 1 + 4 * (U - 1);
}

// f.template operator()<LOGH>() for the runtime logh
template <int L, class F>
int dispatch(int logh, F &&f) {
    if constexpr (L > kMaxLogH) return -1;
    else return logh == L ? f.template operator()<L>() : dispatch<L + 1>(logh, f);
}

struct RunOp {
    const BandDev &b;
    int U;
    void *xu;
    bool fp32;
    const UpsampleTables &t;
    double2 *scratch;
    const BandInputs &in;
    cudaStream_t s;
    template <int L> int operator()() const { return run_t<L>(b, U, xu, fp32, t, scratch, in, s); }
};
struct TablesOp {
    int64_t n;
    int U;
    UpsampleTables &t;
    double2 *ab, *tw, *scratch;
    cudaStream_t s;
    template <int L> int operator()() const { return tables_t<L>(n, U, t, ab, tw, scratch, s); }
};

}  // namespace

int upsample_logh(int64_t n) {
    const bool pow2 = (n & (n - 1)) == 0 && n >= (int64_t(1) << kMinLogN);
    int lm = kMinLogN;
    while ((int64_t(1) << lm) < (pow2 ? n : 2 * n - 1)) ++lm;
    return lm - 1;
}

int64_t upsample_scratch(int logh, int U) { return (int64_t(1) << logh) * (U > 3 ? U : 3); }

int launch_upsample_tables(int64_t n, int U, UpsampleTables &t, double2 *ab, double2 *tw, void *scratch,
                           cudaStream_t s) {
    return dispatch<kMinLogH>(t.logh, TablesOp{n, U, t, ab, tw, reinterpret_cast<double2 *>(scratch), s});
}

int launch_prologue(const Plan &p, const BandDev &b, int U, void *xu, bool xu_fp32, cudaStream_t s) {
    const BandInputs in{b.x, b.n, p.sigma_parts, b.r, static_cast<DF *>(b.r2)};
    if (U == 1) {
        if (xu_fp32) k_copy_series<float><<<kSigmaParts, 256, 0, s>>>(in, (float *)xu);
        else k_copy_series<double><<<kSigmaParts, 256, 0, s>>>(in, (double *)xu);
        return 1;
    }
    return dispatch<kMinLogH>(b.up.logh, RunOp{b, U, xu, xu_fp32, b.up, reinterpret_cast<double2 *>(p.scratch), in, s});
}

}  // namespace fstat
