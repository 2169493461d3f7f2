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
// The FP64 units (1/64 of the FP32 rate) bound the three; the tiles are one warp's
// work or two, so that even short series spread over the SMs.
// Measured on GB300 for a band of a search (with k_band_inputs), U = 2, against a
// Bluestein transform each way (23 launches): n = 86 164 390 -> 92 us, n = 344 656
// 1521 -> 188 us, n = 4096 113 -> 55 us.
#include <math.h>

#include <algorithm>

#include "fft_engine.cuh"
#include "dfloat.cuh"
#include "fstat_internal.h"
#include "reduce64.cuh"

namespace fstat {

namespace {

constexpr int kTS = 32;            // target threads per CTA
constexpr int kMinLogH = kMinLogN - 1, kMaxLogH = kMaxLogN - 1;

template <int LOGH, int PASS>      // PASS 1: columns (length N2), 2: rows (length N1)
struct CfgU {
    static constexpr int N1 = 1 << (LOGH / 2), N2 = 1 << (LOGH - LOGH / 2), H = 1 << LOGH;
    static constexpr int M = PASS == 1 ? N2 : N1;
    static constexpr int PAIRS = (PASS == 1 ? N1 : N2) / 2;
    static constexpr int EH = 8;
    static constexpr int F0 = kTS * EH / M;
    static constexpr int F = F0 < 1 ? 1 : (F0 < PAIRS ? F0 : PAIRS);   // pairs per tile
    static constexpr int THREADS = F * M / EH;
    static constexpr int TILES = PAIRS / F;
    static constexpr size_t PASS_SMEM = eng::smem_bytes<double, M, F>();
    static constexpr size_t SMEM = PASS_SMEM + (PASS == 2 ? 2 * F * M * sizeof(double2) : 0);
};

// Columns 2f, 2f + 1 of the tile: z[m] = x[2m] + i x[2m + 1], zero beyond n.
template <class C>
struct SeriesLoad {
    const double *x;
    int64_t n;
    int c0;
    __device__ __forceinline__ double2 z(int64_t m) const {
        if (2 * m + 1 < n) return __ldg(reinterpret_cast<const double2 *>(x) + m);
        return make_double2(2 * m < n ? __ldg(x + 2 * m) : 0.0, 0.0);
    }
    template <int R, int JPF>
    __device__ __forceinline__ void load(int f, int j, double *ra, double *ia, double *rb, double *ib) const {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int64_t m = c0 + 2 * f + (int64_t)C::N1 * (j + r * JPF);
            const double2 a = z(m), b = z(m + 1);
            ra[r] = a.x; ia[r] = a.y; rb[r] = b.x; ib[r] = b.y;
        }
    }
};

// Transposed store A[l2][k1] with the four-step twiddle W_H^{k1 l2} (table in the
// same order).
template <class C>
struct ColumnStore {
    double2 *A;
    const double2 *tw;
    int c0;
    template <int R, int JPF>
    __device__ __forceinline__ void store(int f, int j, double *ra, double *ia, double *rb, double *ib) const {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int64_t i = (int64_t)(j + r * JPF) * C::N1 + c0 + 2 * f;
            const double2 ta = __ldg(tw + i), tb = __ldg(tw + i + 1);
            A[i] = make_double2(ra[r] * ta.x - ia[r] * ta.y, ra[r] * ta.y + ia[r] * ta.x);
            A[i + 1] = make_double2(rb[r] * tb.x - ib[r] * tb.y, rb[r] * tb.y + ib[r] * tb.x);
        }
    }
};

// Rows of pair p: p and N2 - p, or the two that are their own partners, 0 and N2/2.
template <class C>
struct RowPair {
    int p0;
    __device__ __forceinline__ int a(int f) const { return p0 + f; }
    __device__ __forceinline__ int b(int f) const { return p0 + f == 0 ? C::N2 / 2 : C::N2 - (p0 + f); }
};

template <class C>
struct RowLoad {
    const double2 *A;
    RowPair<C> rows;
    template <int R, int JPF>
    __device__ __forceinline__ void load(int f, int j, double *ra, double *ia, double *rb, double *ib) const {
        const double2 *a = A + (int64_t)rows.a(f) * C::N1, *b = A + (int64_t)rows.b(f) * C::N1;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const double2 va = a[j + r * JPF], vb = b[j + r * JPF];
            ra[r] = va.x; ia[r] = va.y; rb[r] = vb.x; ib[r] = vb.y;
        }
    }
};

// Row transforms parked in shared memory (natural order).
template <class C>
struct RowPark {
    double2 *z;   // [2 f + (0: a, 1: b)][N1]
    template <int R, int JPF>
    __device__ __forceinline__ void store(int f, int j, double *ra, double *ia, double *rb, double *ib) const {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            z[(2 * f) * C::N1 + j + r * JPF] = make_double2(ra[r], ia[r]);
            z[(2 * f + 1) * C::N1 + j + r * JPF] = make_double2(rb[r], ib[r]);
        }
    }
};

// alpha Z + beta conj(Z[H - k]); with k = N2 l1 + l2 the partner of (l2, l1) is
// (N2 - l2, N1 - 1 - l1), or (0, -l1 mod N1) in row 0.
template <class C>
struct ProductLoad {
    const double2 *z;
    const double2 *ab;   // [l2][l1][2]
    RowPair<C> rows;
    __device__ __forceinline__ double2 one(double2 z0, double2 q, const double2 *t) const {
        const double2 al = __ldg(t), be = __ldg(t + 1);
        return make_double2(al.x * z0.x - al.y * z0.y + be.x * q.x + be.y * q.y,
                            al.x * z0.y + al.y * z0.x + be.y * q.x - be.x * q.y);
    }
    template <int R, int JPF>
    __device__ __forceinline__ void load(int f, int j, double *ra, double *ia, double *rb, double *ib) const {
        const double2 *za = z + (2 * f) * C::N1, *zb = za + C::N1;
        const int la = rows.a(f), lb = rows.b(f);
        const bool self = la == 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int l1 = j + r * JPF;
            const double2 qa = self ? za[(C::N1 - l1) & (C::N1 - 1)] : zb[C::N1 - 1 - l1];
            const double2 qb = self ? zb[C::N1 - 1 - l1] : za[C::N1 - 1 - l1];
            const double2 a = one(za[l1], qa, ab + 2 * ((int64_t)la * C::N1 + l1));
            const double2 b = one(zb[l1], qb, ab + 2 * ((int64_t)lb * C::N1 + l1));
            ra[r] = a.x; ia[r] = a.y; rb[r] = b.x; ib[r] = b.y;
        }
    }
};

// Inverse rows back to global memory, times conj(W_H^{k1 l2}).
template <class C>
struct RowStore {
    double2 *B;
    const double2 *tw;
    RowPair<C> rows;
    template <int R, int JPF>
    __device__ __forceinline__ void store(int f, int j, double *ra, double *ia, double *rb, double *ib) const {
        const int64_t a = (int64_t)rows.a(f) * C::N1, b = (int64_t)rows.b(f) * C::N1;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int k1 = j + r * JPF;
            const double2 ta = __ldg(tw + a + k1), tb = __ldg(tw + b + k1);
            B[a + k1] = make_double2(ra[r] * ta.x + ia[r] * ta.y, ia[r] * ta.x - ra[r] * ta.y);
            B[b + k1] = make_double2(rb[r] * tb.x + ib[r] * tb.y, ib[r] * tb.x - rb[r] * tb.y);
        }
    }
};

template <class C>
struct ColumnLoad {
    const double2 *B;
    int c0;
    template <int R, int JPF>
    __device__ __forceinline__ void load(int f, int j, double *ra, double *ia, double *rb, double *ib) const {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int64_t i = (int64_t)(j + r * JPF) * C::N1 + c0 + 2 * f;
            const double2 a = B[i], b = B[i + 1];
            ra[r] = a.x; ia[r] = a.y; rb[r] = b.x; ib[r] = b.y;
        }
    }
};

// xu[U k + s] = y[k]; the launch of sub-phase 1 also stores sub-phase 0, x itself.
template <class C, typename TO>
struct SeriesStore {
    const double *x;
    TO *xu;
    int64_t n;
    int U, s, c0;
    __device__ __forceinline__ void put(int64_t m, double ye, double yo) const {
        const int64_t k = 2 * m;
        if (k >= n) return;
        const bool odd = k + 1 < n;
        if (U == 2 && odd) {   // four neighbours of the upsampled series
            const double2 v = __ldg(reinterpret_cast<const double2 *>(x) + m);
            if constexpr (sizeof(TO) == 4) {
                reinterpret_cast<float4 *>(xu)[m] = make_float4((float)v.x, (float)ye, (float)v.y, (float)yo);
            } else {
                reinterpret_cast<double2 *>(xu)[2 * m] = make_double2(v.x, ye);
                reinterpret_cast<double2 *>(xu)[2 * m + 1] = make_double2(v.y, yo);
            }
            return;
        }
        xu[U * k + s] = (TO)ye;
        if (odd) xu[U * (k + 1) + s] = (TO)yo;
        if (s == 1) {
            xu[U * k] = (TO)__ldg(x + k);
            if (odd) xu[U * (k + 1)] = (TO)__ldg(x + k + 1);
        }
    }
    template <int R, int JPF>
    __device__ __forceinline__ void store(int f, int j, double *ra, double *ia, double *rb, double *ib) const {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int64_t m = c0 + 2 * f + (int64_t)C::N1 * (j + r * JPF);
            put(m, ra[r], ia[r]);
            put(m + 1, rb[r], ib[r]);
        }
    }
};

__device__ __forceinline__ unsigned char *up_smem() {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    return smem_raw;
}

template <int LOGH>
__global__ void __launch_bounds__(CfgU<LOGH, 1>::THREADS)
k_up_columns(const double *__restrict__ x, int64_t n, double2 *__restrict__ A, const double2 *__restrict__ tw,
             const double *__restrict__ w) {
    using C = CfgU<LOGH, 1>;
    const int c0 = blockIdx.x * 2 * C::F;
    SeriesLoad<C> ld{x, n, c0};
    ColumnStore<C> st{A, tw, c0};
    eng::run_pass<double, C::M, C::F, C::EH, -1, eng::kMapFJ>(ld, st, w);
}

// grid.z: sub-phases.  A is read by every sub-phase, B holds one region each.
template <int LOGH>
__global__ void __launch_bounds__(CfgU<LOGH, 2>::THREADS)
k_up_rows(const double2 *__restrict__ A, double2 *__restrict__ B, const double2 *__restrict__ ab,
          const double2 *__restrict__ tw, const double *__restrict__ w) {
    using C = CfgU<LOGH, 2>;
    const RowPair<C> rows{(int)blockIdx.x * C::F};
    double2 *z = reinterpret_cast<double2 *>(up_smem() + C::PASS_SMEM);
    RowLoad<C> ld{A, rows};
    RowPark<C> park{z};
    eng::run_pass<double, C::M, C::F, C::EH, -1, eng::kMapJ>(ld, park, w);
    __syncthreads();
    ProductLoad<C> pl{z, ab + 2 * (int64_t)C::H * blockIdx.z, rows};
    RowStore<C> st{B + (int64_t)C::H * blockIdx.z, tw, rows};
    eng::run_pass<double, C::M, C::F, C::EH, 1, eng::kMapJ>(pl, st, w);
}

// Plan time: the kernel's transform in the rows' order.
template <int LOGH>
__global__ void __launch_bounds__(CfgU<LOGH, 2>::THREADS)
k_up_rows_forward(const double2 *__restrict__ A, double2 *__restrict__ Z, const double *__restrict__ w) {
    using C = CfgU<LOGH, 2>;
    const RowPair<C> rows{(int)blockIdx.x * C::F};
    double2 *z = reinterpret_cast<double2 *>(up_smem() + C::PASS_SMEM);
    RowLoad<C> ld{A, rows};
    RowPark<C> park{z};
    eng::run_pass<double, C::M, C::F, C::EH, -1, eng::kMapJ>(ld, park, w);
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * C::F * C::N1; i += C::THREADS) {
        const int q = i / C::N1, l1 = i % C::N1;
        Z[(int64_t)(q & 1 ? rows.b(q >> 1) : rows.a(q >> 1)) * C::N1 + l1] = z[i];
    }
}

template <int LOGH, typename TO>
__global__ void __launch_bounds__(CfgU<LOGH, 1>::THREADS)
k_up_output(const double2 *__restrict__ B, const double *__restrict__ x, TO *__restrict__ xu, int64_t n, int U,
            const double *__restrict__ w) {
    using C = CfgU<LOGH, 1>;
    const int c0 = blockIdx.x * 2 * C::F;
    ColumnLoad<C> ld{B + (int64_t)C::H * blockIdx.z, c0};
    SeriesStore<C, TO> st{x, xu, n, U, (int)blockIdx.z + 1, c0};
    eng::run_pass<double, C::M, C::F, C::EH, 1, eng::kMapFJ>(ld, st, w);
}

template <typename TO>
__global__ void k_copy_series(const double *__restrict__ x, int64_t n, TO *__restrict__ xu) {
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k < n) xu[k] = (TO)x[k];
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

// Partial sums of x^2 (compensated), one per block of the first kSigmaParts, and
// the ephemeris as double-float pairs (FP32 form; r2 null otherwise): both only
// read the band's inputs, one launch.
__global__ void __launch_bounds__(256) k_band_inputs(const double *__restrict__ x, int64_t n,
                                                     double *__restrict__ partials, const double *__restrict__ r,
                                                     DF *__restrict__ r2) {
    __shared__ double sh[8];
    if (r2)
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < 3 * n; i += (int64_t)gridDim.x * blockDim.x)
            r2[i] = df_from_double(r[i]);
    if (blockIdx.x >= kSigmaParts) return;
    KahanD k;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)kSigmaParts * blockDim.x)
        k.add(x[i] * x[i]);
    const double s = block_sum256(k.s - k.c, sh);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

inline unsigned blocks(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

template <class K>
void smem_limit(K k, size_t bytes) {
    if (bytes > 48 * 1024) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int LOGH>
void forward_columns(const double *x, int64_t n, double2 *A, const UpsampleTables &t, cudaStream_t s) {
    using C1 = CfgU<LOGH, 1>;
    auto k1 = k_up_columns<LOGH>;
    smem_limit(k1, C1::SMEM);
    k1<<<C1::TILES, C1::THREADS, C1::SMEM, s>>>(x, n, A, t.tw, t.w_cols);
}

template <int LOGH>
int run_t(const BandDev &b, int U, void *xu, bool fp32, const UpsampleTables &t, double2 *scratch, cudaStream_t s) {
    using C1 = CfgU<LOGH, 1>;
    using C2 = CfgU<LOGH, 2>;
    double2 *A = scratch, *B = scratch + C1::H;
    forward_columns<LOGH>(b.x, b.n, A, t, s);
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
        forward_columns<LOGH>(h, 2 * H, A, t, s);
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
    cudaStream_t s;
    template <int L> int operator()() const { return run_t<L>(b, U, xu, fp32, t, scratch, s); }
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

int launch_band_inputs(const BandDev &b, double *sigma_parts, cudaStream_t s) {
    const unsigned grid = b.r2 ? std::max<unsigned>(kSigmaParts, std::min<unsigned>(1024, blocks(3 * b.n, 256))) : kSigmaParts;
    k_band_inputs<<<grid, 256, 0, s>>>(b.x, b.n, sigma_parts, b.r, static_cast<DF *>(b.r2));
    return 1;
}

int launch_upsample(const Plan &p, const BandDev &b, int U, void *xu, bool xu_fp32, cudaStream_t s) {
    if (U == 1) {
        if (xu_fp32) k_copy_series<float><<<blocks(b.n, 256), 256, 0, s>>>(b.x, b.n, (float *)xu);
        else k_copy_series<double><<<blocks(b.n, 256), 256, 0, s>>>(b.x, b.n, (double *)xu);
        return 1;
    }
    return dispatch<kMinLogH>(b.up.logh, RunOp{b, U, xu, xu_fp32, b.up, reinterpret_cast<double2 *>(p.scratch), s});
}

}  // namespace fstat
