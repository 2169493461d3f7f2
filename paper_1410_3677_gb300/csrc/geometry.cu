// Per-sky steps of the search (Sect. 2, Fig. 1; the per-band ones are in upsample.cu):
//   per sky:  Roemer delay nhat . r, detector time of every barycentric sample,
//             amplitude modulations a(t), b(t), Keys-cubic resampling and the
//             band-offset phase demodulation ("amplitude and phase
//             demodulation", "resampling", done once per sky position), and the
//             FP64 compensated sums S_aa, S_bb, S_ab.
#include <math.h>

#include "dfloat.cuh"
#include "fstat_internal.h"
#include "reduce64.cuh"
#include "unit_phase.cuh"

namespace fstat {

namespace {

constexpr double kTwoPi = 6.283185307179586476925286766559;
constexpr double kOmegaR = kTwoPi / 86164.0905;   // sidereal rotation rate, rad/s

// The FP32 form's three S terms at once: each warp adds its 32 terms of each in
// FP32 (relative error ~1e-7), one barrier, then three threads add the block's
// warp sums in FP64 and write the block's partials (blockDim.x = 256); the
// blocks' partials are then added with compensation.  The S sums thus keep FP64
// accumulation where the term count is large, and spend no FP64 instructions per
// sample.
__device__ void block_sum3_f(float a, float b, float c, double *sh, double *out) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
        c += __shfl_down_sync(0xffffffffu, c, o);
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) {
        sh[w] = (double)a;
        sh[8 + w] = (double)b;
        sh[16 + w] = (double)c;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double t = 0.0;
#pragma unroll
        for (int i = 0; i < 8; ++i) t += sh[8 * threadIdx.x + i];
        out[threadIdx.x] = t;
    }
}

// ------------------------------------------------------------------ geometry
// FP32 form: the delay of sample j reduced once, in double-float arithmetic
// (FP64 runs at 1/64 of the FP32 rate on GB300), to the sample shift
// d_j / dt = I + phi (integer part exact, fraction in FP32) and to the
// band-offset phase f_off d_j mod 1 with its increment f_off (d_{j+1} - d_j), so
// that the detector-time inversion and the phase interpolation run in integer
// and FP32 arithmetic (positions and phases to ~1e-7 samples and cycles).
struct DelayRec {
    int I;
    float phi, psi, dpsi;
};

struct GeoArgs {
    const double *r;
    const double *d;          // per-sample delays of the sky batch, [sky][stride]
    const DelayRec *dr;       // FP32 form: the same as shift records
    int64_t d_stride;
    const void *xu;
    int64_t m_up;
    int U;
    int64_t n;
    double dt, inv_dt, f_off, phi0;
    int dt_pow2;              // dt is a power of two: t / dt == t * inv_dt exactly
    const double2 *unit_tab;  // FP64 form
    const SkyConst *sky;
    int64_t s0;
    void *w;
    int64_t w_stride;
    double *partials;
    int nblk;
    double *dbg_y, *dbg_a, *dbg_b;
    uint8_t *dbg_mask;
};

// The delay chain is evaluated with explicitly rounded operations (no fused
// multiply-add): the band-offset phase 2 pi f_off d reaches ~1e5 rad, so the
// rounding of d decides the FP64 agreement of F at the 1e-10 level.
__device__ __forceinline__ double delay_at(const double *__restrict__ r, const SkyConst &sc,
                                           int64_t j) {
    return __dadd_rn(__dadd_rn(__dmul_rn(sc.nx, r[3 * j]), __dmul_rn(sc.ny, r[3 * j + 1])),
                     __dmul_rn(sc.nz, r[3 * j + 2]));
}

// Linear interpolation of the delay at fractional sample u from the per-sample
// delays dk; the end segments extend beyond the data.
__device__ __forceinline__ double delay_lin(const double *__restrict__ dk, int64_t n, double u) {
    int64_t j = (int64_t)floor(u);
    j = j < 0 ? 0 : (j > n - 2 ? n - 2 : j);
    const double f = __dsub_rn(u, (double)j);
    const double d0 = dk[j], d1 = dk[j + 1];
    return __dadd_rn(d0, __dmul_rn(f, __dsub_rn(d1, d0)));
}

// Roemer delay nhat . r_k of every sample of skies [s0, s0 + gridDim.y).
__global__ void __launch_bounds__(256) k_delays(const double *__restrict__ r,
                                                const SkyConst *__restrict__ sky, int64_t s0,
                                                int64_t n, int64_t stride,
                                                double *__restrict__ d) {
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int sl = blockIdx.y;
    if (k < n) d[(int64_t)sl * stride + k] = delay_at(r, sky[s0 + sl], k);
}

// Shift records of every sample of skies [s0, s0 + gridDim.y): the delay
// nhat . r_k and its reductions in double-float arithmetic (about 2^-46
// relative: 1e-11 samples and 1e-9 cycles at the delays and offsets of a
// search, against the 6e-8 of the FP32 results); d_{k+1} of the phase
// increment comes from the next thread (the block's first thread evaluates
// the one past the block).  The increment of the last sample is never used
// (the interpolation segment index is <= n - 2).
__global__ void __launch_bounds__(256) k_delays_split(const DF *__restrict__ r2,
                                                      const SkyConst *__restrict__ sky, int64_t s0,
                                                      int64_t n, int64_t stride, DF inv_dt, DF f_off,
                                                      int phase, DelayRec *__restrict__ out) {
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int sl = blockIdx.y;
    __shared__ DF dsh[257];
    const float *nf = sky[s0 + sl].nf;
    const DF nx{nf[0], nf[1]}, ny{nf[2], nf[3]}, nz{nf[4], nf[5]};
    auto delay = [&](int64_t j) {
        const DF *rj = r2 + 3 * j;
        return df_add(df_add(df_mul(nx, rj[0]), df_mul(ny, rj[1])), df_mul(nz, rj[2]));
    };
    const DF dk = k < n ? delay(k) : DF{0.f, 0.f};
    DelayRec o;
    float phi;
    o.I = (int)df_split_floor(df_mul(dk, inv_dt), &phi);
    o.phi = phi;
    o.psi = 0.f;
    o.dpsi = 0.f;
    if (phase) {   // uniform: no phase records for a band at zero offset
        dsh[threadIdx.x] = dk;
        if (threadIdx.x == 0) {
            const int64_t kn = k + blockDim.x;
            dsh[blockDim.x] = kn < n ? delay(kn) : DF{0.f, 0.f};
        }
        __syncthreads();
        float psi;
        df_split_floor(df_mul(f_off, dk), &psi);
        o.psi = psi;
        if (k + 1 < n) {
            const DF dd = df_add(dsh[threadIdx.x + 1], df_neg(dk));
            o.dpsi = (f_off.hi + f_off.lo) * (dd.hi + dd.lo);
        }
    }
    if (k < n) out[(int64_t)sl * stride + k] = o;
}

__global__ void __launch_bounds__(256) k_geometry(GeoArgs g) {
    __shared__ double sh[24];
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int sl = blockIdx.y;
    float saa_f = 0.f, sbb_f = 0.f, sab_f = 0.f;
    // the sky's constants in FP32, converted once per block
    __shared__ float cf[12];
    if (threadIdx.x < 12) {
        const SkyConst &sc = g.sky[g.s0 + sl];
        const int i = threadIdx.x;
        cf[i] = i < 5 ? (float)sc.A[i] : i < 9 ? (float)sc.B[i - 5]
              : i == 9 ? (float)(sc.alpha - g.phi0) : i == 10 ? (float)g.dt : 0.f;
    }
    __syncthreads();
    if (k < g.n) {
        // detector time t of barycentric sample k, t = k dt - d(k dt - d(k dt)),
        // as u = t / dt = A - F1: A an exact integer, F1 an FP32 fraction
        const int n = (int)g.n, kk = (int)k;
        const DelayRec *dr = g.dr + (int64_t)sl * g.d_stride;
        const DelayRec rk = dr[kk];
        const int a0 = kk - rk.I;                       // u0 = a0 - phi_k
        const int j0 = min(max(a0 - 1, 0), n - 2);
        const float f0 = (float)(a0 - j0) - rk.phi;     // u0 - j0
        const DelayRec p0 = dr[j0], p1 = dr[j0 + 1];
        const float F1 = p0.phi + f0 * ((float)(p1.I - p0.I) + (p1.phi - p0.phi));
        const int A = kk - p0.I;
        const float fl1 = floorf(-F1);
        int j = A + (int)fl1;
        float f = -F1 - fl1;                            // u - j in [0, 1)
        const int jc = min(max(j, 0), n - 2);
        f += (float)(j - jc);
        j = jc;
        const bool valid = F1 <= (float)A && F1 >= (float)(A - (n - 1));
        // band-offset phase at t, cycles: psi_j + f dpsi_j (mod 1)
        const DelayRec q0 = dr[j];
        const float cyc = q0.psi + f * q0.dpsi;
        const float frs = cyc - rintf(cyc);
        // hour angle h = alpha - phi0 - Omega_r t (|h| < 20 rad, error ~1e-6 rad
        // from t rounded to FP32)
        const float uf = (float)A - F1;
        const float hr = cf[9] - (float)kOmegaR * (uf * cf[10]);
        float s1, c1;
        sincosf(hr, &s1, &c1);
        const float c2 = c1 * c1 - s1 * s1, s2 = 2.f * s1 * c1;
        const float av = cf[0] * c2 + cf[1] * s2 + cf[2] * c1 + cf[3] * s1 + cf[4];
        const float bv = cf[5] * c2 + cf[6] * s2 + cf[7] * c1 + cf[8] * s1;
        float yr = 0.f, yi = 0.f;
        if (valid) {
            // Keys cubic (a = -1/2) at p = U u = U A - U F1 on the upsampled series,
            // periodic indexing (only tap -1 and taps >= U n wrap, a single step)
            const float up = -(float)g.U * F1;
            const float upf = floorf(up);
            const float mu = up - upf;
            const int64_t i0 = (int64_t)g.U * A + (int64_t)upf - 1;
            const float w0 = ((-0.5f * mu + 1.f) * mu - 0.5f) * mu;
            const float w1 = (1.5f * mu - 2.5f) * mu * mu + 1.f;
            const float w2 = ((-1.5f * mu + 2.f) * mu + 0.5f) * mu;
            const float w3 = (0.5f * mu - 0.5f) * mu * mu;
            const float *xu = (const float *)g.xu;
            float x4[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int64_t v = i0 + q;
                x4[q] = xu[v < 0 ? v + g.m_up : (v >= g.m_up ? v - g.m_up : v)];
            }
            const float v = w0 * x4[0] + w1 * x4[1] + w2 * x4[2] + w3 * x4[3];
            float sp, cp;
            sincospif(2.f * frs, &sp, &cp);
            yr = v * cp;
            yi = -v * sp;
            saa_f = av * av;
            sbb_f = bv * bv;
            sab_f = av * bv;
        }
        float4 *w = (float4 *)g.w + (int64_t)sl * g.w_stride;
        w[k] = make_float4(yr * av, yi * av, yr * bv, yi * bv);
        if (g.dbg_y) {
            g.dbg_y[2 * k] = yr; g.dbg_y[2 * k + 1] = yi;
            g.dbg_a[k] = av; g.dbg_b[k] = bv; g.dbg_mask[k] = valid;
        }
    }
    block_sum3_f(saa_f, sbb_f, sab_f, sh, g.partials + ((int64_t)sl * g.nblk + blockIdx.x) * 3);
}

// FP64 form.  Bound by the FP64 units (1/64 of the FP32 rate), so it spends FP64
// instructions only where the result needs them: one hour-angle and one phase
// factor from the unit-phase table, the S sums over kGeo64 samples of a thread
// before the block's reduction, and the delay in samples as a multiplication when
// dt is a power of two (the same value as the division).
// Measured at n = 86 164: 50 -> 18.2 us per sky position (one position a launch before).
constexpr int kGeo64 = 4;
__global__ void __launch_bounds__(256) k_geometry64(GeoArgs g) {
    __shared__ double sh[24];
    const int sl = blockIdx.y;
    double saa = 0.0, sbb = 0.0, sab = 0.0;
    const SkyConst &sc = g.sky[g.s0 + sl];
    const double *dd = g.d + (int64_t)sl * g.d_stride;
    const bool pow2 = g.dt_pow2 != 0;
    auto in_samples = [&](double t) { return pow2 ? __dmul_rn(t, g.inv_dt) : __ddiv_rn(t, g.dt); };
    int64_t k = blockIdx.x * (int64_t)(256 * kGeo64) + threadIdx.x;
#pragma unroll 1
    for (int it = 0; it < kGeo64 && k < g.n; ++it, k += 256) {
        // detector time t of barycentric sample k: t = k dt - d(k dt - d(k dt)),
        // in the oracle's rounding sequence, for 1e-10 agreement of F
        const double u0 = __dsub_rn((double)k, in_samples(dd[k]));
        const double d1 = delay_lin(dd, g.n, u0);
        const double u = __dsub_rn((double)k, in_samples(d1));
        const double d2 = delay_lin(dd, g.n, u);
        const bool valid = (u >= 0.0) && (u <= (double)(g.n - 1));
        const double h = sc.alpha - (g.phi0 + kOmegaR * (u * g.dt));
        const double turns = h * (1.0 / kTwoPi);
        const double2 eh = p64::unit_phase(g.unit_tab, turns - floor(turns));
        const double c1 = eh.x, s1 = -eh.y;
        const double c2 = c1 * c1 - s1 * s1, s2 = 2.0 * s1 * c1;
        const double av = sc.A[0] * c2 + sc.A[1] * s2 + sc.A[2] * c1 + sc.A[3] * s1 + sc.A[4];
        const double bv = sc.B[0] * c2 + sc.B[1] * s2 + sc.B[2] * c1 + sc.B[3] * s1;
        double yr = 0.0, yi = 0.0;
        if (valid) {
            // Keys cubic (a = -1/2) on the upsampled series, periodic indexing: taps
            // i0 .. i0 + 3 around floor(p); inside the window p lies in [0, U (n - 1)],
            // so only i0 = -1 and indices >= U n wrap (a single step)
            const double p = (double)g.U * u;
            const double pf = floor(p);
            const int64_t i0 = (int64_t)pf - 1;
            const double *xu = (const double *)g.xu;
            double x4[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int64_t v = i0 + q;
                x4[q] = xu[v < 0 ? v + g.m_up : (v >= g.m_up ? v - g.m_up : v)];
            }
            const double mu = p - pf;
            const double w0 = ((-0.5 * mu + 1.0) * mu - 0.5) * mu;
            const double w1 = (1.5 * mu - 2.5) * mu * mu + 1.0;
            const double w2 = ((-1.5 * mu + 2.0) * mu + 0.5) * mu;
            const double w3 = (0.5 * mu - 0.5) * mu * mu;
            const double v = w0 * x4[0] + w1 * x4[1] + w2 * x4[2] + w3 * x4[3];
            // band-offset phase, cycles, reduced in FP64
            const double cyc = __dmul_rn(g.f_off, d2);
            const double2 e = p64::unit_phase(g.unit_tab, __dsub_rn(cyc, floor(cyc)));
            yr = v * e.x;
            yi = v * e.y;
            saa = fma(av, av, saa);
            sbb = fma(bv, bv, sbb);
            sab = fma(av, bv, sab);
        }
        // {y a, y b} as two double2 (32 bytes per sample)
        double2 *w = (double2 *)g.w + 2 * ((int64_t)sl * g.w_stride + k);
        w[0] = make_double2(yr * av, yi * av);
        w[1] = make_double2(yr * bv, yi * bv);
        if (g.dbg_y) {
            g.dbg_y[2 * k] = yr; g.dbg_y[2 * k + 1] = yi;
            g.dbg_a[k] = av; g.dbg_b[k] = bv; g.dbg_mask[k] = valid;
        }
    }
    double *o = g.partials + ((int64_t)sl * g.nblk + blockIdx.x) * 3;
    const double ta = block_sum256(saa, sh);
    const double tb = block_sum256(sbb, sh);
    const double tab = block_sum256(sab, sh);
    if (threadIdx.x == 0) {
        o[0] = ta; o[1] = tb; o[2] = tab;
    }
}

// S sums per sky (Kahan over the block partials) and the normalisations
// 1/(sigma^2 S_aa), 1/(sigma^2 S_bb).  Warp w adds term w % 3 over the w / 3-th
// quarter of the partials: with one warp for all three terms the dependent FP64
// chain over 337 partials took 10 us a launch.
// A further warp finishes the noise variance from the band's partials.
constexpr int kNormWarps = 12;
__global__ void __launch_bounds__(32 * (kNormWarps + 1))
k_reduce_norms(const double *__restrict__ partials, int nblk, const double *__restrict__ sigma_parts, int64_t n,
               double user_sigma2, double *__restrict__ S, double *__restrict__ norm, int full) {
    const int sl = blockIdx.x;
    __shared__ double sh[kNormWarps + 1];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    KahanD k;
    if (w == kNormWarps)
        for (int i = l; i < kSigmaParts; i += 32) k.add(sigma_parts[i]);
    else
        for (int i = 32 * (w / 3) + l; i < nblk; i += 32 * (kNormWarps / 3)) k.add(partials[((int64_t)sl * nblk + i) * 3 + w % 3]);
    const double v = warp_sum(k.s - k.c);
    if (l == 0) sh[w] = v;
    __syncthreads();
    double out[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        out[c] = 0.0;
#pragma unroll
        for (int q = 0; q < kNormWarps / 3; ++q) out[c] += sh[3 * q + c];
    }
    if (threadIdx.x == 0) {
        const double s2 = user_sigma2 > 0.0 ? user_sigma2 : sh[kNormWarps] / (double)n;
        S[3 * sl] = out[0];
        S[3 * sl + 1] = out[1];
        S[3 * sl + 2] = out[2];
        // F = na |F_a|^2 + nb |F_b|^2 + nab Re(F_a conj F_b)
        double na = 0.0, nb = 0.0, nab = 0.0;
        if (full) {
            const double D = out[0] * out[1] - out[2] * out[2];
            if (D > 0.0) {
                na = out[1] / (s2 * D);
                nb = out[0] / (s2 * D);
                nab = -2.0 * out[2] / (s2 * D);
            }
        } else {
            na = out[0] > 0.0 ? 1.0 / (s2 * out[0]) : 0.0;
            nb = out[1] > 0.0 ? 1.0 / (s2 * out[1]) : 0.0;
        }
        norm[kNormStride * sl] = na;
        norm[kNormStride * sl + 1] = nb;
        norm[kNormStride * sl + 2] = nab;
        norm[kNormStride * sl + 3] = 0.0;
        // FP32 copies for the FP32 epilogues (no conversion in every CTA)
        float *nf = reinterpret_cast<float *>(norm + kNormStride * sl + 4);
        nf[0] = (float)na;
        nf[1] = (float)nb;
        nf[2] = (float)nab;
        nf[3] = 0.f;
    }
}

inline unsigned blocks(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }
// blocks of a geometry launch per sky position, each leaving one partial of the S sums
inline int geo_blocks(int64_t n, bool fp32) { return (int)blocks(n, fp32 ? 256 : 256 * kGeo64); }

}  // namespace

// ================================================================== launchers
int launch_geometry(const Plan &p, const BandDev &b, int64_t s0, int64_t ns, bool fp32,
                    void *w, double *dbg_y, double *dbg_a, double *dbg_b, uint8_t *dbg_mask,
                    cudaStream_t s) {
    GeoArgs g;
    g.r = b.r;
    g.d = p.dbuf;
    g.dr = reinterpret_cast<const DelayRec *>(p.dbuf);
    g.d_stride = p.n_max;
    g.xu = b.xu;
    g.U = p.desc.upsample;
    g.m_up = (int64_t)g.U * b.n;
    g.n = b.n;
    g.dt = b.dt;
    g.inv_dt = 1.0 / b.dt;
    int e2 = 0;
    g.dt_pow2 = frexp(b.dt, &e2) == 0.5 && isnormal(g.inv_dt);
    g.unit_tab = p.unit_tab;
    g.f_off = b.f_off;
    g.phi0 = b.phi0;
    g.sky = p.sky;
    g.s0 = s0;
    g.w = w;
    g.w_stride = p.w_stride;
    g.partials = p.partials;
    g.nblk = geo_blocks(b.n, fp32);
    g.dbg_y = dbg_y;
    g.dbg_a = dbg_a;
    g.dbg_b = dbg_b;
    g.dbg_mask = dbg_mask;
    dim3 grid(g.nblk, (unsigned)ns);
    if (fp32) {
        k_delays_split<<<grid, 256, 0, s>>>(static_cast<const DF *>(b.r2), p.sky, s0, b.n, p.n_max,
                                            df_from_double(g.inv_dt), df_from_double(b.f_off),
                                            b.f_off != 0.0 ? 1 : 0, reinterpret_cast<DelayRec *>(p.dbuf));
        k_geometry<<<grid, 256, 0, s>>>(g);
    } else {
        k_delays<<<dim3(blocks(b.n, 256), (unsigned)ns), 256, 0, s>>>(b.r, p.sky, s0, b.n, p.n_max, p.dbuf);
        k_geometry64<<<grid, 256, 0, s>>>(g);
    }
    return 2;
}

int launch_reduce_norms(const Plan &p, const BandDev &b, int64_t ns, double *norm, cudaStream_t s) {
    k_reduce_norms<<<(unsigned)ns, 32 * (kNormWarps + 1), 0, s>>>(
        p.partials, geo_blocks(b.n, p.desc.form == FSTAT_FP32_BATCHED), p.sigma_parts, b.n, p.desc.sigma2, p.S, norm,
        p.desc.statistic == FSTAT_F_FULL ? 1 : 0);
    return 1;
}

}  // namespace fstat
