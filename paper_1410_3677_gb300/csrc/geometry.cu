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

// ------------------------------------------------------------------ geometry
struct GeoArgs {
    const double *d;          // FP64 form: per-sample delays of the sky batch, [sky][stride]
    int64_t d_stride;
    const DF *r2;             // FP32 form: the ephemeris as double-float pairs
    DF inv_dt2, f_off2;       // 1 / dt and f_off
    DF phi0_turns, turn_dt;   // phi0 / 2 pi and Omega_r dt / 2 pi
    float w_dt;               // Omega_r dt
    const void *xu;
    int64_t m_up;
    int U;
    int64_t n;
    double dt, inv_dt, f_off, phi0;
    int dt_pow2;              // dt is a power of two: t / dt == t * inv_dt exactly
    const double2 *unit_tab;  // FP64 form
    const float4 *turn_tab;   // FP32 form
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

// Roemer delay nhat . r_k of every sample of skies [s0, s0 + gridDim.y).
__global__ void __launch_bounds__(256) k_delays(const double *__restrict__ r,
                                                const SkyConst *__restrict__ sky, int64_t s0,
                                                int64_t n, int64_t stride,
                                                double *__restrict__ d) {
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int sl = blockIdx.y;
    if (k < n) d[(int64_t)sl * stride + k] = delay_at(r, sky[s0 + sl], k);
}

// FP32 form, one launch per sky batch: delay, detector time, a(t) and b(t), the
// resampled and phase-demodulated series and the S sums of a tile of kGeo32
// consecutive samples of one sky position.
//
// The delay n . r is evaluated in double-float arithmetic (about 2^-46 relative;
// FP64 runs at 1/64 of the FP32 rate) at the tile's own samples, which only pick
// the interpolation segments, and on the window of samples where those segments
// lie, d/dt samples earlier and as long as the tile because the delay changes by
// ~1e-4 per sample.  The window stays in shared memory: no delay records go
// through memory, and the two dependent look-ups per sample are shared-memory
// reads.  From d_j the detector-time inversion runs on d_j / dt = I + phi (I an exact
// integer, phi in FP32) and the band-offset phase on f_off d_j mod 1 plus the FP32
// increment, as before.  A segment outside the window (an ephemeris that moves
// by more than the margin within a tile) is evaluated directly.
// The hour angle is a rotation by the tile's reference angle (once per tile, its cosine
// and sine as double-float pairs) and the small angle from it (Taylor series), instead of a sincos.
// Rounded to FP32, the reference's error is the same for a whole tile: with the four tiles of
// 4096 samples it modulated a(t) and b(t) in steps, and the bins beside a line of 2F = 400 were off
// by 7.6e-6 (1.0e-5 over 128 positions); with the pairs 1.2e-6 (3.0e-6), against 2.8e-6 (4.4e-6)
// of a sincos per sample.  It costs 1 % (63.4 -> 64.0 us per 64 positions).
// Bound by instruction issue.  Measured at n = 86 164 per 64 positions, f_off != 0, with the
// norms: 110 -> 64 us (delay records through memory and one sincos per sample before).
constexpr int kGeo32 = 1024;                 // samples per tile
constexpr int kGeoThreads = 256, kGeoPer = kGeo32 / kGeoThreads;
constexpr int kGeoMargin = 4;                // samples before the first segment
constexpr int kGeoWin = kGeo32 + 12;         // window length

// r2: the x, y and z of every sample, one component after the other (coalesced).
__device__ __forceinline__ DF delay_df(const DF *__restrict__ r2, int n, DF nx, DF ny, DF nz, int j) {
    return df_dot3(nx, r2[j], ny, r2[n + j], nz, r2[2 * n + j]);
}

// x = I + f: I the integer nearest to the high part, |f| <= 1/2 up to the low part.
__device__ __forceinline__ int df_split_near(DF x, float &f) {
    const float r = rintf(x.hi);
    f = (x.hi - r) + x.lo;
    return (int)r;
}

// cos and sin of 2 pi c by the nearest quarter turn, |c| < 2^20.
__device__ __forceinline__ void unit_f(float c, float &cs, float &sn) {
    constexpr float magic = 12582912.f;   // 1.5 2^23: the low bits of the sum are the integer
    const float qm = fmaf(c, 4.f, magic);
    fstat::unit_f(__float_as_int(qm), fmaf(qm - magic, -0.25f, c), cs, sn);
}

// cos and sin of 2 pi h as double-float pairs: the nearest of kTurnTab table entries (cos hi,
// lo, sin hi, lo) rotated by the rest, |d| <= pi / kTurnTab (first term left out d^4/24, 3e-13).
constexpr int kTurnTab = 2048;
__device__ __forceinline__ void unit_df(const float4 *__restrict__ tab, DF h, DF &c, DF &s) {
    const float x = (h.hi - rintf(h.hi)) * kTurnTab, m = rintf(x);
    const float d = ((x - m) + h.lo * kTurnTab) * (float)(kTwoPi / kTurnTab);
    const float4 t = __ldg(tab + ((int)m & (kTurnTab - 1)));
    const float cm = -0.5f * d * d, sd = fmaf(d * d, d * (-1.f / 6.f), d);
    c = df_fast_two_sum(t.x, fmaf(t.x, cm, fmaf(-t.z, sd, t.y)));
    s = df_fast_two_sum(t.z, fmaf(t.z, cm, fmaf(t.x, sd, t.w)));
}
__global__ void k_turn_table(float4 *t) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kTurnTab) return;
    double s, c;
    sincospi(2.0 * (double)i / (double)kTurnTab, &s, &c);
    const DF cd = df_from_double(c), sd = df_from_double(s);
    t[i] = make_float4(cd.hi, cd.lo, sd.hi, sd.lo);
}

// Sums over the 32 lanes of the 16 values v[0 .. 15] at once: each step halves the
// values a lane carries by trading the other half with lane ^ mask, 16 shuffles in
// place of 80.  Value i ends in lanes with bits 4 .. 1 equal to i (low bit: either).
__device__ __forceinline__ float warp_sum16(float *v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = 8; h >= 1; h >>= 1) {
        const bool up = (lane & (2 * h)) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const float keep = up ? v[i + h] : v[i], send = up ? v[i] : v[i + h];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * h);
        }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

__global__ void __launch_bounds__(kGeoThreads, 4) k_geometry(GeoArgs g) {
    __shared__ DF win[kGeoWin];
    __shared__ float4 cf[4];   // A0 .. A4, B0 .. B3, cos and sin of the reference angle: high parts, low parts
    __shared__ int s_js;
    __shared__ float sums[3][kGeoThreads / 32 * kGeoPer];
    const int n = (int)g.n, tid = threadIdx.x, sl = blockIdx.y;
    const int k0 = blockIdx.x * kGeo32;
    const SkyConst &sc = g.sky[g.s0 + sl];
    const DF nx{sc.nf[0], sc.nf[1]}, ny{sc.nf[2], sc.nf[3]}, nz{sc.nf[4], sc.nf[5]};
    const bool pow2 = g.dt_pow2 != 0;
    auto in_samples = [&](DF d) {   // d / dt; a power of two scales both parts exactly
        return pow2 ? DF{d.hi * g.inv_dt2.hi, d.lo * g.inv_dt2.hi} : df_mul(d, g.inv_dt2);
    };
    // u0 = k - d_k / dt = a0 - ph at the tile's own samples
    int a0[kGeoPer];
    float ph[kGeoPer];
#pragma unroll
    for (int i = 0; i < kGeoPer; ++i) {
        const int k = min(k0 + tid + i * kGeoThreads, n - 1);
        a0[i] = k - df_split_near(in_samples(delay_df(g.r2, n, nx, ny, nz, k)), ph[i]);
    }
    if (tid == 0) s_js = min(max(a0[0] - 1 - kGeoMargin, -(kGeoWin - 4)), n - 4);
    __syncthreads();
    const int js = s_js;
#pragma unroll
    for (int i = 0; i < (kGeoWin + kGeoThreads - 1) / kGeoThreads; ++i) {
        const int e = tid + i * kGeoThreads;
        if (e < kGeoWin) win[e] = delay_df(g.r2, n, nx, ny, nz, min(max(js + e, 0), n - 1));
    }
    const int mc = js + kGeoWin / 2;   // reference sample of the hour angle
    float *cs = reinterpret_cast<float *>(cf);
    if (tid < 9) {
        cs[tid] = tid < 5 ? (float)sc.A[tid] : (float)sc.B[tid - 5];
    } else if (tid == 32) {
        // h = alpha - phi0 - Omega_r dt mc, in turns
        const DF h = df_add(df_add(DF{sc.nf[6], sc.nf[7]}, df_neg(g.phi0_turns)),
                            df_neg(df_mul(g.turn_dt, DF{(float)mc, 0.f})));
        DF c, s;
        unit_df(g.turn_tab, h, c, s);
        cs[9] = c.hi;
        cs[10] = s.hi;
        cs[11] = c.lo;
        cs[12] = s.lo;
    }
    __syncthreads();
    float sv[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) sv[i] = 0.f;
#pragma unroll
    for (int i = 0; i < kGeoPer; ++i) {
        const int k = k0 + tid + i * kGeoThreads;
        if (k >= n) break;
        auto delay2 = [&](int j, DF &d0, DF &d1) {   // delays of samples j, j + 1
            const int e = j - js;
            if ((unsigned)e < (unsigned)(kGeoWin - 1)) {
                d0 = win[e];
                d1 = win[e + 1];
            } else {
                d0 = delay_df(g.r2, n, nx, ny, nz, j);
                d1 = delay_df(g.r2, n, nx, ny, nz, j + 1);
            }
        };
        // detector time t of barycentric sample k, t = k dt - d(k dt - d(k dt)),
        // as u = t / dt = A - F1: A an exact integer, F1 an FP32 fraction
        const int j0 = min(max(a0[i] - (ph[i] > 0.f ? 1 : 0), 0), n - 2);
        const float f0 = (float)(a0[i] - j0) - ph[i];     // u0 - j0
        DF d0, d1;
        delay2(j0, d0, d1);
        float phi0;
        const int A = k - df_split_near(in_samples(d0), phi0);
        const float F1 = phi0 + f0 * (((d1.hi - d0.hi) + (d1.lo - d0.lo)) * g.inv_dt2.hi);
        const float fl1 = floorf(-F1);
        int j = A + (int)fl1;
        float f = -F1 - fl1;                            // u - j in [0, 1)
        const int jc = min(max(j, 0), n - 2);
        f += (float)(j - jc);
        j = jc;
        // Keys cubic (a = -1/2) at p = U u = U A - U F1 on the upsampled series; inside the
        // window p lies in [0, U (n - 1)]
        const float up = -(float)g.U * F1;
        const float upf = floorf(up);
        const int i0 = (int)((unsigned)g.U * (unsigned)A + (unsigned)(int)upf) - 1;
        const bool valid = F1 <= (float)A && F1 >= (float)(A - (n - 1)) &&
                           (unsigned)(i0 + 1) <= (unsigned)(g.U * (n - 1));
        // hour angle: the reference rotated by -Omega_r dt (u - mc)
        const float dl = g.w_dt * (F1 - (float)(A - mc));
        float sd, cm;   // sin dl, cos dl - 1
        if (fabsf(dl) <= 0.25f) {   // first terms left out: d^9/9! and d^8/8!, below 4e-10
            const float q = dl * dl;
            sd = dl * fmaf(q, fmaf(q, fmaf(q, -1.f / 5040.f, 1.f / 120.f), -1.f / 6.f), 1.f);
            cm = q * fmaf(q, fmaf(q, -1.f / 720.f, 1.f / 24.f), -0.5f);
        } else {
            sincosf(dl, &sd, &cm);
            cm -= 1.f;
        }
        const float4 q0 = cf[0], q1 = cf[1], q2 = cf[2];
        const float c1 = q2.y + fmaf(q2.y, cm, fmaf(-q2.z, sd, q2.w));
        const float s1 = q2.z + fmaf(q2.z, cm, fmaf(q2.y, sd, cf[3].x));
        const float c2 = c1 * c1 - s1 * s1, s2 = 2.f * s1 * c1;
        const float av = q0.x * c2 + q0.y * s2 + q0.z * c1 + q0.w * s1 + q1.x;
        const float bv = q1.y * c2 + q1.z * s2 + q1.w * c1 + q2.x * s1;
        float yr = 0.f, yi = 0.f;
        if (valid) {
            const float mu = up - upf;
            const float *xu = (const float *)g.xu;
            const int m_up = (int)g.m_up;
            float x4[4];
            if (i0 >= 0 && i0 + 3 < m_up) {
#pragma unroll
                for (int q = 0; q < 4; ++q) x4[q] = __ldg(xu + i0 + q);
            } else {   // periodic: only tap -1 and taps >= U n wrap, a single step
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int v = i0 + q;
                    x4[q] = __ldg(xu + (v < 0 ? v + m_up : (v >= m_up ? v - m_up : v)));
                }
            }
            // x1 + mu/2 (x2 - x0 + mu (2 x0 - 5 x1 + 4 x2 - x3 + mu (3 (x1 - x2) + x3 - x0)))
            const float a3 = fmaf(3.f, x4[1] - x4[2], x4[3] - x4[0]);
            const float a2 = fmaf(2.f, x4[0], fmaf(-5.f, x4[1], fmaf(4.f, x4[2], -x4[3])));
            const float v = fmaf(0.5f * mu, fmaf(mu, fmaf(mu, a3, a2), x4[2] - x4[0]), x4[1]);
            yr = v;
            if (g.f_off2.hi != 0.f) {   // uniform: a band at zero offset has no phase
                // band-offset phase at t, cycles: f_off d_j mod 1 + f f_off (d_{j+1} - d_j)
                if (j != j0) delay2(j, d0, d1);
                const float p = __fmul_rn(g.f_off2.hi, d0.hi);
                const float e = fmaf(g.f_off2.lo, d0.hi, fmaf(g.f_off2.hi, d0.lo, fmaf(g.f_off2.hi, d0.hi, -p)));
                const float psi = (p - rintf(p)) + e;
                float sp, cp;
                unit_f(psi + f * (g.f_off2.hi * ((d1.hi - d0.hi) + (d1.lo - d0.lo))), cp, sp);
                yr = v * cp;
                yi = -v * sp;
            }
            sv[i] = av * av;
            sv[4 + i] = bv * bv;
            sv[8 + i] = av * bv;
        }
        float4 *w = (float4 *)g.w + (int64_t)sl * g.w_stride;
        w[k] = make_float4(yr * av, yi * av, yr * bv, yi * bv);
        if (g.dbg_y) {
            g.dbg_y[2 * k] = yr; g.dbg_y[2 * k + 1] = yi;
            g.dbg_a[k] = av; g.dbg_b[k] = bv; g.dbg_mask[k] = valid;
        }
    }
    static_assert(kGeoPer == 4, "twelve sums of a warp in the sixteen slots");
    // S sums: each warp adds 32 terms in FP32 (relative error ~1e-7), the rest in FP64
    const float ws = warp_sum16(sv);
    const int lane = tid & 31, wp = tid >> 5, id = lane >> 1;
    if (!(lane & 1) && id < 12) sums[id >> 2][4 * wp + (id & 3)] = ws;
    __syncthreads();
    if (wp < 3) {
        const double t = warp_sum((double)sums[wp][lane]);
        if (lane == 0) g.partials[((int64_t)sl * g.nblk + blockIdx.x) * 3 + wp] = t;
    }
}

// FP64 form.  Bound by the FP64 units (1/64 of the FP32 rate), so it spends FP64
// instructions only where the result needs them, about 100 a sample: floors by a rounding
// addition whose low word is the integer, the hour angle as one multiply-add in turns, unit phases
// from the table, the Keys cubic in Horner form, the window test on integers, the S sums
// over kGeo64 samples of a thread before the block's reduction, and the delay in samples
// as a multiplication when dt is a power of two (the same value as the division).
// Measured at n = 86 164, 192 positions: 50 -> 17.2 us a position with the delays and the norms.
constexpr int kGeo64 = 4;

// Linear interpolation of the delay at fractional sample u from the per-sample delays dk,
// in the oracle's rounding sequence; the end segments extend beyond the data.  j = floor(u),
// or -1 or n far outside, and f = u - floor(u).
__device__ __forceinline__ double delay_lin(const double *__restrict__ dk, int n, double u, int &j, double &f) {
    f = __dsub_rn(u, p64::floor_int(u, j));
    if ((__double2hiint(u) & 0x7fffffff) >= 0x41d00000) j = u < 0.0 ? -1 : n;   // beyond 2^30 samples, or not a number
    const int jc = j < 0 ? 0 : (j > n - 2 ? n - 2 : j);
    const double g = jc == j ? f : __dsub_rn(u, (double)jc);
    const double d0 = dk[jc], d1 = dk[jc + 1];
    return __dadd_rn(d0, __dmul_rn(g, __dsub_rn(d1, d0)));
}

__global__ void __launch_bounds__(256) k_geometry64(GeoArgs g) {
    __shared__ double sh[24];
    const int sl = blockIdx.y;
    double saa = 0.0, sbb = 0.0, sab = 0.0;
    const SkyConst &sc = g.sky[g.s0 + sl];
    const double *dd = g.d + (int64_t)sl * g.d_stride;
    const bool pow2 = g.dt_pow2 != 0;
    const int n = (int)g.n;
    auto in_samples = [&](double t) { return pow2 ? __dmul_rn(t, g.inv_dt) : __ddiv_rn(t, g.dt); };
    // h / 2 pi = (alpha - phi0) / 2 pi - Omega_r dt u / 2 pi
    const double turn0 = (sc.alpha - g.phi0) * (1.0 / kTwoPi), turn_dt = kOmegaR / kTwoPi * g.dt;
    int k = blockIdx.x * (256 * kGeo64) + threadIdx.x;
#pragma unroll 1
    for (int it = 0; it < kGeo64 && k < n; ++it, k += 256) {
        // detector time t of barycentric sample k: t = k dt - d(k dt - d(k dt)),
        // in the oracle's rounding sequence, for 1e-10 agreement of F
        const double kd = (double)k;
        int j;
        double f;
        const double u0 = __dsub_rn(kd, in_samples(dd[k]));
        const double d1 = delay_lin(dd, n, u0, j, f);
        const double u = __dsub_rn(kd, in_samples(d1));
        const double d2 = delay_lin(dd, n, u, j, f);
        // 0 <= u <= n - 1
        const bool valid = j >= 0 && (j < n - 1 || (j == n - 1 && f == 0.0));
        const double2 eh = p64::unit_phase(g.unit_tab, fma(-turn_dt, u, turn0));
        const double c1 = eh.x, s1 = -eh.y;
        const double c2 = c1 * c1 - s1 * s1, s2 = 2.0 * s1 * c1;
        const double av = sc.A[0] * c2 + sc.A[1] * s2 + sc.A[2] * c1 + sc.A[3] * s1 + sc.A[4];
        const double bv = sc.B[0] * c2 + sc.B[1] * s2 + sc.B[2] * c1 + sc.B[3] * s1;
        double yr = 0.0, yi = 0.0;
        if (valid) {
            // Keys cubic (a = -1/2) on the upsampled series at p = U u = U j + U f, taps
            // i0 .. i0 + 3 around floor(p), periodic: p lies in [0, U (n - 1)], so only
            // i0 = -1 and indices >= U n wrap (a single step)
            const double p = (double)g.U * u;
            int ip;
            const double mu = p - p64::floor_int(p, ip);
            const int i0 = ip - 1, m_up = (int)g.m_up;
            const double *xu = (const double *)g.xu;
            double x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int v = i0 + q;
                x[q] = xu[v < 0 ? v + m_up : (v >= m_up ? v - m_up : v)];
            }
            // x1 + mu/2 (x2 - x0 + mu (2 x0 - 5 x1 + 4 x2 - x3 + mu (3 (x1 - x2) + x3 - x0)))
            const double a3 = fma(3.0, x[1] - x[2], x[3] - x[0]);
            const double a2 = fma(2.0, x[0], fma(-5.0, x[1], fma(4.0, x[2], -x[3])));
            const double v = fma(0.5 * mu, fma(mu, fma(mu, a3, a2), x[2] - x[0]), x[1]);
            // band-offset phase in cycles
            const double2 e = p64::unit_phase(g.unit_tab, __dmul_rn(g.f_off, d2));
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
static_assert(256 * kGeo64 == kGeo32, "both forms: 1024 samples a block");
inline int geo_blocks(int64_t n) { return (int)blocks(n, kGeo32); }

}  // namespace

// ================================================================== launchers
int64_t turn_table_entries() { return kTurnTab; }
void launch_turn_table(float4 *t, cudaStream_t s) { k_turn_table<<<kTurnTab / 256, 256, 0, s>>>(t); }

int launch_geometry(const Plan &p, const BandDev &b, int64_t s0, int64_t ns, bool fp32,
                    void *w, double *dbg_y, double *dbg_a, double *dbg_b, uint8_t *dbg_mask,
                    cudaStream_t s) {
    GeoArgs g;
    g.d = p.dbuf;
    g.r2 = static_cast<const DF *>(b.r2);
    g.f_off2 = df_from_double(b.f_off);
    g.inv_dt2 = df_from_double(1.0 / b.dt);
    g.phi0_turns = df_from_double(b.phi0 / kTwoPi);
    g.turn_dt = df_from_double(kOmegaR * b.dt / kTwoPi);
    g.w_dt = (float)(kOmegaR * b.dt);
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
    g.turn_tab = p.turn_tab;
    g.f_off = b.f_off;
    g.phi0 = b.phi0;
    g.sky = p.sky;
    g.s0 = s0;
    g.w = w;
    g.w_stride = p.w_stride;
    g.partials = p.partials;
    g.nblk = geo_blocks(b.n);
    g.dbg_y = dbg_y;
    g.dbg_a = dbg_a;
    g.dbg_b = dbg_b;
    g.dbg_mask = dbg_mask;
    dim3 grid(g.nblk, (unsigned)ns);
    if (fp32) {
        k_geometry<<<grid, kGeoThreads, 0, s>>>(g);
        return 1;
    } else {
        k_delays<<<dim3(blocks(b.n, 256), (unsigned)ns), 256, 0, s>>>(b.r, p.sky, s0, b.n, p.n_max, p.dbuf);
        k_geometry64<<<grid, 256, 0, s>>>(g);
    }
    return 2;
}

int launch_reduce_norms(const Plan &p, const BandDev &b, int64_t ns, double *norm, cudaStream_t s) {
    k_reduce_norms<<<(unsigned)ns, 32 * (kNormWarps + 1), 0, s>>>(
        p.partials, geo_blocks(b.n), p.sigma_parts, b.n, p.desc.sigma2, p.S, norm,
        p.desc.statistic == FSTAT_F_FULL ? 1 : 0);
    return 1;
}

}  // namespace fstat
