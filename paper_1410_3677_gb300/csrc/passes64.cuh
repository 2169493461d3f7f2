// The FP64 search passes (FSTAT_FP64_PLAIN), N_fft = 2^12 .. 2^20: the two-stage
// engine (fft_engine2.cuh) in double precision, a batch of cells per launch.
//
// What bounds them: the FP64 units (2 multiply-adds per clock and SM on GB300,
// 1/64 of the FP32 rate).  Everything else -- integer work, shuffles, table
// loads, shared-memory traffic -- runs in their shadow, so the passes are laid
// out for the fewest FP64 instructions:
//  - the first DFT of a column skips the inputs in the zero padding (half, or
//    five eighths when n <= 3N/8), the last DFT of a row the outputs outside the
//    bin range's half;
//  - spindown phases are evaluated once for the two transforms of a sample (lane
//    pairs) from a table of unit phases and a short Taylor step (unit_phase)
//    instead of sincospi;
//  - the four-step twiddle is read from a full table W_N^{k1 l2}, written once
//    per plan in the order pass 2 reads it, instead of a recurrence;
//  - both passes run on many cells, so that the 128 tiles of one 2^18 transform
//    no longer leave a sixth of the 152 SMs idle.
// Measured on GB300 at N = 86 164, N_fft = 2^18 (192 sky positions, one spindown), per
// cell: pass 1 52.9 -> 25.9 us, pass 2 44.9 -> 29.3 us against the radix-8 engine, one
// cell a launch, the FP64 pipe 85 % active; 128 cells at 2^13: 80 -> 1.73 us for both.
#pragma once

#include "passes2.cuh"
#include "unit_phase.cuh"

namespace fstat {
namespace p64 {

constexpr int kTS = 128;           // threads per CTA
constexpr int kMinLog = 12, kMaxLog = 20;

template <int LOGN, int PASS>
struct Cfg64 : Cfg2<LOGN, PASS, kTS> {
    using B = Cfg2<LOGN, PASS, kTS>;
    static constexpr size_t SMEM = eng2::smem_bytes<double, B::M, B::SEQ>();
};
// rows per pass-2 tile: the blocking of the scratch and of the twiddle table
template <int LOGN>
constexpr int row_block() { return Cfg64<LOGN, 2>::F; }

// Pass 1 input: w[k] = {y a, y b}, read as the complex half t; times the spindown
// phase e^{-2 pi i frac(rate k^2)}.  Lanes 2f and 2f + 1 hold the two halves of
// the same samples: lane t evaluates the phases of the elements r = 2i + t.
template <class C>
struct Load64 {
    const double2 *w;         // two double2 per sample
    int64_t w_stride;
    int n;
    const double *chirp;
    int n_spin;
    int64_t c0, s0;
    const double2 *tab;
    const double2 *ws;
    double rate;
    int k1_0;
    __device__ void init(int tile, int64_t cell) {
        const int64_t c = c0 + cell;
        const int64_t sky = (int64_t)((uint32_t)c / (uint32_t)n_spin);
        ws = w + 2 * (sky - s0) * w_stride;
        rate = chirp[c - sky * n_spin];
        k1_0 = tile * C::F;
    }
    template <int R, int JPF>
    __device__ __forceinline__ void load(const eng2::Job &q, double *re, double *im) const {
        static_assert(R % 2 == 0, "elements in pairs");
        const int kb = k1_0 + q.f + C::N1 * q.j;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int k = kb + C::N1 * JPF * r;
            double2 v = make_double2(0.0, 0.0);
            if (k < n) v = __ldg(ws + 2 * k + q.t);
            re[r] = v.x; im[r] = v.y;
        }
        double2 e[R / 2];
#pragma unroll
        for (int i = 0; i < R / 2; ++i) {
            const int k = kb + C::N1 * JPF * (2 * i + q.t);
            e[i] = make_double2(1.0, 0.0);
            if (k < n) {
                const double kd = (double)k;
                e[i] = unit_phase(tab, rate * (kd * kd));
            }
        }
        const int lane = (int)threadIdx.x & 31;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int src = (lane & ~1) | (r & 1);   // the lane that evaluated element r
            const double c = __shfl_sync(0xffffffffu, e[r / 2].x, src);
            const double s = __shfl_sync(0xffffffffu, e[r / 2].y, src);
            if (kb + C::N1 * JPF * r < n) {
                const double x = re[r], y = im[r];
                re[r] = x * c - y * s;
                im[r] = x * s + y * c;
            }
        }
    }
};

// Pass 1 output, blocked by pass-2 tiles: A[l2 / RB][k1][l2 % RB][t], so that a
// pass-2 tile is one run and its lanes (consecutive rows and transforms) read
// consecutive elements.
template <class C, int RB>
struct Store64 {
    static constexpr bool kStoreEarly = true;
    double2 *scratch;
    double2 *base;
    __device__ void init(int tile, int64_t slot) {
        base = scratch + slot * 2 * C::N + 2 * RB * (int64_t)(tile * C::F);
    }
    template <int R, int JPF>
    __device__ __forceinline__ void store(const eng2::Job &q, double *re, double *im) const {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int l2 = q.j + r * JPF;
            __stcg(base + 2 * RB * ((int64_t)(l2 / RB) * C::N1 + q.f) + 2 * (l2 % RB) + q.t,
                   make_double2(re[r], im[r]));
        }
    }
};

// Pass 2 input: the tile's rows times W_N^{k1 l2} from the table in the same order.
template <class C>
struct RowLoad64 {
    const double2 *scratch;
    const double2 *tw;
    const double2 *base, *twb;
    __device__ void init(int tile, int64_t slot) {
        base = scratch + slot * 2 * C::N + 2 * (int64_t)tile * C::N1 * C::F;
        twb = tw + (int64_t)tile * C::N1 * C::F;
    }
    template <int R, int JPF>
    __device__ __forceinline__ void load(const eng2::Job &q, double *re, double *im) const {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const double2 v = __ldcg(base + 2 * C::F * (q.j + r * JPF) + 2 * q.f + q.t);
            re[r] = v.x; im[r] = v.y;
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const double2 e = __ldg(twb + C::F * (q.j + r * JPF) + q.f);
            const double x = re[r], y = im[r];
            re[r] = x * e.x - y * e.y;
            im[r] = x * e.y + y * e.x;
        }
    }
};

// F per bin, strict 2F > thr, compaction.  Lanes 2f (F_a) and 2f + 1 (F_b) hold
// the same bins: the a lane evaluates the first half of the outputs, the b lane
// the second.  LOWER: the bin range lies below N/2 (outputs r < R/2 only).
template <class C, bool LOWER>
struct Epi64 {
    const double *norm;
    int n_spin;
    int64_t c0, s0;
    uint32_t cell_base;
    int64_t bin_lo, bin_hi;
    int tile0;   // first row tile of a launch over some of the rows
    double thr;
    CandRecord *out;
    unsigned long long *count;
    unsigned long long cap;
    double na, nb, nab;
    uint32_t cell;
    int l2_0;
    __device__ void init(int tile, int64_t cl) {
        const int64_t c = c0 + cl;
        const int64_t sky = (int64_t)((uint32_t)c / (uint32_t)n_spin);
        const double *nf = norm + kNormStride * (sky - s0);
        na = nf[0];
        nb = nf[1];
        nab = nf[2];
        cell = cell_base + (uint32_t)c;
        l2_0 = tile * C::F;
    }
    template <int R, int JPF>
    __device__ __forceinline__ void store(const eng2::Job &q, double *re, double *im) const {
        constexpr int H = (LOWER ? R / 2 : R) / 2;
        const int lane = (int)threadIdx.x & 31;
        double Fv[H];
        bool pr[H];
        bool any = false;
        const int bin0 = C::N2 * (q.j + q.t * H * JPF) + l2_0 + q.f;
        const int lo = (int)bin_lo;
        const unsigned span = (unsigned)(bin_hi - bin_lo);
        const bool full = nab != 0.0;
#pragma unroll
        for (int r = 0; r < H; ++r) {
            if (full) {
                const double sr = q.t == 0 ? re[r + H] : re[r], si = q.t == 0 ? im[r + H] : im[r];
                const double orr = __shfl_xor_sync(0xffffffffu, sr, 1);
                const double oi = __shfl_xor_sync(0xffffffffu, si, 1);
                const double ar = q.t == 0 ? re[r] : orr, ai = q.t == 0 ? im[r] : oi;
                const double br = q.t == 0 ? orr : re[r + H], bi = q.t == 0 ? oi : im[r + H];
                Fv[r] = (ar * ar + ai * ai) * na + (br * br + bi * bi) * nb + (ar * br + ai * bi) * nab;
            } else {
                const double p_lo = re[r] * re[r] + im[r] * im[r];
                const double p_hi = re[r + H] * re[r + H] + im[r + H] * im[r + H];
                const double other = __shfl_xor_sync(0xffffffffu, q.t == 0 ? p_hi : p_lo, 1);
                Fv[r] = q.t == 0 ? p_lo * na + other * nb : other * na + p_hi * nb;
            }
            const unsigned off = (unsigned)(bin0 + r * C::N2 * JPF - lo);
            pr[r] = (off <= span) && (2.0 * Fv[r] > thr);
            any |= pr[r];
        }
        if (!__any_sync(0xffffffffu, any)) return;
#pragma unroll
        for (int r = 0; r < H; ++r) {
            const unsigned m = __ballot_sync(0xffffffffu, pr[r]);
            if (m) {
                const int leader = __ffs(m) - 1;
                unsigned long long b0 = 0;
                if (lane == leader) b0 = atomicAdd(count, (unsigned long long)__popc(m));
                b0 = __shfl_sync(0xffffffffu, b0, leader);
                if (pr[r]) {
                    const unsigned long long idx = b0 + __popc(m & ((1u << lane) - 1u));
                    if (idx < cap) out[idx] = CandRecord{cell, (uint32_t)(bin0 + r * C::N2 * JPF), Fv[r]};
                }
            }
        }
    }
};

// 128 threads with 32 complex doubles each (128 registers of data): two CTAs per SM (three,
// with 168 registers a thread, measured the same).
template <int LOGN, int PASS, class LD, class ST, int Z1>
__global__ void __launch_bounds__(kTS, 2) k_pass64(LD ld, ST st, const double *__restrict__ tw) {
    using C = Cfg64<LOGN, PASS>;
    int tile = (int)blockIdx.x;
    if constexpr (PASS == 2) tile = (tile + st.tile0) & (C::TILES - 1);
    ld.init(tile, blockIdx.y);
    st.init(tile, blockIdx.y);
    eng2::run_pass<double, C::M, C::SEQ, C::EH, eng2::kMapFJ, LD, ST, PASS == 1 ? Z1 : 8, true>(ld, st, tw);
}

}  // namespace p64
}  // namespace fstat
