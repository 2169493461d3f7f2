// The FP32 search passes in packed arithmetic (packed.cuh): the 512-point rows
// (N_fft = 2^18, N1 = N2 = 512, the two-sidereal-day segments; as an option its
// columns too), the shorter rows of 2^12 .. 2^17 and of the interbinning form, the
// 1024-point rows of 2^19 and 2^20 and the 1024-point columns of 2^20.  Same
// four-step split and scratch layout as the second engine's passes (passes2.cuh);
// what changes is how a thread's 32 elements are transformed, for 512 points:
//
//  - the radix-32 first stage of a pass is split by one decimation-in-frequency
//    step into two 16-point DFTs, a_m = x_m + x_{m+16} and
//    b_m = (x_m - x_{m+16}) W_32^m, which run as one packed 16-point DFT; its
//    outputs come out as the pairs (X_{2k}, X_{2k+1}) of adjacent outputs;
//  - those pairs are exactly the two stage-1 jobs (2k, 2k + 1) a thread takes
//    next, so the exchange holds them side by side, (Re X_{2k}, Re X_{2k+1},
//    Im X_{2k}, Im X_{2k+1}) in one 16-byte word, and the radix-16 second stage,
//    its twiddles and the F epilogue run packed as well;
//  - in pass 2 the four-step twiddle W_N^{k1 l2} of inputs m and m + 16 folds
//    into the split: with T_m = W_N^{l2 (j + 16 m)} and c = W_N^{256 l2},
//    a_m = T_m (s_m + c s_{m+16}) and b_m = T_m W_32^m (s_m - c s_{m+16}).
#pragma once

#include "packed.cuh"
#include "passes2.cuh"

namespace fstat {
namespace p3 {

using pk::PC;

constexpr int kM = 512;          // pass length (both passes at N_fft = 2^18)
constexpr int kR0 = 32, kR1 = 16;
constexpr int kCol1024Ld = 1026;   // exchange row of a 1024-point column

// Stage-1 twiddles of a 512-point pass as packed pairs: entry [r][k] =
// (cos a_{2k}, cos a_{2k+1}, -sin a_{2k}, -sin a_{2k+1}), a_j = 2 pi r j / 512,
// r < 16, k < 16 (built on the host, 4 KiB).
__device__ __forceinline__ PC tw1(const float4 *__restrict__ t, int r, int k) {
    const float4 v = __ldg(t + r * 16 + k);
    return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}

// e^{-2 pi i m / 32} on one scalar complex value
__device__ __forceinline__ void w32_scalar(int m, float &xr, float &xi) { eng2::mul_w32(m, xr, xi); }

// --------------------------------------------------------------------- pass 1
// Columns k1 of the demodulated series: SearchLoad2 gives the stage-0 inputs
// (12 of 32 non-zero: the upper five eighths of each column lie in the zero
// padding when n <= 3 N_fft / 8), ScratchStore2 writes the transposed outputs.
// 256 threads: 8 columns x 2 transforms, 16 threads per sequence; CTA-wide
// exchange in the 16-byte layout of the second engine (element i at i + 2 (i/32)).
template <int LOGN, int Z1>
__global__ void __launch_bounds__(256, 3)
k_pass1p(SearchLoad2<Cfg2<LOGN, 1>> ld, ScratchStore2<Cfg2<LOGN, 1>> st, const float4 *__restrict__ tws) {
    using C = Cfg2<LOGN, 1>;
    static_assert(C::M == kM && C::SEQ == 16 && C::THREADS == 256, "512-point columns, 16 sequences");
    static_assert(Z1 == 3 || Z1 == 4, "known-zero eighths of a column");
    constexpr int SEQ = C::SEQ;
    constexpr int RL = eng2::row_ld16(kM);
    constexpr int NZ = kR0 * Z1 / 8;   // stage-0 inputs that can be non-zero (12 or 16)
    ld.init(blockIdx.x, blockIdx.y, blockIdx.y);
    st.init(blockIdx.x, blockIdx.y, blockIdx.y);
    float2 *sd = reinterpret_cast<float2 *>(eng2::dyn_smem());
    const int s = (int)threadIdx.x % SEQ;   // sequence: column f = s / 2, transform t = s & 1
    const int j = (int)threadIdx.x / SEQ;   // stage-0 butterfly; stage-1 job pair (2j, 2j + 1)
    eng2::Job q{s, s & 1, s >> 1, j};

    // stage 0: elements j + 16 r of the column, r < NZ non-zero
    PC P[16];
    {
        float re[NZ], im[NZ];
        ld.template load<NZ, 16>(q, re, im);
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            // a_m = x_m + x_{m+16}, b_m = (x_m - x_{m+16}) W_32^m; x_{m+16} is zero (m + 16 >= NZ)
            static_assert(NZ <= 16, "the upper half of the first stage lies in the zero padding");
            if (m < NZ) {
                float br = re[m], bi = im[m];
                w32_scalar(m, br, bi);
                P[m] = {make_float2(re[m], br), make_float2(im[m], bi)};
            }
        }
    }
    cod::dft16<NZ>(P);   // P[k] = (X_{2k}, X_{2k+1})
    {
        float4 *p4 = reinterpret_cast<float4 *>(sd + s * RL + eng2::pad16(j * kR0));
#pragma unroll
        for (int k = 0; k < 16; ++k) p4[k] = make_float4(P[k].re.x, P[k].re.y, P[k].im.x, P[k].im.y);
    }
    __syncthreads();
    // stage 1: jobs (2j, 2j + 1), element r at (2j) + 32 r
    PC Q[16];
    {
        const float4 *p4 = reinterpret_cast<const float4 *>(sd + s * RL + 2 * j);
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const float4 v = p4[eng2::pad16(r * kR0) / 2];
            Q[r] = {make_float2(v.x, v.y), make_float2(v.z, v.w)};
        }
    }
#pragma unroll
    for (int r = 1; r < 16; ++r) Q[r] = pk::cmul(Q[r], tw1(tws, r, j));
    cod::dft16<16>(Q);
    // outputs l2 = job + 32 p of the two jobs, one transposed store each
    float re0[16], im0[16], re1[16], im1[16];
#pragma unroll
    for (int p = 0; p < 16; ++p) {
        re0[p] = Q[p].re.x; im0[p] = Q[p].im.x;
        re1[p] = Q[p].re.y; im1[p] = Q[p].im.y;
    }
    eng2::Job q0{s, s & 1, s >> 1, 2 * j}, q1{s, s & 1, s >> 1, 2 * j + 1};
    st.template store<16, kR0>(q0, re0, im0);
    st.template store<16, kR0>(q1, re1, im1);
}

// The same columns with a scalar first stage (the second engine's half-zero
// radix-32 DFT, outputs stored in the packed exchange layout) and the packed
// second stage.
template <int LOGN, int Z1>
__global__ void __launch_bounds__(256, 3)
k_pass1h(SearchLoad2<Cfg2<LOGN, 1>> ld, ScratchStore2<Cfg2<LOGN, 1>> st, const float4 *__restrict__ tws) {
    using C = Cfg2<LOGN, 1>;
    static_assert(C::M == kM && C::SEQ == 16 && C::THREADS == 256, "512-point columns, 16 sequences");
    static_assert(Z1 == 3 || Z1 == 4, "known-zero eighths of a column");
    constexpr int SEQ = C::SEQ;
    constexpr int RL = eng2::row_ld16(kM);
    constexpr int NZ = kR0 * Z1 / 8;
    ld.init(blockIdx.x, blockIdx.y, blockIdx.y);
    st.init(blockIdx.x, blockIdx.y, blockIdx.y);
    float2 *sd = reinterpret_cast<float2 *>(eng2::dyn_smem());
    const int s = (int)threadIdx.x % SEQ;
    const int j = (int)threadIdx.x / SEQ;
    eng2::Job q{s, s & 1, s >> 1, j};
    {
        float re[kR0], im[kR0];
        ld.template load<NZ, 16>(q, re, im);
        eng2::dft<kR0, NZ>(re, im);
        float4 *p4 = reinterpret_cast<float4 *>(sd + s * RL + eng2::pad16(j * kR0));
#pragma unroll
        for (int k = 0; k < 16; ++k) p4[k] = make_float4(re[2 * k], re[2 * k + 1], im[2 * k], im[2 * k + 1]);
    }
    __syncthreads();
    PC Q[16];
    {
        const float4 *p4 = reinterpret_cast<const float4 *>(sd + s * RL + 2 * j);
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const float4 v = p4[eng2::pad16(r * kR0) / 2];
            Q[r] = {make_float2(v.x, v.y), make_float2(v.z, v.w)};
        }
    }
#pragma unroll
    for (int r = 1; r < 16; ++r) Q[r] = pk::cmul(Q[r], tw1(tws, r, j));
    cod::dft16<16>(Q);
    float re0[16], im0[16], re1[16], im1[16];
#pragma unroll
    for (int p = 0; p < 16; ++p) {
        re0[p] = Q[p].re.x; im0[p] = Q[p].im.x;
        re1[p] = Q[p].re.y; im1[p] = Q[p].im.y;
    }
    eng2::Job q0{s, s & 1, s >> 1, 2 * j}, q1{s, s & 1, s >> 1, 2 * j + 1};
    st.template store<16, kR0>(q0, re0, im0);
    st.template store<16, kR0>(q1, re1, im1);
}

// The columns of 1024 points (N_fft = 2^20): 256 threads, 4 columns x 2
// transforms, 32 threads per sequence.  Both radix-32 stages packed by one
// decimation-in-frequency split each: stage 0 as in k_pass1p, stage 1 (one 32-point job
// per thread) with its twiddle folded into the split as in k_pass2q below.
// Measured per 2^18 points: 1.056 -> 0.961 us (a third fewer instructions than the scalar pass;
// the 64-byte runs of its loads and stores cost it the rest against the 512-point columns).
template <int LOGN, int Z1, bool ROWS>
__global__ void __launch_bounds__(256, 3)
k_pass1q(SearchLoad2S<Cfg2<LOGN, 1>> ld, ScratchStore2<Cfg2<LOGN, 1>, ROWS> st, const float4 *__restrict__ tws,
         const float2 *__restrict__ w1024) {
    using C = Cfg2<LOGN, 1>;
    static_assert(C::M == 1024 && C::SEQ == 8 && C::THREADS == 256, "1024-point columns, 8 sequences");
    constexpr int SEQ = C::SEQ, RL = kCol1024Ld;
    constexpr int NZ = kR0 * Z1 / 8;   // stage-0 inputs that can be non-zero (12 or 16)
    ld.init(blockIdx.x, blockIdx.y, blockIdx.y);
    st.init(blockIdx.x, blockIdx.y, blockIdx.y);
    const int s = (int)threadIdx.x % SEQ;   // sequence: column f = s / 2, transform t = s & 1
    const int j = (int)threadIdx.x / SEQ;   // stage-0 butterfly, stage-1 job
    float2 *sd = reinterpret_cast<float2 *>(eng2::dyn_smem()) + s * RL;
    const eng2::Job q{s, s & 1, s >> 1, j};
    PC P[16];
    {
        float re[NZ], im[NZ];
        ld.template load<NZ, 32>(q, re, im);
#pragma unroll
        for (int m = 0; m < NZ; ++m) {   // x_{m+16} is zero
            float br = re[m], bi = im[m];
            w32_scalar(m, br, bi);
            P[m] = {make_float2(re[m], br), make_float2(im[m], bi)};
        }
    }
    cod::dft16<NZ>(P);   // P[k] = (X_{2k}, X_{2k+1})
    // element (output r, butterfly j) at 32 r + (j ^ (r & 1)), rows 2 mod 16 elements apart: a
    // half-warp (8 sequences, 2 butterflies or 2 jobs) falls in 16 different 8-byte banks
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        sd[32 * (2 * k) + j] = make_float2(P[k].re.x, P[k].im.x);
        sd[32 * (2 * k + 1) + (j ^ 1)] = make_float2(P[k].re.y, P[k].im.y);
    }
    const float2 c1 = __ldg(w1024 + 16 * j);
    __syncthreads();
    PC Q[16];
    const float2 *e = sd + 32 * j;
    const int jx = j & 1;
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        const float2 lo = e[m ^ jx], hi = e[(m + 16) ^ jx];
        const float ur = hi.x * c1.x - hi.y * c1.y, ui = hi.x * c1.y + hi.y * c1.x;
        Q[m] = {make_float2(lo.x + ur, lo.x - ur), make_float2(lo.y + ui, lo.y - ui)};
    }
#pragma unroll
    for (int m = 1; m < 16; ++m) {
        const float4 v = __ldg(tws + m * 32 + j);
        Q[m] = pk::cmul(Q[m], PC{make_float2(v.x, v.y), make_float2(v.z, v.w)});
    }
    cod::dft16<16>(Q);   // Q[k] = (Y_2k, Y_2k+1): l2 = j + 32 (2k + e)
    float re[32], im[32];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        re[2 * k] = Q[k].re.x; im[2 * k] = Q[k].im.x;
        re[2 * k + 1] = Q[k].re.y; im[2 * k + 1] = Q[k].im.y;
    }
    st.template store<32, 32>(q, re, im);
}

// --------------------------------------------------------------------- row twiddles
// The four-step twiddle of element k1 = j + G m of row l2 is W_N^{l2 j} (the
// thread's, from two table entries) times W_N^{G l2 m} (the row's).  The rows'
// factors come from a table, 16 packed pairs (256 bytes) per row or row pair, which
// a second bulk copy puts behind the staged rows; every lane reads the same word.
// A recurrence over m in place of the table took as many instructions, but its
// rounding error grew with m (a third of the error of F) and it chained 15
// complex multiplies.  Measured at 2^18: pass 2 0.660 -> 0.648 us a cell, rms error of F
// 6.5e-7 -> 3.2e-7.
constexpr int kRowTw = 16;

template <class C>
struct RowsTMA : ScratchLoadTMA<C> {
    static constexpr int ENTRIES = C::F;                     // table rows per tile
    static constexpr uint32_t TW_BYTES = ENTRIES * kRowTw * sizeof(float4);
    static constexpr uint32_t ROW_BYTES = (uint32_t)(2 * C::F * C::N1 * sizeof(float2));
    static constexpr size_t SMEM = ROW_BYTES + TW_BYTES + 16;   // rows, twiddles, mbarrier
    const float4 *row_tw;   // [row][16]
    const float4 *tws;      // in shared memory
    __device__ void init(int tile, int64_t cell, int64_t slot) {
        ScratchLoadTMA<C>::init(tile, cell, slot);
        unsigned char *sm = eng2::dyn_smem();
        tws = reinterpret_cast<const float4 *>(sm + ROW_BYTES);
        this->bar = reinterpret_cast<uint64_t *>(sm + ROW_BYTES + TW_BYTES);
        row_tw += (int64_t)tile * ENTRIES * kRowTw;
    }
    __device__ void stage() const {
        if (threadIdx.x == 0) {
            ptx::mbar_init(this->bar, 1);
            ptx::fence_mbar_init();
        }
        if constexpr (C::THREADS == 32) __syncwarp(); else __syncthreads();
        if (threadIdx.x == 0) {
            ptx::mbar_arrive_expect_tx(this->bar, ROW_BYTES + TW_BYTES);
            ptx::bulk_g2s(const_cast<float2 *>(this->rows), this->src, ROW_BYTES, this->bar);
            ptx::bulk_g2s(const_cast<float4 *>(tws), row_tw, TW_BYTES, this->bar);
        }
    }
    __device__ __forceinline__ PC tw_m(int entry, int m) const {
        const float4 v = tws[entry * kRowTw + m];
        return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
    }
};

// --------------------------------------------------------------------- pass 2
// Each warp's exchange lies over the row it has staged: 2 transforms x 16 job
// pairs x 16 elements of 16 bytes, exactly the row's 8 KiB, so no warp waits for
// another between the stages.

// Outputs p of a packed 16-point DFT that the F epilogue uses, halved: the bin
// range below N/2 (LOWER) needs p < 8 only.
template <bool LOWER>
__host__ __device__ constexpr int epi_half() { return (LOWER ? 8 : 16) / 2; }

// F per bin of the packed outputs (the epilogue of SearchEpi2 on pairs of values).
// Lanes 2j (F_a) and 2j + 1 (F_b) hold the same bins; the a lane evaluates F on
// the outputs p < H, the b lane on p >= H, each taking the partner's values for
// its half with one shuffle per value.  Output u of this lane's half, pair member
// e, is bin bin0 + off(u) + e step_e; lanes with own = false register nothing.
template <class C, bool LOWER, class Off>
__device__ __forceinline__ void epilogue(const SearchEpi2<C, LOWER> &ep, int t, int bin0, Off off, int step_e,
                                         const PC *Y, bool own = true) {
    constexpr int H = epi_half<LOWER>();
    const bool full = ep.nab != 0.f;
    float2 Fv[H];
#pragma unroll
    for (int u = 0; u < H; ++u) {
        // values are selected, never indexed by the lane's transform (that would
        // move Y to local memory)
        const PC lo = Y[u], hi = Y[u + H];
        if (full) {
            const PC send = t == 0 ? hi : lo, mine = t == 0 ? lo : hi;
            PC oth;
            oth.re.x = __shfl_xor_sync(0xffffffffu, send.re.x, 1);
            oth.re.y = __shfl_xor_sync(0xffffffffu, send.re.y, 1);
            oth.im.x = __shfl_xor_sync(0xffffffffu, send.im.x, 1);
            oth.im.y = __shfl_xor_sync(0xffffffffu, send.im.y, 1);
            const PC a = t == 0 ? mine : oth, b = t == 0 ? oth : mine;
            const float2 pa = pk::pfma(a.re, a.re, pk::pmul(a.im, a.im));
            const float2 pb = pk::pfma(b.re, b.re, pk::pmul(b.im, b.im));
            const float2 cr = pk::pfma(a.re, b.re, pk::pmul(a.im, b.im));
            Fv[u] = pk::pfma(pa, pk::bc(ep.na), pk::pfma(pb, pk::bc(ep.nb), pk::pmul(cr, pk::bc(ep.nab))));
        } else {
            const float2 plo = pk::pfma(lo.re, lo.re, pk::pmul(lo.im, lo.im));
            const float2 phi = pk::pfma(hi.re, hi.re, pk::pmul(hi.im, hi.im));
            const float2 ps = t == 0 ? phi : plo, pm = t == 0 ? plo : phi;
            float2 po;
            po.x = __shfl_xor_sync(0xffffffffu, ps.x, 1);
            po.y = __shfl_xor_sync(0xffffffffu, ps.y, 1);
            const float2 pa = t == 0 ? pm : po, pb = t == 0 ? po : pm;
            Fv[u] = pk::pfma(pa, pk::bc(ep.na), pk::pmul(pb, pk::bc(ep.nb)));
        }
    }
    const int lo = (int)ep.bin_lo;   // bins < 2^20
    const unsigned span = (unsigned)(ep.bin_hi - ep.bin_lo);
    bool pr[2 * H];
    bool any = false;
#pragma unroll
    for (int u = 0; u < H; ++u)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int bin = bin0 + off(u) + step_e * e;
            const float f = e ? Fv[u].y : Fv[u].x;
            pr[2 * u + e] = own && ((unsigned)(bin - lo) <= span) && (f > ep.thr_half);
            any |= pr[2 * u + e];
        }
    if (!__any_sync(0xffffffffu, any)) return;
    unsigned hits = 0;
#pragma unroll
    for (int u = 0; u < 2 * H; ++u) hits |= pr[u] ? 1u << u : 0u;
    unsigned long long idx = warp_slots(__popc(hits), ep.count);
#pragma unroll
    for (int u = 0; u < H; ++u)
#pragma unroll
        for (int e = 0; e < 2; ++e)
            if (hits & (1u << (2 * u + e))) {
                const float f = e ? Fv[u].y : Fv[u].x;
                if (idx < ep.cap) ep.out[idx] = CandRecord{ep.cell, (uint32_t)(bin0 + off(u) + step_e * e), (double)f};
                ++idx;
            }
}

// Rows l2 of the scratch, staged by a bulk copy (ScratchLoadTMA's copy and
// bounded wait), four-step twiddle folded into the split, packed row DFTs, then
// F, threshold and compaction.  A warp per row (F_a in the even lanes, F_b in
// the odd ones), TS / 32 rows per CTA; with one row per CTA (TS = 32, the
// default) 24 CTAs share an SM and each waits only for its own 8 KiB copy.
// ROWS: a launch over the row tiles from ep.tile0 on (modulo their number); a form of its own,
// as the two instructions before the copy is issued cost a launch over all rows 0.7 %.
template <int LOGN, bool LOWER, int TS, bool ROWS>
__global__ void __launch_bounds__(TS, 768 / TS)
k_pass2p(RowsTMA<Cfg2<LOGN, 2, TS>> ld, SearchEpi2<Cfg2<LOGN, 2, TS>, LOWER> ep,
         const float4 *__restrict__ tws) {
    using C = Cfg2<LOGN, 2, TS>;
    static_assert(C::M == kM && C::F == TS / 32 && C::SEQ == 2 * C::F && C::TPF == 16, "512-point rows, a warp per row");
    static_assert(2 * kR1 * kR1 * 16 == 2 * C::N1 * sizeof(float2), "a warp's exchange fills its staged row");
    if constexpr (!ROWS) ld.prefetch_ahead();   // it counts the tiles of a launch over all rows
    const int tile = ROWS ? ((int)blockIdx.x + ep.tile0) & (C::TILES - 1) : (int)blockIdx.x;
    ld.init(tile, blockIdx.y, blockIdx.y);
    const int w = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
    ep.init(tile, blockIdx.y, blockIdx.y);
    ld.stage();
    // lane 2j + t: a warp's loads from the staged row cover 32 consecutive
    // complex floats (F_a and F_b of 16 k1), free of bank conflicts
    const int t = lane & 1;            // transform
    const int j = lane >> 1;           // stage-0 butterfly; stage-1 job pair (2j, 2j + 1)
    const int f = w;                   // tile row
    const int l2 = ld.l2_0 + f;
    // four-step factors: T_0 = W^{l2 j}, c = W^{256 l2}; (W^{16 l2 m}, W^{16 l2 m} W_32^m)
    // come with the row
    const float2 w0 = ld.tw.wn(l2 * j), cc = ld.tw.wn(256 * l2);
    const PC T = {make_float2(w0.x, w0.x), make_float2(w0.y, w0.y)};
    ld.wait();
    PC P[16];
    {
        const float2 *row = ld.rows + 2 * (f * C::N1 + j) + t;   // element k1 at row[2 k1]
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const float2 lo = row[2 * 16 * m], hi = row[2 * 16 * (m + 16)];
            // u = c s_{m+16}; A = s_m + u, D = s_m - u
            const float ur = hi.x * cc.x - hi.y * cc.y, ui = hi.x * cc.y + hi.y * cc.x;
            const PC X = {make_float2(lo.x + ur, lo.x - ur), make_float2(lo.y + ui, lo.y - ui)};
            P[m] = pk::cmul(X, m ? pk::cmul(T, ld.tw_m(f, m)) : T);
        }
    }
    cod::dft16<16>(P);   // P[k] = (X_{2k}, X_{2k+1}) of row l2
    // the warp's exchange covers exactly the row f it has just read: only its own
    // lanes have to be done reading
    __syncwarp();
    float4 *ex = reinterpret_cast<float4 *>(eng2::dyn_smem()) + (2 * f + t) * (kR1 * kR1);
    // element (k, j) at word 16 k + (j ^ 4t ^ k): a quarter-warp holds 4 j of both
    // transforms, and its 8 lanes fall in 8 different 16-byte bank groups both
    // when storing (fixed k) and when loading (fixed r)
    const int jx = j ^ (4 * t);
#pragma unroll
    for (int k = 0; k < 16; ++k) ex[k * 16 + (jx ^ k)] = make_float4(P[k].re.x, P[k].re.y, P[k].im.x, P[k].im.y);
    __syncwarp();
    PC Q[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const float4 v = ex[j * 16 + (r ^ jx)];
        Q[r] = {make_float2(v.x, v.y), make_float2(v.z, v.w)};
    }
#pragma unroll
    for (int r = 1; r < 16; ++r) Q[r] = pk::cmul(Q[r], tw1(tws, r, j));
    cod::dft16<16, LOWER>(Q);
    // bins: job 2j + e, output p = u + t H: l1 = 2j + e + 32 p, bin = N2 l1 + l2
    constexpr int H = epi_half<LOWER>();
    epilogue<C, LOWER>(ep, t, C::N2 * (2 * j + kR0 * t * H) + l2, [](int u) { return C::N2 * kR0 * u; }, C::N2, Q);
}

// --------------------------------------------------------------------- pass 2, short rows
// The rows of N1 = 64, 128 or 256 points (2^12 .. 2^17) in adjacent pairs (l2, l2 + 1)
// packed in pairs: every operation is the same for the two rows except the four-step
// twiddle, which comes as a pair.  A warp takes G = 256 / N1 row pairs (1024 complex
// values of both transforms); lane t + 2 (g + G j) holds butterfly j of transform t of
// pair g: the 16 elements k1 = j + R1 m, R1 = N1 / 16.  Stage 0 is a packed 16-point DFT
// over m, stage 1 for each of G jobs q = j + R1 i the twiddle W_N1^{rq} and a packed
// R1-point DFT over the butterflies r, giving l1 = q + 16 p.  The exchange lies over the
// warp's staged rows (8 KiB) and no warp waits for another.
//
// IB, the interbinning form (transforms of N = n_fft / 2 points): bin 2k is X(k), bin
// 2k + 1 (pi/4)(X(k) - X(k + 1)).  The neighbour of a pair's first row is its second, that
// of the second the next pair's first row, traded through shared memory; the last pair of
// a tile only serves as a neighbour, so tiles advance by one pair less than they hold.
// After the last row comes row 0 at l1 + 1; where only the outputs l1 < N1/2 are formed
// (LOWER), its X(N/2), the sum of stage-1 inputs with alternating signs, is formed aside.
// Bound by issue and latency like the 512-point rows.  Measured, us per 2^18 points of both
// transforms, against the scalar two-stage pass: 64-point rows 1.55 -> 0.79, 128-point
// 1.08 -> 0.66; interbinning (per 2^18 bins) 64-point 1.12 -> 0.64, 128-point 0.76 -> 0.50,
// 256-point 0.636 -> 0.492.
template <int LOGN, int W>
struct RowGeom {
    static constexpr int N1 = 1 << (LOGN / 2), N2 = 1 << (LOGN - LOGN / 2), NP = N2 / 2;
    static constexpr int R1 = N1 / 16, G = 256 / N1;
    static constexpr int PAIRS = W * G;                       // row pairs per tile
    // complex floats between a warp's staged pairs: the padding puts the lanes of the
    // different pairs in different banks
    static constexpr int PAIR_LD = 4 * N1 + (G == 2 ? 8 : G == 4 ? 4 : 0);
    static constexpr uint32_t PAIR_BYTES = 4 * N1 * sizeof(float2), TW_BYTES = kRowTw * sizeof(float4);
    static constexpr size_t WARP_BYTES = (size_t)G * PAIR_LD * sizeof(float2);
    static constexpr size_t SMEM = W * WARP_BYTES + PAIRS * TW_BYTES + 8 * W;
    static constexpr int STEP = PAIRS >= NP ? NP : PAIRS > 1 ? PAIRS - 1 : 1;   // pairs emitted per interbinning tile
    static constexpr int TILES_IB = (NP + STEP - 1) / STEP, TILES = NP / PAIRS;
    static_assert(N1 >= 64 && N1 <= 256, "short rows");
};

template <int LOGN, bool LOWER, bool IB, int W, bool ROWS>
__global__ void __launch_bounds__(32 * W, 24 / W)
k_pass2rows(const float2 *__restrict__ scratch, InterTw<LOGN / 2> tw, const float4 *__restrict__ row_tw,
            const float2 *__restrict__ s1, uint32_t *err, SearchEpi2<Cfg2<LOGN, 2, 32>, LOWER> ep) {
    using C = Cfg2<LOGN, 2, 32>;
    using Q = RowGeom<LOGN, W>;
    constexpr int N1 = Q::N1, N2 = Q::N2, R1 = Q::R1, G = Q::G;
    unsigned char *sm = eng2::dyn_smem();
    const int w = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
    const int t = lane & 1, g = (lane >> 1) & (G - 1), j = lane / (2 * G);
    // the warp's first pair
    const int tile = ROWS ? ((int)blockIdx.x + ep.tile0) & (Q::TILES - 1) : (int)blockIdx.x;
    const int pair0 = tile * (IB ? Q::STEP : Q::PAIRS) + w * G;
    float2 *stage = reinterpret_cast<float2 *>(sm + w * Q::WARP_BYTES);
    float4 *tws = reinterpret_cast<float4 *>(sm + W * Q::WARP_BYTES) + w * G * kRowTw;
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + W * Q::WARP_BYTES + Q::PAIRS * Q::TW_BYTES) + w;
    if (lane == 0) {
        ptx::mbar_init(bar, 1);
        ptx::fence_mbar_init();
        ptx::mbar_arrive_expect_tx(bar, G * (Q::PAIR_BYTES + Q::TW_BYTES));
        const float2 *src = scratch + (int64_t)blockIdx.y * 2 * C::N;
#pragma unroll
        for (int i = 0; i < G; ++i) {
            const int pr = (pair0 + i) & (Q::NP - 1);   // past the last row come the first ones
            ptx::bulk_g2s(stage + i * Q::PAIR_LD, src + (int64_t)pr * 4 * N1, Q::PAIR_BYTES, bar);
            ptx::bulk_g2s(tws + i * kRowTw, row_tw + pr * kRowTw, Q::TW_BYTES, bar);
        }
    }
    __syncwarp();
    ep.init(0, blockIdx.y, blockIdx.y);
    const int P = pair0 + g, l2 = 2 * (P & (Q::NP - 1));   // rows l2 and l2 + 1
    // four-step factors of the two rows: T_0 = W^{l2 j}; the pairs W^{R1 l2 m} come with them
    const float2 wa = tw.wn(l2 * j), wb = tw.wn((l2 + 1) * j);
    const PC T = {make_float2(wa.x, wb.x), make_float2(wa.y, wb.y)};
    mbar_wait_bounded(bar, err);
    PC Pm[16];
    {
        const float2 *ra = stage + g * Q::PAIR_LD + 2 * j + t, *rb = ra + 2 * N1;   // element k1 at r[2 k1]
        const float4 *tp = tws + g * kRowTw;
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const float2 a = ra[2 * R1 * m], b = rb[2 * R1 * m];
            PC F = T;
            if (m) {
                const float4 v = tp[m];
                F = pk::cmul(T, PC{make_float2(v.x, v.y), make_float2(v.z, v.w)});
            }
            Pm[m] = pk::cmul({make_float2(a.x, b.x), make_float2(a.y, b.y)}, F);
        }
    }
    cod::dft16<16>(Pm);   // output k of butterfly j, both rows
    __syncwarp();        // the staged rows have been read: the exchange may overwrite them
    // element (output k, butterfly j) of (t, g) at word (k R1 + j) ^ X(k) of its N1 words;
    // X sends the 8 lanes of a quarter-warp to 8 different 16-byte bank groups, storing
    // (fixed k) and loading (fixed r)
    constexpr int JL = 4 / G;   // butterflies per quarter-warp
    float4 *ex = reinterpret_cast<float4 *>(stage) + (t * G + g) * N1;
    const int x0 = (t * G + g) * JL;
#pragma unroll
    for (int k = 0; k < 16; ++k)
        ex[(k * R1 + j) ^ (x0 ^ (k & (JL - 1)))] = make_float4(Pm[k].re.x, Pm[k].re.y, Pm[k].im.x, Pm[k].im.y);
    __syncwarp();
    constexpr int HR = LOWER ? R1 / 2 : R1;   // outputs kept per job
    PC Y[G * HR];
    PC top = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};   // IB, LOWER: X(N/2) of job 0
#pragma unroll
    for (int i = 0; i < G; ++i) {
        const int q = j + R1 * i;
        PC z[R1];
#pragma unroll
        for (int r = 0; r < R1; ++r) {
            const float4 v = ex[(q * R1 + r) ^ (x0 ^ (q & (JL - 1)))];
            z[r] = {make_float2(v.x, v.y), make_float2(v.z, v.w)};
        }
#pragma unroll
        for (int r = 1; r < R1; ++r) {
            const float2 e = __ldg(s1 + (N1 == 64 ? ((r * q) & 63) : r * 16 + q));   // W_N1^{rq}
            z[r] = {pk::pfma(z[r].re, pk::bc(e.x), pk::pmul(z[r].im, pk::bc(-e.y))),
                    pk::pfma(z[r].re, pk::bc(e.y), pk::pmul(z[r].im, pk::bc(e.x)))};
        }
        if (IB && LOWER && i == 0) {
            top = z[0];
#pragma unroll
            for (int r = 1; r < R1; ++r) top = r & 1 ? pk::sub(top, z[r]) : pk::add(top, z[r]);
        }
        cod::dft<R1, R1, LOWER>(z);
#pragma unroll
        for (int p = 0; p < HR; ++p) Y[i * HR + p] = z[p];   // l1 = q + 16 p
    }
    // output v = i HR + p: l1 = j + R1 i + 16 p; the b lane's half starts TO further on
    constexpr int H = epi_half<LOWER>();
    constexpr int TO = G == 1 ? 16 * H : R1 * G / 2;
    auto l1_of = [](int v) { return R1 * (v / HR) + 16 * (v % HR); };
    const int bin0 = N2 * (j + t * TO) + l2;
    if constexpr (!IB) {
        epilogue<C, LOWER>(ep, t, bin0, [&](int u) { return N2 * l1_of(u); }, 1, Y);
    } else {
        const int pl = w * G + g;                                   // pair within the tile
        const bool own = pl < Q::STEP && P < Q::NP;
        auto off2 = [&](int u) { return 2 * N2 * l1_of(u); };
        epilogue<C, LOWER>(ep, t, 2 * bin0, off2, 2, Y, own);      // even bins
        __syncthreads();                                            // every exchange has been read
        constexpr int LD = (LOWER ? N1 / 2 : N1) + 8;
        float2 *nb = reinterpret_cast<float2 *>(sm);                // [pair][t][LD]: first rows
        static_assert(Q::PAIRS * 2 * LD * sizeof(float2) <= W * Q::WARP_BYTES, "neighbours fit the staged rows");
#pragma unroll
        for (int v = 0; v < G * HR; ++v)
            nb[(2 * pl + t) * LD + j + l1_of(v)] = make_float2(Y[v].re.x, Y[v].im.x);
        if (LOWER && j == 0) nb[(2 * pl + t) * LD + N1 / 2] = make_float2(top.re.x, top.im.x);
        __syncthreads();
        const int pn = pl + 1 < Q::PAIRS ? pl + 1 : 0;
        const bool wrap = P + 1 >= Q::NP;                           // the next row is row 0, at l1 + 1
#pragma unroll
        for (int v = 0; v < G * HR; ++v) {
            int l1 = j + l1_of(v) + (wrap ? 1 : 0);
            if constexpr (!LOWER) l1 &= N1 - 1;
            const float2 n = nb[(2 * pn + t) * LD + l1];
            Y[v] = {make_float2(Y[v].re.x - Y[v].re.y, Y[v].re.y - n.x),
                    make_float2(Y[v].im.x - Y[v].im.y, Y[v].im.y - n.y)};
        }
        constexpr float Q2 = 0.61685027506808491f;                 // (pi / 4)^2
        ep.na *= Q2;
        ep.nb *= Q2;
        ep.nab *= Q2;
        epilogue<C, LOWER>(ep, t, 2 * bin0 + 1, off2, 2, Y, own);  // odd bins
    }
}

// --------------------------------------------------------------------- pass 2, 1024-point rows
// The rows of N_fft = 2^19 and 2^20 (N1 = 1024 = 32 x 32), a row of both transforms per
// 64-thread CTA: thread 2j + t takes the elements k1 = j + 32 m of transform t.
// Both radix-32 stages are split by one decimation-in-frequency step into a packed
// 16-point DFT, the stage's twiddle folded into the split as in k_pass2p: with
// V_m the twiddle of input m and c = V_{m+16} / V_m (the same for every m),
// a_m = V_m (x_m + c x_{m+16}), b_m = V_m W_32^m (x_m - c x_{m+16}); the outputs are
// the pairs (X_2k, X_2k+1).  In stage 1 V_m = W_1024^{mq} and V_m W_32^m =
// W_1024^{m(q+32)} come from one packed table.  A whole row per CTA (16 KiB, twelve
// CTAs per SM) instead of the radix-8 engine's three stages and two exchanges.
// Measured at N = 344 656 (768 cells): pass 2 5.36 -> 2.93 us a cell.
template <int LOGN, bool LOWER, bool ROWS>
__global__ void __launch_bounds__(64, 12)
k_pass2q(RowsTMA<Cfg2<LOGN, 2, 64>> ld, SearchEpi2<Cfg2<LOGN, 2, 64>, LOWER> ep,
         const float4 *__restrict__ tws, const float2 *__restrict__ w1024) {
    using C = Cfg2<LOGN, 2, 64>;
    static_assert(C::M == 1024 && C::F == 1 && C::THREADS == 64, "1024-point rows, one per CTA");
    const int tile = ROWS ? ((int)blockIdx.x + ep.tile0) & (C::TILES - 1) : (int)blockIdx.x;
    ld.init(tile, blockIdx.y, blockIdx.y);
    ep.init(tile, blockIdx.y, blockIdx.y);
    ld.stage();
    const int t = (int)threadIdx.x & 1, j = (int)threadIdx.x >> 1;
    const int l2 = ld.l2_0;
    const float2 w0 = ld.tw.wn(l2 * j), cc = ld.tw.wn(512 * l2);
    const PC T = {make_float2(w0.x, w0.x), make_float2(w0.y, w0.y)};
    const float2 c1 = __ldg(w1024 + 16 * j);
    ld.wait();
    PC P[16];
    {
        const float2 *row = ld.rows + 2 * j + t;   // element k1 at row[2 k1]
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const float2 lo = row[2 * 32 * m], hi = row[2 * 32 * (m + 16)];
            const float ur = hi.x * cc.x - hi.y * cc.y, ui = hi.x * cc.y + hi.y * cc.x;
            const PC X = {make_float2(lo.x + ur, lo.x - ur), make_float2(lo.y + ui, lo.y - ui)};
            P[m] = pk::cmul(X, m ? pk::cmul(T, ld.tw_m(0, m)) : T);
        }
    }
    cod::dft16<16>(P);   // P[k] = (X_{2k}, X_{2k+1}) of butterfly j
    __syncthreads();    // the staged row has been read: the exchange may overwrite it
    // element (output r, butterfly j) at 32 r + (j ^ r ^ 8 t): a half-warp holds 8 j (or,
    // loading, 8 r) of both transforms and falls in 16 different 8-byte banks either way
    float2 *ex = reinterpret_cast<float2 *>(eng2::dyn_smem()) + t * C::N1;
    const int jx = j ^ (8 * t);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        ex[32 * (2 * k) + (jx ^ (2 * k))] = make_float2(P[k].re.x, P[k].im.x);
        ex[32 * (2 * k + 1) + (jx ^ (2 * k + 1))] = make_float2(P[k].re.y, P[k].im.y);
    }
    __syncthreads();
    // stage 1, job q = j: the butterflies of output q
    const int q = j;
    PC Q[16];
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        const float2 lo = ex[32 * q + (m ^ jx)], hi = ex[32 * q + ((m + 16) ^ jx)];
        const float ur = hi.x * c1.x - hi.y * c1.y, ui = hi.x * c1.y + hi.y * c1.x;
        Q[m] = {make_float2(lo.x + ur, lo.x - ur), make_float2(lo.y + ui, lo.y - ui)};
    }
#pragma unroll
    for (int m = 1; m < 16; ++m) {
        const float4 v = __ldg(tws + m * 32 + q);
        Q[m] = pk::cmul(Q[m], PC{make_float2(v.x, v.y), make_float2(v.z, v.w)});
    }
    cod::dft16<16, LOWER>(Q);   // Q[k] = (Y_2k, Y_2k+1): l1 = q + 32 (2k + e)
    constexpr int H = epi_half<LOWER>();
    epilogue<C, LOWER>(ep, t, C::N2 * (q + 64 * t * H) + l2, [](int u) { return C::N2 * 64 * u; }, C::N2 * 32, Q);
}

}  // namespace p3
}  // namespace fstat
