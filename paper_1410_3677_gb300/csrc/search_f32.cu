// FP32 instantiations of the search passes (FSTAT_FP32_BATCHED): the two-stage
// engine for transform lengths 2^12 .. 2^20 (as two launches, or up to 2^19 both
// passes in one ticket-ordered launch), the radix-8 engine otherwise (and whenever the
// plan selects it).
#include <algorithm>

#include "passes2.cuh"
#include "passes3.cuh"
#include "search_launch.cuh"

namespace fstat {
namespace {

template <int LOGN, bool LOWER, int TS = 256>
SearchEpi2<Cfg2<LOGN, 2, TS>, LOWER> make_epi(const Plan &p, int band_idx, const BandDev &b, int64_t c0,
                                              int64_t s0, const CellBufs &cb, int tile0 = 0) {
    SearchEpi2<Cfg2<LOGN, 2, TS>, LOWER> st2{};
    st2.tile0 = tile0;
    st2.norm = cb.norm;
    st2.n_spin = (int)p.desc.n_spin;
    st2.c0 = c0;
    st2.s0 = s0;
    st2.cell_base = (uint32_t)((int64_t)band_idx * p.desc.n_sky * p.desc.n_spin);
    st2.bin_lo = b.lo;
    st2.bin_hi = b.hi;
    st2.thr = (float)p.desc.thr_2F;
    st2.out = p.cand;
    st2.count = p.cand_count;
    st2.cap = (unsigned long long)p.cand_capacity;
    return st2;
}

template <int LOGN, bool LOWER, int TS, class LD2>
void launch_pass2(const Plan &p, int band_idx, const BandDev &b, int64_t s0, int64_t c0, int64_t nc,
                  cudaStream_t s, const CellBufs &cb, const LD2 &ld2, const TwiddleSet *tw, size_t extra) {
    using C2 = Cfg2<LOGN, 2, TS>;
    const auto st2 = make_epi<LOGN, LOWER, TS>(p, band_idx, b, c0, s0, cb);
    auto k2 = k_pass2<LOGN, 2, eng2::kMapW, LD2, SearchEpi2<C2, LOWER>, TS>;
    set_smem(k2, C2::SMEM + extra);
    k2<<<dim3(C2::TILES, (unsigned)nc), C2::THREADS, C2::SMEM + extra, s>>>(ld2, st2, tw->s1_f);
}

// The paired pass 2 (512-point rows) in CTAs of TS / 32 rows, one warp per row.
template <int LOGN, bool LOWER, int TS>
void launch_pass2p(const Plan &p, int band_idx, const BandDev &b, int64_t s0, int64_t c0, int64_t nc,
                   cudaStream_t s, const CellBufs &cb, const ScratchLoad2<Cfg2<LOGN, 2>> &ld2,
                   const TwiddleSet *tw, RowRange rr) {
    using D2 = Cfg2<LOGN, 2, TS>;
    p3::RowsTMA<D2> lt{};
    lt.scratch = ld2.scratch;
    lt.tw = ld2.tw;
    lt.pf_dist = p.pf_dist_pk;   // the paired pass gains nothing from L2 prefetch ahead
    lt.err = p.qerr;
    lt.row_tw = tw->row_tw;
    const auto ep = make_epi<LOGN, LOWER, TS>(p, band_idx, b, c0, s0, cb, rr.tile0);
    auto run = [&](auto k2) {
        constexpr size_t smem2 = p3::RowsTMA<D2>::SMEM;
        set_smem(k2, smem2);
        k2<<<dim3(rr.tiles, (unsigned)nc), D2::THREADS, smem2, s>>>(lt, ep, tw->p512_f);
    };
    if (TS == 32 && rr.tiles < D2::TILES) run(p3::k_pass2p<LOGN, LOWER, TS, TS == 32>);
    else run(p3::k_pass2p<LOGN, LOWER, TS, false>);
}

// Short rows (64 .. 256 points) in packed pairs, zero-padded or interbinning.
bool rows_packed(const Plan &p) { return packed_rows(p) && p.p2_rows; }
// Warps per interbinning tile: few enough rows computed twice (one pair per tile) at 24 warps per SM.
constexpr int ib_warps(int logn) { return logn == 12 || logn == 15 ? 8 : logn <= 14 ? 6 : 12; }

template <int LOGN, bool LOWER, bool IB, int W>
void launch_rows(const Plan &p, int band_idx, const BandDev &b, int64_t s0, int64_t c0, int64_t nc, cudaStream_t s,
                 const CellBufs &cb, const TwiddleSet *tw, RowRange rr) {
    using Q = p3::RowGeom<LOGN, W>;
    const auto ep = make_epi<LOGN, LOWER, 32>(p, band_idx, b, c0, s0, cb, rr.tile0);
    // stage-1 twiddles [r][q], q < 16; the 64-point rows' table is in another order, they take W_64^m
    const float *s1 = Q::N1 == 64 ? tw->in1_f : tw->s1_f;
    auto run = [&](auto k2) {
        set_smem(k2, Q::SMEM);
        k2<<<dim3(rr.tiles, (unsigned)nc), 32 * W, Q::SMEM, s>>>(
            reinterpret_cast<const float2 *>(cb.scratch), InterTw<LOGN / 2>{tw->lo_f, tw->hi_f}, tw->row_tw,
            reinterpret_cast<const float2 *>(s1), p.qerr, ep);
    };
    if (!IB && rr.tiles < Q::TILES) run(p3::k_pass2rows<LOGN, LOWER, IB, W, !IB>);
    else run(p3::k_pass2rows<LOGN, LOWER, IB, W, false>);
}

template <int LOGN, bool LOWER>
int launch_two(const Plan &p, int band_idx, const BandDev &b, int64_t s0, int64_t c0, int64_t nc,
               cudaStream_t s, cudaEvent_t mid, const CellBufs &cb, const SearchLoad2<Cfg2<LOGN, 1>> &ld1,
               const ScratchStore2<Cfg2<LOGN, 1>> &st1, const ScratchLoad2<Cfg2<LOGN, 2>> &ld2,
               const TwiddleSet *tw) {
    using C1 = Cfg2<LOGN, 1>;
    using C2 = Cfg2<LOGN, 2>;
    // 512-point rows (N_fft = 2^18, 2^19): pass 2 in paired FP32 arithmetic; at 2^18
    // (512-point columns) also pass 1 with packed = 2 or 3
    const bool pk2 = (LOGN == 18 || LOGN == 19) && packed_rows(p) && tw->p512_f;
    const bool pk1 = pk2 && LOGN == 18 && p.packed >= 2;
    // A bin range shorter than N2 touches some of the rows l2 = bin mod N2 only (a follow-up
    // about known candidates): the packed pass 2 runs over their tiles, and while they are at
    // most three quarters of the rows pass 1 stores no others.  Measured, 576 cells at 2^18, a whole
    // search (all rows 922 us): 121 bins 1264 -> 911 us with the read-back, 256 bins 920 -> 685 us, 384
    // bins 833 -> 797; without the pass-1 part 748 us at 258 bins.  At 2^20 the test of each
    // store costs more than it saves beyond three quarters (768 of 1024 rows 3786 -> 3747 us,
    // 1022 rows 4208 -> 4290).
    int f2 = 0;   // rows per tile of the packed pass 2 (0: another pass 2, all rows)
    if constexpr (LOGN <= 17) f2 = rows_packed(p) ? 2 * p3::RowGeom<LOGN, 1>::PAIRS : 0;
    if constexpr (LOGN == 18 || LOGN == 19) f2 = pk2 && p.p2_ts == 32 ? 1 : 0;
    if constexpr (C2::M == 1024) f2 = 1;
    const RowRange rr = f2 ? searched_rows(b, C2::N2, f2) : RowRange{0, C2::N2 / std::max(1, p.p2_ts / 32)};
    const bool few = f2 && 4 * rr.tiles * f2 <= 3 * C2::N2 && p.share_chirp;
    ScratchStore2<C1, true> st1r{st1.scratch, rr.tile0 * f2, rr.tiles * f2};
    if constexpr (LOGN == 18) {
        if (pk1) {   // packed = 2: both stages paired; 3: scalar first stage, paired second
            const bool z3 = 8 * b.n <= 3 * (int64_t)C1::N;
            const bool hy = p.packed == 3;
            auto k1 = hy ? (z3 ? p3::k_pass1h<LOGN, 3> : p3::k_pass1h<LOGN, 4>)
                         : (z3 ? p3::k_pass1p<LOGN, 3> : p3::k_pass1p<LOGN, 4>);
            set_smem(k1, C1::SMEM);
            k1<<<dim3(C1::TILES, (unsigned)nc), C1::THREADS, C1::SMEM, s>>>(ld1, st1, tw->p512_f);
        }
    }
    // columns known zero beyond 3/8 of their length (radix-32 first stage) or 1/2
    bool launched = pk1;
    if constexpr (C1::M == 1024) {   // 1024-point columns (2^19, 2^20): packed
        if (p.packed >= 1 && p.share_chirp && tw->p1024_f) {
            SearchLoad2S<C1> l1s{};
            static_cast<SearchLoad2<C1> &>(l1s) = ld1;
            constexpr size_t smem1 = (size_t)C1::SEQ * p3::kCol1024Ld * sizeof(float2);
            auto run = [&](auto k1, const auto &st) {
                set_smem(k1, smem1);
                k1<<<dim3(C1::TILES, (unsigned)nc), C1::THREADS, smem1, s>>>(
                    l1s, st, tw->p1024_f, reinterpret_cast<const float2 *>(tw->in2_f));
            };
            const bool z3 = 8 * b.n <= 3 * (int64_t)C1::N;
            if (few) z3 ? run(p3::k_pass1q<LOGN, 3, true>, st1r) : run(p3::k_pass1q<LOGN, 4, true>, st1r);
            else z3 ? run(p3::k_pass1q<LOGN, 3, false>, st1) : run(p3::k_pass1q<LOGN, 4, false>, st1);
            launched = true;
        }
    }
    if constexpr (eng2::radix0(C1::M) == 32) {
        if (!launched && 8 * b.n <= 3 * (int64_t)C1::N && p.share_chirp) {
            SearchLoad2S<C1> l1s{};
            static_cast<SearchLoad2<C1> &>(l1s) = ld1;
            auto run = [&](auto k1, const auto &st) {
                set_smem(k1, C1::SMEM);
                k1<<<dim3(C1::TILES, (unsigned)nc), C1::THREADS, C1::SMEM, s>>>(l1s, st, tw->s2_f);
            };
            if (few) run(k_pass2<LOGN, 1, eng2::kMapFJ, SearchLoad2S<C1>, ScratchStore2<C1, true>, 256, 3>, st1r);
            else run(k_pass2<LOGN, 1, eng2::kMapFJ, SearchLoad2S<C1>, ScratchStore2<C1>, 256, 3>, st1);
            launched = true;
        }
        if (!launched && 8 * b.n <= 3 * (int64_t)C1::N) {
            auto k1 = k_pass2<LOGN, 1, eng2::kMapFJ, SearchLoad2<C1>, ScratchStore2<C1>, 256, 3>;
            set_smem(k1, C1::SMEM);
            k1<<<dim3(C1::TILES, (unsigned)nc), C1::THREADS, C1::SMEM, s>>>(ld1, st1, tw->s2_f);
            launched = true;
        }
    }
    if (!launched && p.share_chirp) {
        SearchLoad2S<C1> l1s{};
        static_cast<SearchLoad2<C1> &>(l1s) = ld1;
        auto run = [&](auto k1, const auto &st) {
            set_smem(k1, C1::SMEM);
            k1<<<dim3(C1::TILES, (unsigned)nc), C1::THREADS, C1::SMEM, s>>>(l1s, st, tw->s2_f);
        };
        if (few) run(k_pass2<LOGN, 1, eng2::kMapFJ, SearchLoad2S<C1>, ScratchStore2<C1, true>, 256, 4>, st1r);
        else run(k_pass2<LOGN, 1, eng2::kMapFJ, SearchLoad2S<C1>, ScratchStore2<C1>, 256, 4>, st1);
        launched = true;
    }
    if (!launched) {
        auto k1 = k_pass2<LOGN, 1, eng2::kMapFJ, SearchLoad2<C1>, ScratchStore2<C1>, 256, 4>;
        set_smem(k1, C1::SMEM);
        k1<<<dim3(C1::TILES, (unsigned)nc), C1::THREADS, C1::SMEM, s>>>(ld1, st1, tw->s2_f);
    }
    if (mid) record_timing_event(mid, s);
    if constexpr (LOGN <= 17) {   // rows of 64 .. 256 points: packed in pairs
        if (rows_packed(p)) {
            launch_rows<LOGN, LOWER, false, 1>(p, band_idx, b, s0, c0, nc, s, cb, tw, rr);
            return 2;
        }
    }
    if constexpr (LOGN == 18 || LOGN == 19) {
        if (pk2) {
            if (p.p2_ts == 32) launch_pass2p<LOGN, LOWER, 32>(p, band_idx, b, s0, c0, nc, s, cb, ld2, tw, rr);
            else if (p.p2_ts == 64) launch_pass2p<LOGN, LOWER, 64>(p, band_idx, b, s0, c0, nc, s, cb, ld2, tw, rr);
            else launch_pass2p<LOGN, LOWER, 128>(p, band_idx, b, s0, c0, nc, s, cb, ld2, tw, rr);
            return 2;
        }
    }
    if constexpr (C2::M == 1024) {   // 1024-point rows: one per CTA, packed
        using D2 = Cfg2<LOGN, 2, 64>;
        p3::RowsTMA<D2> lt{};
        lt.scratch = ld2.scratch;
        lt.tw = ld2.tw;
        lt.pf_dist = 0;
        lt.err = p.qerr;
        lt.row_tw = tw->row_tw;
        const auto ep = make_epi<LOGN, LOWER, 64>(p, band_idx, b, c0, s0, cb, rr.tile0);
        auto run = [&](auto k2) {
            constexpr size_t smem2 = p3::RowsTMA<D2>::SMEM;
            set_smem(k2, smem2);
            k2<<<dim3(rr.tiles, (unsigned)nc), D2::THREADS, smem2, s>>>(lt, ep, tw->p1024_f,
                                                                         reinterpret_cast<const float2 *>(tw->in1_f));
        };
        if (rr.tiles < D2::TILES) run(p3::k_pass2q<LOGN, LOWER, true>);
        else run(p3::k_pass2q<LOGN, LOWER, false>);
        return 2;
    } else if (p.tma && p.p2_threads == 128) {   // smaller tiles, six CTAs per SM
        ScratchLoadTMA<Cfg2<LOGN, 2, 128>> lt{};
        lt.scratch = ld2.scratch;
        lt.tw = ld2.tw;
        lt.pf_dist = 2 * ld2.pf_dist;
        lt.err = p.qerr;
        launch_pass2<LOGN, LOWER, 128>(p, band_idx, b, s0, c0, nc, s, cb, lt, tw, 16);
    } else if (p.tma) {   // rows staged by bulk copies; an 8-byte mbarrier after the shared memory
        ScratchLoadTMA<C2> lt{};
        lt.scratch = ld2.scratch;
        lt.tw = ld2.tw;
        lt.pf_dist = ld2.pf_dist;
        lt.err = p.qerr;
        launch_pass2<LOGN, LOWER, 256>(p, band_idx, b, s0, c0, nc, s, cb, lt, tw, 16);
    } else {
        launch_pass2<LOGN, LOWER, 256>(p, band_idx, b, s0, c0, nc, s, cb, ld2, tw, 0);
    }
    return 2;
}

template <int LOGN, bool LOWER>
int launch_fused(const Plan &p, int band_idx, const BandDev &b, int64_t s0, int64_t c0, int64_t nc,
                 cudaStream_t s, const CellBufs &cb, const SearchLoad2<Cfg2<LOGN, 1>> &ld1,
                 const ScratchStore2<Cfg2<LOGN, 1>> &st1, const ScratchLoad2<Cfg2<LOGN, 2>> &ld2,
                 const TwiddleSet *tw) {
    using C1 = Cfg2<LOGN, 1>;
    using C2 = Cfg2<LOGN, 2>;
    const auto st2 = make_epi<LOGN, LOWER>(p, band_idx, b, c0, s0, cb);
    // counters zeroed by the caller; the test hook names a plan-wide item (cell)
    const int64_t wh = p.withhold_item >= c0 && p.withhold_item < c0 + nc ? p.withhold_item - c0 : -1;
    const int tpi = std::min(p.fused_tpi, std::min(C1::TILES, C2::TILES));
    FusedCtl ctl{cb.ctl, cb.ctl + 1, cb.ctl + 1 + nc, p.qerr, nc, p.fused_slots, p.fused_ahead, tpi, wh};
    constexpr size_t smem = C1::SMEM > C2::SMEM ? C1::SMEM : C2::SMEM;
    // pass-1 columns known zero beyond 3/8 of their length (radix-32 first stage) or 1/2
    const bool z3 = eng2::radix0(C1::M) == 32 && 8 * b.n <= 3 * (int64_t)C1::N;
    auto k = z3 ? k_search_fused<LOGN, LOWER, eng2::radix0(C1::M) == 32 ? 3 : 4>
                : k_search_fused<LOGN, LOWER, 4>;
    static Resident resident[2];
    const int res = resident[z3 ? 1 : 0](k, 256, smem);
    const int64_t items = (nc + p.fused_ahead) * (int64_t)(C1::TILES / tpi + C2::TILES / tpi);
    const unsigned grid = (unsigned)std::min<int64_t>(items, res);
    k<<<grid, 256, smem, s>>>(ld1, st1, ld2, st2, tw->s1_f, tw->s2_f, ctl);
    return 1;
}

template <int LOGN>
int launch_search2(const Plan &p, int band_idx, const BandDev &b, int64_t s0, int64_t c0,
                   int64_t nc, cudaStream_t s, cudaEvent_t mid, const CellBufs &cb) {
    using C1 = Cfg2<LOGN, 1>;
    using C2 = Cfg2<LOGN, 2>;
    const TwiddleSet *tw = p.twiddles(LOGN);
    const int n_spin = (int)p.desc.n_spin;

    SearchLoad2<C1> ld1{};
    ld1.w = reinterpret_cast<const float4 *>(cb.w);
    ld1.w_stride = p.w_stride;
    ld1.n = (int)b.n;
    ld1.chirp = p.chirp_fx + (int64_t)band_idx * n_spin;
    ld1.n_spin = n_spin;
    ld1.c0 = c0;
    ld1.s0 = s0;
    ScratchStore2<C1> st1{};
    st1.scratch = reinterpret_cast<float2 *>(cb.scratch);
    ScratchLoad2<C2> ld2{};
    ld2.scratch = reinterpret_cast<const float2 *>(cb.scratch);
    ld2.tw = {tw->lo_f, tw->hi_f};
    ld2.pf_dist = p.pf_dist;
    const bool lower = b.hi < (int64_t)C2::N / 2;
    if constexpr (LOGN < 20) if (fused_supported(p, LOGN) && cb.ctl) {
        return lower ? launch_fused<LOGN, true>(p, band_idx, b, s0, c0, nc, s, cb, ld1, st1, ld2, tw)
                     : launch_fused<LOGN, false>(p, band_idx, b, s0, c0, nc, s, cb, ld1, st1, ld2, tw);
    }
    return lower ? launch_two<LOGN, true>(p, band_idx, b, s0, c0, nc, s, mid, cb, ld1, st1, ld2, tw)
                 : launch_two<LOGN, false>(p, band_idx, b, s0, c0, nc, s, mid, cb, ld1, st1, ld2, tw);
}

// Interbinning form: both passes at length 2^LOGN = n_fft / 2 (pass 1 without
// the zero-half assumption), pass 2 in overlapping row tiles.
template <int LOGN>
int launch_interbin(const Plan &p, int band_idx, const BandDev &b, int64_t s0, int64_t c0,
                    int64_t nc, cudaStream_t s, cudaEvent_t mid, const CellBufs &cb) {
    using C1 = Cfg2<LOGN, 1>;
    using C2 = Cfg2<LOGN, 2>;
    const TwiddleSet *tw = p.twiddles(LOGN);
    const int n_spin = (int)p.desc.n_spin;
    SearchLoad2<C1> ld1{};
    ld1.w = reinterpret_cast<const float4 *>(cb.w);
    ld1.w_stride = p.w_stride;
    ld1.n = (int)b.n;
    ld1.chirp = p.chirp_fx + (int64_t)band_idx * n_spin;
    ld1.n_spin = n_spin;
    ld1.c0 = c0;
    ld1.s0 = s0;
    ScratchStore2<C1> st1{};
    st1.scratch = reinterpret_cast<float2 *>(cb.scratch);
    // The last quarter of a column is skipped when it lies beyond the series.  Lane pairs share
    // the spindown phases with a radix-16 or smaller first stage; with radix 32 the 24 or 32
    // inputs leave no registers for the exchange.  Measured (n_fft x cells = 2^30, shared against
    // not): 256-point columns 1.90 against 1.99 ms with the quarter skipped, 2.41 against 2.54
    // without; 512-point 1.95 against 1.91 and 2.43 against 2.34; 1024-point 2.61 against 2.47
    // and 3.04 against 2.75.
    const bool z6 = 4 * b.n <= 3 * (int64_t)C1::N;
    constexpr bool kShare = eng2::radix0(C1::N2) < 32;
    SearchLoad2S<C1> l1s{};
    static_cast<SearchLoad2<C1> &>(l1s) = ld1;
    auto run = [&](auto k1, const auto &ld) {
        set_smem(k1, C1::SMEM);
        k1<<<dim3(C1::TILES, (unsigned)nc), C1::THREADS, C1::SMEM, s>>>(ld, st1, tw->s2_f);
    };
    if (z6 && kShare && p.share_chirp) run(k_pass2<LOGN, 1, eng2::kMapFJ, SearchLoad2S<C1>, ScratchStore2<C1>, 256, 6>, l1s);
    else if (z6) run(k_pass2<LOGN, 1, eng2::kMapFJ, SearchLoad2<C1>, ScratchStore2<C1>, 256, 6>, ld1);
    else if (kShare && p.share_chirp) run(k_pass2<LOGN, 1, eng2::kMapFJ, SearchLoad2S<C1>, ScratchStore2<C1>, 256, 8>, l1s);
    else run(k_pass2<LOGN, 1, eng2::kMapFJ, SearchLoad2<C1>, ScratchStore2<C1>, 256, 8>, ld1);
    if (mid) record_timing_event(mid, s);
    if constexpr (LOGN <= 17) {
        if (rows_packed(p)) {
            constexpr int W = ib_warps(LOGN);
            constexpr RowRange all{0, p3::RowGeom<LOGN, W>::TILES_IB};
            if (b.hi < (int64_t)C2::N) launch_rows<LOGN, true, true, W>(p, band_idx, b, s0, c0, nc, s, cb, tw, all);
            else launch_rows<LOGN, false, true, W>(p, band_idx, b, s0, c0, nc, s, cb, tw, all);
            return 2;
        }
    }
    if (p.tma) {   // 128-thread row tiles staged by bulk copies (8-byte mbarrier after the smem)
        using D2 = Cfg2<LOGN, 2, 128>;
        ScratchLoadIBTMA<D2> ld2{};
        ld2.scratch = reinterpret_cast<const float2 *>(cb.scratch);
        ld2.tw = {tw->lo_f, tw->hi_f};
        ld2.pf_dist = 2 * p.pf_dist;
        ld2.err = p.qerr;
        const auto ep = make_epi<LOGN, false, 128>(p, band_idx, b, c0, s0, cb);
        auto k2 = k_pass2_ib<LOGN, 128, ScratchLoadIBTMA<D2>>;
        set_smem(k2, D2::SMEM + 16);
        k2<<<dim3(IBGeom<LOGN, 128>::TILES, (unsigned)nc), D2::THREADS, D2::SMEM + 16, s>>>(ld2, ep, tw->in1_f);
        return 2;
    }
    ScratchLoadIB<C2> ld2{};
    ld2.scratch = reinterpret_cast<const float2 *>(cb.scratch);
    ld2.tw = {tw->lo_f, tw->hi_f};
    const auto ep = make_epi<LOGN, false>(p, band_idx, b, c0, s0, cb);
    auto k2 = k_pass2_ib<LOGN, 256, ScratchLoadIB<C2>>;
    set_smem(k2, C2::SMEM);
    k2<<<dim3(IBGeom<LOGN>::TILES, (unsigned)nc), C2::THREADS, C2::SMEM, s>>>(ld2, ep, tw->in1_f);
    return 2;
}

// Row factors of the four-step twiddle: entry [i][m] holds the pair (W_N^{G l2 m},
// W_N^{G l2 m} W_32^m) of row l2 = i (512- and 1024-point rows, G = 16 and 32), or
// (W_N^{G l2 m}, W_N^{G (l2+1) m}) of the rows l2 = 2i, 2i + 1 (N1 <= 256, G = N1 / 16).
__global__ void k_row_twiddles(float4 *t, int logn) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int n1 = log_n1(logn), n2 = log_n2(logn);
    const bool pairs = n1 <= 8;
    if (i >= (p3::kRowTw << (pairs ? n2 - 1 : n2))) return;
    const int e = i / p3::kRowTw, m = i % p3::kRowTw;
    const double N = (double)(int64_t(1) << log_n(logn));
    const int64_t g = pairs ? 1 << (n1 - 4) : 1 << (n1 - 5);
    const double a = pairs ? (double)(g * 2 * e * m) / N : (double)(g * e * m) / N;
    const double b = pairs ? (double)(g * (2 * e + 1) * m) / N : a + (double)m / 32.0;
    double sa, ca, sb, cb;
    sincospi(2.0 * a, &sa, &ca);
    sincospi(2.0 * b, &sb, &cb);
    t[i] = make_float4((float)ca, (float)cb, (float)-sa, (float)-sb);
}

}  // namespace

int64_t row_twiddle_entries(int logn) {
    const int n1 = log_n1(logn), n2 = log_n2(logn);
    return n1 < 6 || n1 > 10 ? 0 : (int64_t)p3::kRowTw << (n1 <= 8 ? n2 - 1 : n2);
}

void launch_row_twiddles(float4 *t, int logn, cudaStream_t s) {
    k_row_twiddles<<<(unsigned)((row_twiddle_entries(logn) + 255) / 256), 256, 0, s>>>(t, logn);
}

// 2^19 points as 512-point columns and 1024-point rows: the columns move in 128-byte runs
// where 1024-point columns have 64, and the packed 1024-point rows cost less than that.
// Measured per 2^18 points, both passes: 0.977 + 0.627 -> 0.755 + 0.735 us (n <= 3N/8), 1.081 +
// 0.627 -> 0.860 + 0.734 (n > 3N/8).
int search_key_f32(const Plan &p, int logn) {
    const bool tall = logn == 19 && p.engine == 2 && !p.interbin && !p.fused && packed_rows(p);
    return tall ? kTall + logn : logn;
}

int pass2_threads_f32(const Plan &p, const BandDev &b) {
    const int lg = b.logn - (p.interbin ? 1 : 0);
    if (p.interbin) return lg <= 17 && rows_packed(p) ? 32 * ib_warps(lg) : p.tma ? 128 : 256;
    if (p.engine == 1 || lg < 12 || fused_supported(p, lg)) return 256;
    const int key = search_key_f32(p, lg);
    if (log_n1(key) == 10) return 64;
    if (key >= 18 && packed_rows(p)) return p.p2_ts;
    if (key <= 17 && rows_packed(p)) return 32;
    return p.tma ? p.p2_threads : 256;
}

bool interbin_supported(int logn) { return logn - 1 >= 12 && logn - 1 <= 19; }

bool fused_supported(const Plan &p, int logn) {
    return p.engine == 2 && p.fused && !p.interbin && logn >= 12 && logn <= 19;
}

int launch_search_cells_f32(const Plan &p, int band_idx, const BandDev &b, int64_t s0,
                            int64_t c0, int64_t nc, cudaStream_t s, cudaEvent_t mid,
                            const CellBufs &cb) {
    if (p.interbin) {
        switch (b.logn - 1) {
            case 12: return launch_interbin<12>(p, band_idx, b, s0, c0, nc, s, mid, cb);
            case 13: return launch_interbin<13>(p, band_idx, b, s0, c0, nc, s, mid, cb);
            case 14: return launch_interbin<14>(p, band_idx, b, s0, c0, nc, s, mid, cb);
            case 15: return launch_interbin<15>(p, band_idx, b, s0, c0, nc, s, mid, cb);
            case 16: return launch_interbin<16>(p, band_idx, b, s0, c0, nc, s, mid, cb);
            case 17: return launch_interbin<17>(p, band_idx, b, s0, c0, nc, s, mid, cb);
            case 18: return launch_interbin<18>(p, band_idx, b, s0, c0, nc, s, mid, cb);
            case 19: return launch_interbin<19>(p, band_idx, b, s0, c0, nc, s, mid, cb);
            default: return -1;
        }
    }
    if (p.engine == 2) {
        switch (b.logn) {
            case 12: return launch_search2<12>(p, band_idx, b, s0, c0, nc, s, mid, cb);
            case 13: return launch_search2<13>(p, band_idx, b, s0, c0, nc, s, mid, cb);
            case 14: return launch_search2<14>(p, band_idx, b, s0, c0, nc, s, mid, cb);
            case 15: return launch_search2<15>(p, band_idx, b, s0, c0, nc, s, mid, cb);
            case 16: return launch_search2<16>(p, band_idx, b, s0, c0, nc, s, mid, cb);
            case 17: return launch_search2<17>(p, band_idx, b, s0, c0, nc, s, mid, cb);
            case 18: return launch_search2<18>(p, band_idx, b, s0, c0, nc, s, mid, cb);
            case 19:
                return search_key_f32(p, 19) == 19 ? launch_search2<19>(p, band_idx, b, s0, c0, nc, s, mid, cb)
                                                   : launch_search2<kTall + 19>(p, band_idx, b, s0, c0, nc, s, mid, cb);
            case 20: return launch_search2<20>(p, band_idx, b, s0, c0, nc, s, mid, cb);
            default: break;
        }
    }
    return launch_search_dispatch<float>(p, band_idx, b, s0, c0, nc, s, mid, cb);
}
}  // namespace fstat
