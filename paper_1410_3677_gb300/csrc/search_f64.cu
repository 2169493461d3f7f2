// FP64 search passes (FSTAT_FP64_PLAIN): the two-stage engine in double precision
// (passes64.cuh) for transform lengths 2^12 .. 2^20, the radix-8 engine below
// (2^8 .. 2^11, whose rows are shorter than the two-stage engine takes).
#include "passes64.cuh"
#include "search_launch.cuh"

namespace fstat {
namespace {

__global__ void k_unit_table(double2 *t) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= p64::kUnitTab) return;
    double s, c;
    sincospi(2.0 * (double)i / (double)p64::kUnitTab, &s, &c);
    t[i] = make_double2(c, -s);
}

// W_N^{k1 l2} in the order of the scratch: [l2 / rb][k1][l2 % rb]
__global__ void k_inter_table(double2 *t, int logn, int rb) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t N = int64_t(1) << logn, n1 = int64_t(1) << (logn / 2);
    if (i >= N) return;
    const int64_t f = i % rb, k1 = (i / rb) % n1, l2 = i / rb / n1 * rb + f;
    double s, c;
    sincospi(2.0 * (double)(k1 * l2) / (double)N, &s, &c);
    t[i] = make_double2(c, -s);
}

template <int LOGN, bool LOWER, int Z1>
int launch_t(const Plan &p, int band_idx, const BandDev &b, int64_t s0, int64_t c0, int64_t nc, cudaStream_t s,
             cudaEvent_t mid, const CellBufs &cb) {
    using C1 = p64::Cfg64<LOGN, 1>;
    using C2 = p64::Cfg64<LOGN, 2>;
    const TwiddleSet *tw = p.twiddles(LOGN);
    const int n_spin = (int)p.desc.n_spin;
    using LD1 = p64::Load64<C1>;
    using ST1 = p64::Store64<C1, C2::F>;
    LD1 ld1{};
    ld1.w = reinterpret_cast<const double2 *>(cb.w);
    ld1.w_stride = p.w_stride;
    ld1.n = (int)b.n;
    ld1.chirp = p.chirp_d + (int64_t)band_idx * n_spin;
    ld1.n_spin = n_spin;
    ld1.c0 = c0;
    ld1.s0 = s0;
    ld1.tab = p.unit_tab;
    ST1 st1{};
    st1.scratch = reinterpret_cast<double2 *>(cb.scratch);
    auto k1 = p64::k_pass64<LOGN, 1, LD1, ST1, Z1>;
    set_smem(k1, C1::SMEM);
    k1<<<dim3(C1::TILES, (unsigned)nc), C1::THREADS, C1::SMEM, s>>>(ld1, st1, tw->s2_d);
    if (mid) record_timing_event(mid, s);

    using LD2 = p64::RowLoad64<C2>;
    using ST2 = p64::Epi64<C2, LOWER>;
    LD2 ld2{};
    ld2.scratch = reinterpret_cast<const double2 *>(cb.scratch);
    ld2.tw = tw->inter_d;
    ST2 st2{};
    st2.norm = cb.norm;
    st2.n_spin = n_spin;
    st2.c0 = c0;
    st2.s0 = s0;
    st2.cell_base = (uint32_t)((int64_t)band_idx * p.desc.n_sky * p.desc.n_spin);
    st2.bin_lo = b.lo;
    st2.bin_hi = b.hi;
    st2.thr = p.desc.thr_2F;
    st2.out = p.cand;
    st2.count = p.cand_count;
    st2.cap = (unsigned long long)p.cand_capacity;
    auto k2 = p64::k_pass64<LOGN, 2, LD2, ST2, 8>;
    set_smem(k2, C2::SMEM);
    const RowRange rr = searched_rows(b, C2::N2, C2::F);
    st2.tile0 = rr.tile0;
    k2<<<dim3(rr.tiles, (unsigned)nc), C2::THREADS, C2::SMEM, s>>>(ld2, st2, tw->s1_d);
    return 2;
}

template <int LOGN>
int launch_n(const Plan &p, int band_idx, const BandDev &b, int64_t s0, int64_t c0, int64_t nc, cudaStream_t s,
             cudaEvent_t mid, const CellBufs &cb) {
    const int64_t N = int64_t(1) << LOGN;
    const bool lower = b.hi < N / 2;
    if constexpr (eng2::radix0(1 << (LOGN - LOGN / 2)) == 32) {
        if (8 * b.n <= 3 * N)
            return lower ? launch_t<LOGN, true, 3>(p, band_idx, b, s0, c0, nc, s, mid, cb)
                         : launch_t<LOGN, false, 3>(p, band_idx, b, s0, c0, nc, s, mid, cb);
    }
    return lower ? launch_t<LOGN, true, 4>(p, band_idx, b, s0, c0, nc, s, mid, cb)
                 : launch_t<LOGN, false, 4>(p, band_idx, b, s0, c0, nc, s, mid, cb);
}

template <int L>
int block_of(int logn) {
    if constexpr (L > p64::kMaxLog) return 0;
    else return logn == L ? p64::row_block<L>() : block_of<L + 1>(logn);
}

}  // namespace

int64_t unit_table_entries() { return p64::kUnitTab; }
bool inter_table_needed(int logn) { return logn >= p64::kMinLog && logn <= p64::kMaxLog; }

void launch_unit_table(double2 *t, cudaStream_t s) { k_unit_table<<<p64::kUnitTab / 256, 256, 0, s>>>(t); }

void launch_inter_table(double2 *t, int logn, cudaStream_t s) {
    const int64_t N = int64_t(1) << logn;
    k_inter_table<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(t, logn, block_of<p64::kMinLog>(logn));
}

int launch_search_cells_f64(const Plan &p, int band_idx, const BandDev &b, int64_t s0,
                            int64_t c0, int64_t nc, cudaStream_t s, cudaEvent_t mid,
                            const CellBufs &cb) {
    switch (b.logn) {
        case 12: return launch_n<12>(p, band_idx, b, s0, c0, nc, s, mid, cb);
        case 13: return launch_n<13>(p, band_idx, b, s0, c0, nc, s, mid, cb);
        case 14: return launch_n<14>(p, band_idx, b, s0, c0, nc, s, mid, cb);
        case 15: return launch_n<15>(p, band_idx, b, s0, c0, nc, s, mid, cb);
        case 16: return launch_n<16>(p, band_idx, b, s0, c0, nc, s, mid, cb);
        case 17: return launch_n<17>(p, band_idx, b, s0, c0, nc, s, mid, cb);
        case 18: return launch_n<18>(p, band_idx, b, s0, c0, nc, s, mid, cb);
        case 19: return launch_n<19>(p, band_idx, b, s0, c0, nc, s, mid, cb);
        case 20: return launch_n<20>(p, band_idx, b, s0, c0, nc, s, mid, cb);
        case 8: return launch_search_t<double, 8, 256, 0>(p, band_idx, b, s0, c0, nc, s, mid, cb);
        case 9: return launch_search_t<double, 9, 256, 0>(p, band_idx, b, s0, c0, nc, s, mid, cb);
        case 10: return launch_search_t<double, 10, 256, 0>(p, band_idx, b, s0, c0, nc, s, mid, cb);
        case 11: return launch_search_t<double, 11, 256, 0>(p, band_idx, b, s0, c0, nc, s, mid, cb);
        default: return -1;
    }
}
}  // namespace fstat
