// fstat_cell_F_noalloc: the F-statistic of every bin of one cell from an
// already resampled and demodulated series, with no device allocation.  The two
// FFT passes are those of the FP32 search's two-stage engine; the intermediate between
// them lives in a file-scope device array instead of plan-owned memory.
//
// One cell is bound by latency: launches, the depth of a pass, the wait of the host.  So
// the tiles are small (64 or 128 threads: 8 to 128 CTAs instead of 2 to 64), the second
// launch is a programmatic dependent of the first (its launch and prologue run under the
// first pass) and a length's function attributes are set once.  Measured, per call
// from Python with the wait: 2^13 22.8 -> 15.7 us, 2^18 25.1 -> 19.2 us.
#include <mutex>

#include "passes2.cuh"

namespace fstat {

namespace {

constexpr int kNoallocMaxLogN = 18;
constexpr int64_t kNoallocScratch = int64_t(2) << kNoallocMaxLogN;   // float2: two transforms

// Twiddle tables per transform length 2^L, L = 12 .. 18, interleaved complex: the stage-1
// twiddles W_M^{rj} of the rows (M = N1 entries, [r][j]) and the columns (M = N2), W_N^k
// (k < N1), W_N^{k N1} (k < N2); the region of length L starts at tw_off(L).
constexpr int tw_len(int L) { return 2 * 2 * ((1 << (L / 2)) + (1 << (L - L / 2))); }
constexpr int tw_off(int L) { return L <= 12 ? 0 : tw_off(L - 1) + tw_len(L - 1); }
constexpr int kNoallocTw = tw_off(kNoallocMaxLogN + 1);

// Shared by every call in the process (on each device that loads the library).
static __device__ __align__(256) float2 g_noalloc_scratch[kNoallocScratch];
static __device__ __align__(256) float g_noalloc_tw[kNoallocTw];

// Device addresses of the two arrays, resolved once per device with that device
// current (in host code the symbol names are only host-side stand-ins), and which
// twiddle lengths have been filled on that device.
constexpr int kMaxDevices = 64;
struct DevState {
    float2 *scratch = nullptr;
    float *tw = nullptr;
    bool tw_ready[kNoallocMaxLogN + 1] = {};
    bool attr_set[kNoallocMaxLogN + 1][4] = {};   // function attributes of a length's variants
};
DevState g_dev[kMaxDevices];
std::mutex g_dev_mu;

__global__ void k_noalloc_twiddles(float *tw, int L) {
    const int n1 = 1 << (L / 2), n2 = 1 << (L - L / 2);
    const int64_t N = int64_t(1) << L;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    // e^{-2 pi i k / M} = (cospi(2k/M), -sinpi(2k/M)), evaluated in FP64
    auto put = [&](int slot, int64_t k, int64_t M) {
        double s, c;
        sincospi(2.0 * (double)k / (double)M, &s, &c);
        tw[2 * slot] = (float)c;
        tw[2 * slot + 1] = (float)-s;
    };
    auto stage1 = [&](int e, int M) { const int R0 = eng2::radix0(M); return (int64_t)((e / R0) * (e % R0) % M); };
    if (i < n1) put(i, stage1(i, n1), n1);
    else if (i < n1 + n2) put(i, stage1(i - n1, n2), n2);
    else if (i < 2 * n1 + n2) put(i, i - n1 - n2, N);
    else if (i < 2 * n1 + 2 * n2) put(i, (int64_t)(i - 2 * n1 - n2) * n1, N);
}

// Resolves the arrays' addresses and fills the twiddles of length 2^L on first
// use on the current device.  Returns false on a CUDA error.
bool setup_current_device(int L, DevState **out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return false;
    std::lock_guard<std::mutex> lk(g_dev_mu);
    DevState &d = g_dev[dev];
    if (!d.scratch) {
        void *a = nullptr, *b = nullptr;
        if (cudaGetSymbolAddress(&a, g_noalloc_scratch) != cudaSuccess) return false;
        if (cudaGetSymbolAddress(&b, g_noalloc_tw) != cudaSuccess) return false;
        d.scratch = static_cast<float2 *>(a);
        d.tw = static_cast<float *>(b);
    }
    if (!d.tw_ready[L]) {
        const int n = tw_len(L) / 2;
        k_noalloc_twiddles<<<(n + 255) / 256, 256>>>(d.tw + tw_off(L), L);
        if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) return false;
        d.tw_ready[L] = true;
    }
    *out = &d;
    return true;
}

// Pass-1 input: the search's loader on one series, with Taylor phases: the special function
// unit's were most of the error of F (rms over the lengths 2.8-3.9e-7 -> 1.9-2.4e-7; 2.6-4.3e-7 on
// the radix-8 passes) and these cost a lone cell no time.  The dependent launch may start at
// once; it waits for this grid's stores.
template <class C>
struct CellLoad : SearchLoad2S<C, true> {
    __device__ void init(int tile, int64_t, int64_t) {
        asm volatile("griddepcontrol.launch_dependents;");
        this->ws = reinterpret_cast<const float2 *>(this->w);
        this->k1_0 = tile * C::F;
    }
};

// Pass-2 input: the rows once the first grid is done.  The four-step twiddle comes from the
// tables for every fourth element and by one to three steps of a recurrence between: a
// recurrence over all of them adds a third to the rounding error of F, table entries for
// all of them 3 us to the longest call.
template <class C>
struct CellRows : ScratchLoad2<C> {
    template <int R, int JPF>
    __device__ __forceinline__ void load(const eng2::Job &q, float *re, float *im) const {
        constexpr int S = R < 4 ? R : 4;
        const int l2 = this->l2_0 + q.f;
        float2 w[R / S];
#pragma unroll
        for (int r = 0; r < R / S; ++r) w[r] = this->tw.wn(l2 * (q.j + S * r * JPF));
        const float2 st = this->tw.wn(l2 * JPF);
        asm volatile("griddepcontrol.wait;" ::: "memory");
        const float2 *row = this->base + 2 * ((int64_t)l2 * C::N1 + q.j) + q.t;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float2 v = __ldcg(row + 2 * r * JPF);
            re[r] = v.x; im[r] = v.y;
        }
#pragma unroll
        for (int r = 0; r < R; r += S) this->tw.template apply<S>(w[r / S], st, re + r, im + r);
    }
};

// Pass-2 output: F of every bin in [lo, hi] into out[bin - lo].  Lanes l (F_a) and l ^ 16
// (F_b) hold the same bins; the a lane evaluates the first half of the outputs, the b lane
// the second.
template <class C, bool LOWER>
struct CellFOut {
    float *out;
    float na, nb;
    int lo, hi;
    int l2_0;
    __device__ void init(int tile, int64_t, int64_t) { l2_0 = tile * C::F; }
    template <int R, int JPF>
    __device__ __forceinline__ void store(const eng2::Job &q, float *re, float *im) const {
        constexpr int H = (LOWER ? R / 2 : R) / 2;
        const int bin0 = C::N2 * (q.j + q.t * H * JPF) + l2_0 + q.f;
#pragma unroll
        for (int r = 0; r < H; ++r) {
            const float p_lo = re[r] * re[r] + im[r] * im[r];
            const float p_hi = re[r + H] * re[r + H] + im[r + H] * im[r + H];
            const float other = __shfl_xor_sync(0xffffffffu, q.t == 0 ? p_hi : p_lo, 16);
            const int bin = bin0 + r * C::N2 * JPF;
            if (bin >= lo && bin <= hi) out[bin - lo] = q.t == 0 ? p_lo * na + other * nb : other * na + p_hi * nb;
        }
    }
};

template <int LOGN, bool LOWER, int Z1>
fstat_status run_cell(const float4 *w, int n, uint64_t afx, float na, float nb, int lo, int hi, float *out,
                      float2 *scratch, const float *s1, const float *s2, const float *tw_lo, const float *tw_hi,
                      bool first, cudaStream_t s) {
    constexpr int TS1 = LOGN <= 15 ? 64 : 128, TS2 = 64;
    using C1 = Cfg2<LOGN, 1, TS1>;
    using C2 = Cfg2<LOGN, 2, TS2>;
    CellLoad<C1> ld1{};
    ld1.w = w;
    ld1.n = n;
    ld1.afx = afx;
    ScratchStore2<C1> st1{};
    st1.scratch = scratch;
    auto k1 = k_pass2<LOGN, 1, eng2::kMapFJ, CellLoad<C1>, ScratchStore2<C1>, TS1, Z1>;
    CellRows<C2> ld2{};
    ld2.scratch = scratch;
    ld2.tw = {tw_lo, tw_hi};
    CellFOut<C2, LOWER> st2{out, na, nb, lo, hi, 0};
    auto k2 = k_pass2<LOGN, 2, eng2::kMapW, CellRows<C2>, CellFOut<C2, LOWER>, TS2>;
    if (first &&
        (cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C1::SMEM) != cudaSuccess ||
         cudaFuncSetAttribute(k2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C2::SMEM) != cudaSuccess))
        return FSTAT_ERR_CUDA;
    k1<<<dim3(C1::TILES, 1), C1::THREADS, C1::SMEM, s>>>(ld1, st1, s2);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(C2::TILES, 1);
    cfg.blockDim = dim3(C2::THREADS);
    cfg.dynamicSmemBytes = C2::SMEM;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, k2, ld2, st2, s1) != cudaSuccess) return FSTAT_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? FSTAT_OK : FSTAT_ERR_CUDA;
}

template <int LOGN>
fstat_status run_length(DevState &d, const float4 *w, int n, uint64_t afx, float na, float nb, int lo, int hi,
                        float *out, cudaStream_t s) {
    constexpr int N = 1 << LOGN, n1 = 1 << (LOGN / 2), n2 = 1 << (LOGN - LOGN / 2);
    const float *s1 = d.tw + tw_off(LOGN), *s2 = s1 + 2 * n1, *tw_lo = s2 + 2 * n2, *tw_hi = tw_lo + 2 * n1;
    const bool lower = hi < N / 2;
    const bool z3 = eng2::radix0(n2) == 32 && 8 * (int64_t)n <= 3 * (int64_t)N;
    bool &set = d.attr_set[LOGN][(lower ? 2 : 0) + (z3 ? 1 : 0)];
    const bool first = !set;
    auto run = [&](auto f) {
        const fstat_status st = f(w, n, afx, na, nb, lo, hi, out, d.scratch, s1, s2, tw_lo, tw_hi, first, s);
        if (st == FSTAT_OK) set = true;
        return st;
    };
    if constexpr (eng2::radix0(n2) == 32)
        if (z3) return lower ? run(run_cell<LOGN, true, 3>) : run(run_cell<LOGN, false, 3>);
    return lower ? run(run_cell<LOGN, true, 4>) : run(run_cell<LOGN, false, 4>);
}

}  // namespace

}  // namespace fstat

extern "C" fstat_status fstat_cell_F_noalloc(const float *w, int64_t n, int64_t n_fft,
                                             double chirp_rate, double norm_a, double norm_b,
                                             int64_t bin_lo, int64_t bin_hi, float *F_out,
                                             void *cuda_stream) {
    using namespace fstat;
    int lg = 0;
    while ((int64_t(1) << lg) < n_fft) ++lg;
    // w is read as float4 (16-byte loads) and F_out written as floats: a view that
    // starts off those boundaries is refused here instead of faulting on the GPU
    if (!w || !F_out || (reinterpret_cast<uintptr_t>(w) & 15) != 0 ||
        (reinterpret_cast<uintptr_t>(F_out) & 3) != 0 || n < 1 || (int64_t(1) << lg) != n_fft || lg < 12 ||
        lg > kNoallocMaxLogN || 2 * n > n_fft || bin_lo < 0 || bin_hi < bin_lo || bin_hi >= n_fft ||
        !(norm_a >= 0.0) || !(norm_b >= 0.0))
        return FSTAT_ERR_ARG;
    DevState *d = nullptr;
    if (!setup_current_device(lg, &d)) return FSTAT_ERR_CUDA;
    // frac(rate) in 2^-64 cycles (the rate is |fdot| dt^2 / 2 << 1/4)
    if (!(fabs(chirp_rate) < 0.25)) return FSTAT_ERR_ARG;
    const uint64_t afx = (uint64_t)(int64_t)llround(ldexp(chirp_rate, 64));
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    const float4 *w4 = reinterpret_cast<const float4 *>(w);
    fstat_status st = FSTAT_ERR_ARG;
#define FSTAT_NOALLOC_CASE(L)                                                                                     \
    case L:                                                                                                       \
        st = run_length<L>(*d, w4, (int)n, afx, (float)norm_a, (float)norm_b, (int)bin_lo, (int)bin_hi, F_out, s); \
        break;
    switch (lg) {
        FSTAT_NOALLOC_CASE(12)
        FSTAT_NOALLOC_CASE(13)
        FSTAT_NOALLOC_CASE(14)
        FSTAT_NOALLOC_CASE(15)
        FSTAT_NOALLOC_CASE(16)
        FSTAT_NOALLOC_CASE(17)
        FSTAT_NOALLOC_CASE(18)
        default: return FSTAT_ERR_ARG;
    }
#undef FSTAT_NOALLOC_CASE
    if (st != FSTAT_OK) return st;
    return cudaStreamSynchronize(s) == cudaSuccess ? FSTAT_OK : FSTAT_ERR_CUDA;
}
