"""The allocation-free single-cell entry point, for callers that cannot allocate
device memory (they hold the device memory budget themselves and pass views).

It must reproduce, through the C ABI, the F of every bin that the plan-based
search computes for the same cell, on two calls in a row (two different cells),
within the FP32 tolerance of the other GPU tests, and refuse lengths beyond its
maximum.  This file is collected last."""
import math

import numpy as np
import pytest

from paper_1410_3677_gb300 import synth as S

pytestmark = pytest.mark.gpu


def _case(fs, w, cells):
    import torch
    band = w.bands[0]
    p = fs.Plan(w.bands, w.alpha, w.delta, w.fdot, -1.0, lat=w.lat, gamma=w.gamma,
                upsample=w.upsample, form=fs.FP32_BATCHED, cand_capacity=1 << 20)
    nb = band.n_fft // 2 - 1
    sigma2 = math.fsum(np.asarray(band.x, np.float64) ** 2) / band.n
    stream = torch.cuda.current_stream()
    out = torch.empty(nb, dtype=torch.float32, device="cuda")
    for sky, spin in cells:          # two calls in a row, different cells
        cell = sky * w.n_spin + spin
        assert p.search(cell, cell + 1) == fs.FSTAT_OK
        c, total = p.candidates()
        assert total == nb and np.array_equal(c["bin"], np.arange(1, nb + 1))
        g = p.debug_sky(0, sky, band.n)
        y = g["y"]
        a = g["a"].astype(np.float32)
        b = g["b"].astype(np.float32)
        yr, yi = y.real.astype(np.float32), y.imag.astype(np.float32)
        w4 = np.ascontiguousarray(np.stack([yr * a, yi * a, yr * b, yi * b], 1), np.float32)
        wt = torch.from_numpy(w4).cuda()
        out.fill_(float("nan"))
        rate = 0.5 * float(w.fdot[spin]) * band.dt * band.dt
        rc = fs.cell_F_noalloc(wt.data_ptr(), band.n, band.n_fft, rate, 1.0 / (sigma2 * g["S"][0]),
                               1.0 / (sigma2 * g["S"][1]), 1, nb, out.data_ptr(),
                               stream.cuda_stream)
        assert rc == fs.FSTAT_OK
        F = out.cpu().numpy().astype(np.float64)
        err = np.abs(F - c["F"]) / np.maximum(c["F"], 2.0)
        assert np.all(np.isfinite(F)) and err.max() <= 1e-4, (sky, spin, err.max())
    p.close()


def test_noalloc_matches_plan_two_calls():
    from paper_1410_3677_gb300 import fstat as fs
    _case(fs, S.workload(1, n_sky=6, n_spin=4), [(1, 2), (4, 0)])          # N_fft = 2^13
    w = S.workload(2, n_sky=1024, n_spin=1)
    inj = w.bands[0].injections[0]
    w2 = S.Workload(w.name, w.bands, w.alpha[[3, inj.sky]], w.delta[[3, inj.sky]], w.fdot, w.thr_2F)
    _case(fs, w2, [(1, 0), (0, 0)])                                          # N_fft = 2^18


def test_noalloc_rejects_beyond_maximum():
    import torch
    from paper_1410_3677_gb300 import fstat as fs
    buf = torch.zeros(4 * 8, dtype=torch.float32, device="cuda")
    out = torch.zeros(8, dtype=torch.float32, device="cuda")
    assert fs.cell_F_noalloc(buf.data_ptr(), 8, 1 << 19, 0.0, 1.0, 1.0, 1, 7, out.data_ptr()) == fs.FSTAT_ERR_ARG
    assert fs.cell_F_noalloc(buf.data_ptr(), 8, 1 << 11, 0.0, 1.0, 1.0, 1, 7, out.data_ptr()) == fs.FSTAT_ERR_ARG
    assert fs.cell_F_noalloc(0, 8, 1 << 12, 0.0, 1.0, 1.0, 1, 7, out.data_ptr()) == fs.FSTAT_ERR_ARG
    # views that start off the 16-byte (series) or 4-byte (output) boundary are
    # refused on the host, before anything is launched
    assert fs.cell_F_noalloc(buf.data_ptr() + 4, 8, 1 << 12, 0.0, 1.0, 1.0, 1, 7,
                             out.data_ptr()) == fs.FSTAT_ERR_ARG
    assert fs.cell_F_noalloc(buf.data_ptr(), 8, 1 << 12, 0.0, 1.0, 1.0, 1, 7,
                             out.data_ptr() + 2) == fs.FSTAT_ERR_ARG


def test_noalloc_allocates_no_device_memory():
    """The property the entry point exists for: once the kernels of a length are
    loaded (first call), further calls leave the device's free memory unchanged."""
    import torch
    from paper_1410_3677_gb300 import fstat as fs
    n, n_fft = 3000, 1 << 13
    rng = np.random.default_rng(7)
    w = torch.from_numpy(rng.standard_normal((n, 4)).astype(np.float32)).cuda()
    out = torch.empty(n_fft // 2 - 1, dtype=torch.float32, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    args = (w.data_ptr(), n, n_fft, 1e-7, 1.0, 1.0, 1, n_fft // 2 - 1, out.data_ptr(), stream)
    assert fs.cell_F_noalloc(*args) == fs.FSTAT_OK     # first call: set-up and module load
    first = out.clone()                                 # torch's own allocation, outside the window
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    for _ in range(3):
        assert fs.cell_F_noalloc(*args) == fs.FSTAT_OK
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free0
    assert torch.equal(out, first)                      # the shared scratch keeps no state
    del first


@pytest.mark.parametrize("lg", range(12, 19))
@pytest.mark.parametrize("frac,whole", [(0.33, False), (0.5, True)])
def test_noalloc_every_length(lg, frac, whole):
    """Every length, both column variants (n <= 3N/8 and n = N/2), half and whole bin range,
    an odd output window: against an FP64 transform of the same series."""
    import torch
    from paper_1410_3677_gb300 import fstat as fs
    N = 1 << lg
    n = int(frac * N)
    rng = np.random.default_rng(lg)
    w = rng.standard_normal((n, 4)).astype(np.float32)
    rate, na, nb = -1.7e-8, 1.0 / n, 2.0 / n
    k = np.arange(n, dtype=np.float64)
    ph = np.exp(-2j * np.pi * np.mod(rate * k * k, 1.0))
    A = np.fft.fft((w[:, 0] + 1j * w[:, 1].astype(np.float64)) * ph, N)
    B = np.fft.fft((w[:, 2] + 1j * w[:, 3].astype(np.float64)) * ph, N)
    lo, hi = (3, N - 2) if whole else (1, N // 2 - 1)
    ref = (np.abs(A) ** 2 * na + np.abs(B) ** 2 * nb)[lo:hi + 1]
    wd = torch.from_numpy(w).cuda()
    out = torch.full((hi - lo + 3,), -1.0, dtype=torch.float32, device="cuda")
    assert fs.cell_F_noalloc(wd.data_ptr(), n, N, rate, na, nb, lo, hi, out.data_ptr() + 4) == fs.FSTAT_OK
    got = out.cpu().numpy()
    assert got[0] == -1.0 and got[-1] == -1.0            # nothing outside the window
    assert np.max(np.abs(got[1:-1] - ref) / np.maximum(ref, 2.0)) <= 1e-4


@pytest.mark.parametrize("lg", range(12, 19))
@pytest.mark.parametrize("eighths,more", [(3, 0), (3, 1), (4, 0)])
def test_noalloc_rounding(lg, eighths, more):
    """Rms error of F over all bins of a noise series with a spindown of many cycles, against an
    FP64 transform.  About ten roundings of 2^-24 (uniform: 2^-24 / sqrt 3 rms) a transform value
    make 1.1e-7 of its amplitude, twice that of F; 2.5e-7 leaves an eighth.  n = 3N/8 is the
    longest series whose columns skip five eighths, 3N/8 + 1 the first whose do not."""
    import torch
    from paper_1410_3677_gb300 import fstat as fs
    N = 1 << lg
    n = eighths * N // 8 + more
    rng = np.random.default_rng(100 + lg)
    rate, na, nb, lo, hi = -1.7e-8, 1.0 / n, 2.0 / n, 1, N // 2 - 1
    rate *= (1 << 36) / float(n) ** 2                    # 1168 cycles over the series at any length
    k = np.arange(n, dtype=np.float64)
    ph = np.exp(-2j * np.pi * np.mod(rate * k * k, 1.0))
    sq, count = 0.0, 0
    for _ in range(max(1, (1 << 17) >> lg)):
        w = rng.standard_normal((n, 4)).astype(np.float32)
        A = np.fft.fft((w[:, 0] + 1j * w[:, 1].astype(np.float64)) * ph, N)
        B = np.fft.fft((w[:, 2] + 1j * w[:, 3].astype(np.float64)) * ph, N)
        ref = (np.abs(A) ** 2 * na + np.abs(B) ** 2 * nb)[lo:hi + 1]
        wd = torch.from_numpy(w).cuda()
        out = torch.empty(hi - lo + 1, dtype=torch.float32, device="cuda")
        assert fs.cell_F_noalloc(wd.data_ptr(), n, N, rate, na, nb, lo, hi, out.data_ptr()) == fs.FSTAT_OK
        sq += float(np.sum(((out.cpu().numpy() - ref) / np.maximum(ref, 2.0)) ** 2))
        count += ref.size
    assert np.sqrt(sq / count) <= 2.5e-7, np.sqrt(sq / count)
