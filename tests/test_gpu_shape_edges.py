"""Every bin against the FP64 oracle at the edges of the launch rules: series just inside
and just beyond the lengths where a kernel skips more of the zero padding, the shortest and
longest transforms of each engine, and grids whose last sky batch and last launch are ragged.
Tolerances as in test_gpu_parity: |F - F_ref| / max(F_ref, 2) <= 1e-10 (FP64), 1e-4 (FP32).
"""
import math
import os

import numpy as np
import pytest

import oracle as O
from paper_1410_3677_gb300 import synth as S

pytestmark = pytest.mark.gpu

TOL = {0: 1e-10, 1: 1e-4}
NTHREADS = os.cpu_count() or 4


@pytest.fixture(scope="module")
def fs():
    from paper_1410_3677_gb300 import fstat
    return fstat


def _check(fs, form, n, n_fft, n_sky, n_spin, dt=2.0, f_off=100.5, full_range=False, full=False, U=2,
           interbin=False, window=None):
    """Every bin (or `window` bins at three places of the range) of every cell."""
    alpha, delta = S.fibonacci_sky(n_sky)
    fdot = S.spindown_grid(n_spin, -1e-8, 0.0)
    b = S.make_band(n, dt, 31 + n, 1.0, alpha, delta, fdot, [], f_off=f_off, n_fft=n_fft)
    top = n_fft - 1 if full_range else n_fft // 2 - 1
    ranges = [(0 if full_range else 1, top)]
    if window:
        ranges = [(lo, lo + window - 1) for lo in (ranges[0][0], top // 2, top - window + 1)]
    prm = O.params(S.LAT_DEFAULT, S.GAMMA_DEFAULT, U, 0.0, full, 0, interbin)
    sky, spin = np.repeat(np.arange(n_sky), n_spin), np.tile(np.arange(n_spin), n_sky)
    for lo, hi in ranges:
        ref = O.cells_F(b, prm, alpha, delta, fdot, sky, spin, lo, hi, NTHREADS)
        with fs.Plan([b], alpha, delta, fdot, -1.0, lat=S.LAT_DEFAULT, gamma=S.GAMMA_DEFAULT, upsample=U, form=form,
                     bin_lo=lo, bin_hi=hi, cand_capacity=ref.size, full=full, interbin=interbin) as p:
            p.search()
            c, total = p.candidates()
        assert total == ref.size
        assert np.array_equal(c["bin"], np.tile(np.arange(lo, hi + 1), sky.size))
        assert np.array_equal(c["sky"] * n_spin + c["spin"], np.repeat(np.arange(sky.size), hi - lo + 1))
        err = np.abs(c["F"].reshape(ref.shape) - ref) / np.maximum(ref, 2.0)
        assert err.max() <= TOL[form], (lo, hi, err.max(), np.unravel_index(np.argmax(err), err.shape))


@pytest.mark.parametrize("n,n_fft,n_sky,n_spin,kw", [
    (1900, 1 << 12, 70, 3, {}),                                  # shortest two-stage length, ragged sky batch
    (2048, 1 << 12, 3, 2, dict(full_range=True)),                # n = N / 2, both halves of the spectrum
    (1001, 1 << 11, 5, 3, {}),                                   # longest of the radix-8 engine, batched
    (49152, 1 << 17, 2, 2, dict(full=True)),                     # n = 3N/8: five eighths of a column skipped
    (49153, 1 << 17, 2, 2, dict(full_range=True)),               # one sample more: half skipped
    (300001, 1 << 20, 3, 7, dict(dt=0.5, window=300)),           # longest, 1024-point rows, ragged last launch
])
def test_fp64_batches(fs, n, n_fft, n_sky, n_spin, kw):
    _check(fs, fs.FP64_PLAIN, n, n_fft, n_sky, n_spin, **kw)


@pytest.mark.parametrize("n,U", [(16, 2), (128, 3), (255, 2), (256, 2), (257, 5), (1024, 2), (2047, 8), (4097, 4),
                                 (8191, 3), (65536, 2), (86165, 3), (262147, 2)])
def test_upsample(fs, n, U):
    """The FFT upsample at odd and even lengths, powers of two (circular convolution of that
    length) and just beside them, and several factors, through the FP64 form's F at identity
    resampling positions of the upsampled series: an ephemeris that moves the samples by a
    constant j + s/U picks sub-phase s alone (s and U: s/U is a multiple of 1/U)."""
    rng = np.random.default_rng(n + U)
    nf = max(256, S.n_fft_auto(n))
    x = rng.standard_normal(n)
    one = np.zeros(1)
    for s in {1, U // 2, U - 1}:
        r = np.zeros((n, 3))
        r[:, 0] = -2.0 * s / U          # nhat = (1, 0, 0): every sample read s/U later, dt = 2
        b = S.Band(n=n, dt=2.0, f_off=0.0, x=x, r=r, phi0=0.3, eps=0.0, n_fft=nf, sigma=1.0)
        prm = O.params(S.LAT_DEFAULT, S.GAMMA_DEFAULT, U, 1.0, False, 0)
        lo, hi = 1, min(nf // 2 - 1, 3000)
        ref = O.cells_F(b, prm, one, one, one, np.array([0]), np.array([0]), lo, hi, NTHREADS)
        with fs.Plan([b], one, one, one, -1.0, lat=S.LAT_DEFAULT, gamma=S.GAMMA_DEFAULT, upsample=U, form=fs.FP64_PLAIN,
                     sigma2=1.0, bin_lo=lo, bin_hi=hi, cand_capacity=ref.size) as p:
            p.search()
            c, total = p.candidates()
        assert total == ref.size
        err = np.abs(c["F"] - ref[0]) / np.maximum(ref[0], 2.0)
        assert err.max() <= TOL[0], (s, err.max())


@pytest.mark.parametrize("n,n_fft,n_sky,n_spin,kw", [
    (300001, 1 << 20, 3, 5, dict(dt=0.5, window=2000)),
    (393216, 1 << 20, 2, 2, dict(dt=0.5, window=2000, full=True)),          # n = 3N/8
    (393217, 1 << 20, 2, 2, dict(dt=0.5, window=2000, full_range=True)),    # half of a column, both spectrum halves
    (524288, 1 << 20, 1, 2, dict(dt=0.5, window=2000, f_off=0.0)),          # n = N / 2
    (172328, 1 << 19, 2, 3, dict(window=2000)),                             # 512-point columns
    (196608, 1 << 19, 2, 2, dict(window=2000, full=True)),                  # n = 3N/8
    (196609, 1 << 19, 2, 2, dict(window=2000, full_range=True)),
])
def test_fp32_1024_point_rows(fs, n, n_fft, n_sky, n_spin, kw):
    _check(fs, fs.FP32_BATCHED, n, n_fft, n_sky, n_spin, **kw)


@pytest.mark.parametrize("n,dt,scale", [(1023, 2.0, 1.0), (1024, 2.0, 1.0), (1025, 0.5, 1.0), (3000, 0.3, 1.0), (5000, 60.0, 1.0),
                                        (2049, 0.01, 1.0), (3000, 2.0, 8.0)])
def test_fp32_sky_stage_tiles(fs, n, dt, scale):
    """The per-sky stage around its 1024-sample tiles: sampling intervals that are no power of
    two, long ones (the hour angle turns far within a tile), short ones (the delay is many tiles
    long and most samples fall outside the window), and an orbit eight times too large, whose
    delay drifts past the shared window's margin within a tile.  Tolerances of
    test_sky_stage_matches_oracle; S on the scale of its own sum."""
    nf = max(4096, S.n_fft_auto(n))
    one = np.array([0.7]), np.array([0.4]), np.array([0.0])
    b = S.make_band(n, dt, 5 + n, 1.0, *one, [], f_off=100.5, n_fft=nf)
    b.r = b.r * scale + (0.02 * np.sin(np.arange(n) * 0.7)[:, None] if scale > 1 else 0.0)
    prm = O.params(S.LAT_DEFAULT, S.GAMMA_DEFAULT, 2, 0.0)
    xu = O.upsample(b.x, 2)
    with fs.Plan([b], *one, 20.0, lat=S.LAT_DEFAULT, gamma=S.GAMMA_DEFAULT, form=fs.FP32_BATCHED) as p:
        g = p.debug_sky(0, 0, n)
    r = O.sky_prepare(b, prm, xu, float(one[0][0]), float(one[1][0]))
    assert np.array_equal(g["mask"], r["mask"])
    assert np.max(np.abs(g["a"] - r["a"])) < 2e-6 and np.max(np.abs(g["b"] - r["b"])) < 2e-6
    # phase: 2 pi (FP32 rounding of the position, 1.2e-7 samples, times f_off d' dt plus 1e-7 cycles) and
    # the interpolated series' slope (pi per sample) times the position's error, against 2e-5
    assert np.max(np.abs(g["y"] - r["y"])) / max(1.0, np.max(np.abs(r["y"]))) < 2e-5
    m = r["mask"]
    if m.any():
        sc = np.array([r["S"][0], r["S"][1], math.sqrt(r["S"][0] * r["S"][1])])
        assert np.max(np.abs(g["S"] - r["S"]) / sc) < 1e-5


@pytest.mark.parametrize("interbin", [False, True])
@pytest.mark.parametrize("lg", [12, 13, 14, 15, 16, 17])
@pytest.mark.parametrize("kw", [dict(), dict(full=True), dict(full_range=True)])
def test_packed_short_rows(fs, lg, interbin, kw):
    """Rows of 64, 128 and 256 points in packed pairs (transforms of 2^12 .. 2^17; for the
    interbinning form n_fft is twice that), every bin: both statistics, the lower half and the
    whole of the spectrum (the interbinning form's wrap from the last row to row 0)."""
    nf = 1 << (lg + 1 if interbin else lg)
    _check(fs, fs.FP32_BATCHED, nf // 3 + 7, nf, 2, 2, interbin=interbin, **kw)


@pytest.mark.parametrize("n", [1 << 13, (1 << 13) - 1, 3 << 11, (3 << 11) + 1])
def test_interbin_long_series(fs, n):
    """Interbinning at n = N (no zero padding left in the half-length transform) and around
    three quarters of it."""
    _check(fs, fs.FP32_BATCHED, n, 1 << 14, 3, 2, interbin=True)


@pytest.mark.parametrize("form,n,n_fft", [(1, n, f) for n, f in (
    (2000, 1 << 12), (4096, 1 << 13), (5000, 1 << 14), (16000, 1 << 15), (20000, 1 << 16), (60000, 1 << 17),
    (86164, 1 << 18), (131000, 1 << 18), (172328, 1 << 19), (250000, 1 << 19), (344656, 1 << 20),
    (500000, 1 << 20))] + [(0, 2000, 1 << 12), (0, 20000, 1 << 16), (0, 86164, 1 << 18)])
def test_narrow_bin_ranges(fs, form, n, n_fft):
    """Bin ranges shorter than the N2 rows of the transform search some rows only: one bin, a
    range across the last row and the first, half of the rows and one row more, all rows but one,
    all; below and above N / 2."""
    n2 = 1 << ((n_fft.bit_length() - 1 + 1) // 2)
    alpha, delta = S.fibonacci_sky(2)
    fdot = S.spindown_grid(2, -1e-8, 0.0)
    b = S.make_band(n, 0.5, 17 + n, 1.0, alpha, delta, fdot, [], f_off=100.5, n_fft=n_fft)
    prm = O.params(S.LAT_DEFAULT, S.GAMMA_DEFAULT, 2, 0.0, False, 0, False)
    sky, spin = np.repeat(np.arange(2), 2), np.tile(np.arange(2), 2)
    base = 3 * n2
    ranges = [(base + 5, base + 5), (base - 3, base + 2), (base + 1, base + n2 // 2), (base + 1, base + n2 // 2 + 1),
              (base + 2, base + n2), (base + 2, base + n2 + 1), (n_fft - n2 - 3, n_fft - n2 + 2),
              (n_fft // 2 - 2, n_fft // 2 + 1)]
    for lo, hi in ranges:
        ref = O.cells_F(b, prm, alpha, delta, fdot, sky, spin, lo, hi, NTHREADS)
        with fs.Plan([b], alpha, delta, fdot, -1.0, lat=S.LAT_DEFAULT, gamma=S.GAMMA_DEFAULT, form=form,
                     bin_lo=lo, bin_hi=hi, cand_capacity=ref.size + 64) as p:
            p.search()
            c, total = p.candidates()
        assert total == ref.size, (lo, hi)
        assert np.array_equal(c["bin"], np.tile(np.arange(lo, hi + 1), sky.size))
        err = np.abs(c["F"].reshape(ref.shape) - ref) / np.maximum(ref, 2.0)
        assert err.max() <= TOL[form], (lo, hi, err.max())


@pytest.mark.parametrize("lg,n_sky,n_spin", [(13, 8, 4), (13, 128, 4), (12, 32, 2), (14, 32, 2), (15, 32, 2)])
def test_fp32_error_beside_a_strong_line(fs, lg, n_sky, n_spin):
    """Short segments with a line of SNR 20 (at 2^13 the tiny grid), every bin: an amplitude
    error of the demodulated series that is common to many samples shows in the weak bins
    beside the line.  A relative amplitude error e of the line changes a bin of F by up to
    2 e sqrt(F F_max), relative to max(F, 2) at most 2 e sqrt(F_max / 2); the bound allows
    e = 4 x 2^-24."""
    if lg == 13:
        w = S.workload(1, n_sky=n_sky, n_spin=n_spin)
        b, alpha, delta, fdot = w.bands[0], w.alpha, w.delta, w.fdot
    else:
        alpha, delta = S.fibonacci_sky(n_sky)
        fdot = S.spindown_grid(n_spin, -3e-9, 0.0)
        inj = S.Injection(sky=5, spin=1, bin=int(0.2 * (1 << lg)), snr=20.0, cos_iota=0.3, psi=0.2, phi0=1.0)
        b = S.make_band(1 << (lg - 1), 2.0, 1000 + lg, 1.0, alpha, delta, fdot, [inj], n_fft=1 << lg)
    prm = O.params(S.LAT_DEFAULT, S.GAMMA_DEFAULT, 2, 0.0, False, 0)
    sky, spin = np.repeat(np.arange(n_sky), n_spin), np.tile(np.arange(n_spin), n_sky)
    ref = O.cells_F(b, prm, alpha, delta, fdot, sky, spin, nthreads=NTHREADS)
    with fs.Plan([b], alpha, delta, fdot, -1.0, lat=S.LAT_DEFAULT, gamma=S.GAMMA_DEFAULT, form=fs.FP32_BATCHED,
                 cand_capacity=ref.size) as p:
        p.search()
        c, total = p.candidates()
    assert total == ref.size and ref.max() > 100.0
    err = np.abs(c["F"].reshape(ref.shape) - ref) / np.maximum(ref, 2.0)
    assert err.max() <= 4 * 2.0 ** -24 * 2.0 * math.sqrt(ref.max() / 2.0), (err.max(), ref.max())


@pytest.mark.parametrize("form,n,n_fft", [(1, 2000, 1 << 12), (1, 5000, 1 << 14), (1, 60000, 1 << 17), (1, 86164, 1 << 18),
                                          (1, 172328, 1 << 19), (1, 344656, 1 << 20), (0, 20000, 1 << 16)])
def test_narrow_bin_ranges_full_statistic(fs, form, n, n_fft):
    """The launches over some of the rows with the cross term give the records of a search of all
    bins, bit for bit: one bin, a range across the last row and the first, and half of the rows."""
    n2 = 1 << ((n_fft.bit_length() - 1 + 1) // 2)
    alpha, delta = S.fibonacci_sky(2)
    fdot = S.spindown_grid(2, -1e-8, 0.0)
    b = S.make_band(n, 0.5, 19 + n, 1.0, alpha, delta, fdot, [], f_off=100.5, n_fft=n_fft)

    def records(lo, hi):
        with fs.Plan([b], alpha, delta, fdot, -1e9, lat=S.LAT_DEFAULT, gamma=S.GAMMA_DEFAULT, form=form, full=True,
                     bin_lo=lo, bin_hi=hi, cand_capacity=4 * (hi - lo + 1)) as p:
            p.search()
            c, total = p.candidates()
        assert total == c.size == 4 * (hi - lo + 1)
        return c

    whole = records(0, 6 * n2)
    for lo, hi in ((3 * n2 + 5, 3 * n2 + 5), (3 * n2 - 3, 3 * n2 + 2), (n2 + 1, n2 + n2 // 2)):
        assert np.array_equal(records(lo, hi), whole[(whole["bin"] >= lo) & (whole["bin"] <= hi)])
