"""Read-back order of large candidate sets: above 65536 records the plan sorts
them on the device (stable radix sort by cell and bin) before the copy.  With a
threshold below every F the candidates are all searched bins of all cells, so
the expected list is known exactly; F must equal, record for record, the F of
the same search at a threshold whose few candidates take the host sort."""
import numpy as np
import pytest

from paper_1410_3677_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fs():
    from paper_1410_3677_gb300 import fstat
    return fstat


def _plan(fs, w, thr, **kw):
    return fs.Plan(w.bands, w.alpha, w.delta, w.fdot, thr, lat=w.lat, gamma=w.gamma,
                   upsample=w.upsample, cand_capacity=1 << 21, **kw)


@pytest.mark.parametrize("kw", [dict(form=1), dict(form=1, interbin=True), dict(form=0)],
                         ids=["fp32", "fp32-interbin", "fp64"])
def test_every_bin_in_order(fs, kw):
    w = S.workload(1)
    n_fft = w.bands[0].n_fft
    p = _plan(fs, w, -1.0, **kw)
    assert p.search() == 0, p.error()
    c, total = p.candidates()
    q = _plan(fs, w, 20.0, **kw)
    assert q.search() == 0
    few, _ = q.candidates()
    q.close()
    bins = np.arange(1, n_fft // 2)
    assert total == c.size == w.n_sky * w.n_spin * bins.size > (1 << 16)
    assert np.array_equal(c["bin"], np.tile(bins, w.n_sky * w.n_spin))
    cell = c["sky"] * w.n_spin + c["spin"]
    assert np.array_equal(cell, np.repeat(np.arange(w.n_sky * w.n_spin), bins.size))
    assert np.all(c["band"] == 0)
    # F attached to the right record: the few candidates of the higher threshold
    idx = (few["sky"] * w.n_spin + few["spin"]) * bins.size + (few["bin"] - 1)
    assert few.size > 0 and np.array_equal(c["F"][idx], few["F"])
    # a second read-back of the same search gives the same list
    c2, _ = p.candidates()
    p.close()
    assert np.array_equal(c, c2)


def test_sub_range_and_multi_band_order(fs):
    """Four float32 bands of the banded workload, a cell range that starts inside
    band 1: the sort key is relative to the first searched cell."""
    w = S.workload(4, n_sky=4, n_spin=2, n_bands=4)
    p = fs.Plan(w.bands, w.alpha, w.delta, w.fdot, -1.0, lat=w.lat, gamma=w.gamma,
                upsample=w.upsample, form=fs.FP32_BATCHED, cand_capacity=1 << 24)
    per_band = w.n_sky * w.n_spin
    lo, hi = per_band + 3, 3 * per_band + 5
    assert p.search(lo, hi) == 0, p.error()
    c, total = p.candidates()
    p.close()
    assert total == c.size > (1 << 16)
    key = np.stack([c["band"], c["sky"], c["spin"], c["bin"]])
    order = np.lexsort(key[::-1])
    assert np.array_equal(order, np.arange(c.size))
    cell = c["band"].astype(np.int64) * per_band + c["sky"] * w.n_spin + c["spin"]
    assert cell.min() == lo and cell.max() == hi - 1
    counts = np.bincount(cell - lo)
    for k, n in enumerate(counts):
        b = (lo + k) // per_band
        assert n == w.bands[b].n_fft // 2 - 1


def test_measured_roofline_denominators(fs):
    """The FP32 FMA rate lies between half and 1.05x of 128 FMA lanes per SM at the
    maximum clock; the L2-resident copy beats the HBM copy rate."""
    import torch
    props = torch.cuda.get_device_properties(0)
    tf = fs.measure_fp32_fma()
    nominal = props.multi_processor_count * 128 * 2 * 2.07e9 / 1e12
    assert 0.5 * nominal < tf < 1.05 * nominal, (tf, nominal)
    l2 = fs.measure_l2_copy(32 << 20)
    assert l2 > 7000.0, l2


@pytest.mark.parametrize("n_bins", [15, 64, 511, 512, 513, 1023, 1024, 1025, 2500])
def test_read_back_paths(fs, n_bins):
    """Read-backs of 8 cells x n_bins records on either side of the limits between the copy that
    comes with the search, the host sort and the device sort (4096 and 8192 records): the order,
    a limited read (cap), a second read, and the count."""
    w = S.workload(1, n_sky=4, n_spin=2)
    p = fs.Plan(w.bands, w.alpha, w.delta, w.fdot, -1.0, lat=w.lat, gamma=w.gamma, bin_lo=100, bin_hi=99 + n_bins,
                form=fs.FP32_BATCHED, cand_capacity=1 << 16)
    p.search()
    n = 8 * n_bins
    assert p.candidates_get_status(0)[2] == n
    few, total = p.candidates(cap=min(37, n))
    c, total2 = p.candidates()
    again, _ = p.candidates()
    p.close()
    assert total == total2 == n == c.size
    assert np.array_equal(c["sky"] * 2 + c["spin"], np.repeat(np.arange(8), n_bins))
    assert np.array_equal(c["bin"], np.tile(np.arange(100, 100 + n_bins), 8))
    assert np.array_equal(c["alpha"], w.alpha[c["sky"]]) and np.array_equal(c["fdot"], w.fdot[c["spin"]])
    assert np.array_equal(c["freq"], w.bands[0].f_off + c["bin"] / (w.bands[0].n_fft * w.bands[0].dt))
    assert np.array_equal(few, c[:few.size]) and np.array_equal(again, c)
