"""Plans beside little free device memory: a plan whose usual batches do not fit is created with
smaller ones and gives the same records."""
import os

import numpy as np
import pytest

from paper_1410_3677_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fs():
    from paper_1410_3677_gb300 import fstat
    return fstat


def _plan(fs, b, grid, form, thr, limit=None):
    if limit:
        os.environ["FSTAT_TEST_MEM_LIMIT"] = str(limit << 20)
    try:
        return fs.Plan([b], *grid, thr, lat=S.LAT_DEFAULT, gamma=S.GAMMA_DEFAULT, form=form, cand_capacity=1 << 20)
    finally:
        os.environ.pop("FSTAT_TEST_MEM_LIMIT", None)


# limits in MiB: one FP64 cell or 64 to 256 FP32 positions at a time, and a little more
@pytest.mark.parametrize("form,n,n_fft,n_sky,n_spin,thr,limits", [
    (0, 86164, 1 << 18, 70, 1, 26.0, (53, 150)),
    (0, 4096, 1 << 13, 32, 4, 16.0, (18, 25)),
    (0, 300001, 1 << 20, 2, 2, 30.0, (156,)),
    (0, 1000, 1 << 11, 5, 3, 8.0, (17,)),
    (1, 86164, 1 << 18, 1024, 1, 28.0, (2071,)),
    (1, 4096, 1 << 13, 700, 1, 16.0, (97,)),
])
def test_plan_fits_in_smaller_batches(fs, form, n, n_fft, n_sky, n_spin, thr, limits):
    alpha, delta = S.fibonacci_sky(n_sky)
    grid = alpha, delta, S.spindown_grid(n_spin, -1e-8, 0.0) if n_spin > 1 else np.array([-1e-9])
    b = S.make_band(n, 2.0, 3, 1.0, *grid, [], n_fft=n_fft)
    with _plan(fs, b, grid, form, thr) as p:
        assert p.info()["device_bytes"] > limits[0] << 20
        p.search()
        ref, total = p.candidates()
    assert total > 0
    for limit in limits:
        with _plan(fs, b, grid, form, thr, limit) as p:
            assert p.info()["device_bytes"] <= limit << 20
            p.search()
            c, total = p.candidates()
            p.search(n_sky * n_spin // 3, n_sky * n_spin - 1)      # part of the grid
            part, _ = p.candidates()
        assert np.array_equal(c, ref)
        cell = ref["sky"] * n_spin + ref["spin"]
        assert np.array_equal(part, ref[(cell >= n_sky * n_spin // 3) & (cell < n_sky * n_spin - 1)])
    with pytest.raises(fs.FstatError) as e:
        _plan(fs, b, grid, form, thr, 10)
    assert e.value.code == fs.FSTAT_ERR_OOM


@pytest.mark.parametrize("n_sky,n_spin,n_bins", [(4, 2, 1024), (4, 2, 4000), (70, 8, 117), (70, 8, 118)])
def test_read_back_without_room_to_sort(fs, n_sky, n_spin, n_bins):
    """8192 to 65 535 records are sorted on the host when the device has no room for the sort's
    second buffer, more are FSTAT_ERR_OOM; with room again the same plan sorts on the device."""
    w = S.workload(1, n_sky=n_sky, n_spin=n_spin)
    n = n_sky * n_spin * n_bins
    with fs.Plan(w.bands, w.alpha, w.delta, w.fdot, -1.0, lat=w.lat, gamma=w.gamma, bin_lo=50, bin_hi=49 + n_bins,
                 cand_capacity=1 << 17) as p:
        p.search()
        os.environ["FSTAT_TEST_MEM_LIMIT"] = str(p.info()["device_bytes"])
        try:
            got = [p.candidates_get_status(n) for _ in range(2)]
        finally:
            del os.environ["FSTAT_TEST_MEM_LIMIT"]
        rc, c, total = p.candidates_get_status(n)
        assert rc == fs.FSTAT_OK and total == n == c.size
        assert np.array_equal(c["sky"] * n_spin + c["spin"], np.repeat(np.arange(n_sky * n_spin), n_bins))
        assert np.array_equal(c["bin"], np.tile(np.arange(50, 50 + n_bins), n_sky * n_spin))
        for rc, early, total in got:
            if n < 65536:
                assert rc == fs.FSTAT_OK and np.array_equal(early, c)
            else:
                assert rc == fs.FSTAT_ERR_OOM and total == n
        p.search()                                   # not poisoned
        assert np.array_equal(p.candidates()[0], c)
