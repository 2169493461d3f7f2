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
