"""The zonal sums' column lists at their ends: one band (several chunks of
columns, the last one ragged), two, and more bands than rows of columns (empty
bands, bands of one column), against the oracle on the same state. Tolerances
as in the other zonal tests: 1e-12 on the weights (a sum of at most 642
float64 values), 1e-9 of the largest value elsewhere."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1607_05535_gb300 as thor
from harness import Pair
from oracle import climate as ocl
import workloads as wls

SMALL = wls.HS_G4.with_(name="hs_g3_L12", glevel=3, nv=12, n_large=2)


@pytest.mark.parametrize("precision", [thor.THOR_FP64, thor.THOR_MIXED])
@pytest.mark.parametrize("nlat", [1, 2, 360])
def test_bands_of_any_size(precision, nlat):
    p = Pair(SMALL, precision=precision)
    try:
        thor.thor_step(p.state, SMALL.n_large, SMALL.n_small, SMALL.dt)
        thor.thor_zonal_accumulate(p.state, nlat)
        got, n = thor.thor_zonal_read(p.state, nlat, SMALL.nv)
        assert n == 1
        with np.errstate(all="ignore"):
            ref = ocl.zonal_band_means(p.model, p.get(), nlat)
        full = ref[..., 0] > 0
        assert not got[~full].any()                          # empty bands stay zero
        np.testing.assert_allclose(got[..., 0][full], ref[..., 0][full], rtol=1e-12)
        for q in range(1, 9):
            scale = np.abs(ref[..., q][full]).max() + 1e-300
            lim = 1e-9 * scale
            if q >= 5:                                       # a covariance: against the size of its two products
                a, b = {5: (1, 2), 6: (2, 3), 7: (1, 1), 8: (2, 2)}[q]
                lim = 1e-9 * max(scale, np.abs(ref[..., a][full]).max() * np.abs(ref[..., b][full]).max())
            assert np.abs(got[..., q] - ref[..., q])[full].max() <= lim, (ocl.QUANTITIES[q],)
    finally:
        p.close()
