"""The FP32 correlators that stage every field of a wavenumber at once
(k_correlate_tile in csrc/gke_correlate_f64.cu, k1_correlate32 in
csrc/gke1h.cu), against the FP64 paths on the same inputs: edges of the tiles,
snapshot counts around the staging's rounding and its limit of 16, where the
first leaves the call to k_correlate and the second adds groups.  Bars as in
test_gpu_split.py (1e-6) and test_gpu_one_homog.py (1e-5 of each term's largest
value)."""
import numpy as np
import pytest

import synthetic as S
from test_gpu_one_homog import TOL32, _run
from test_gpu_split import N, TOL_SPLIT, rel_err, run_gpu  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny,ns", [(5, 1), (16, 3), (17, 2), (32, 16), (33, 1), (48, 5), (49, 17), (64, 16), (65, 2)])
def test_channel_tiles(N, ny, ns):  # noqa: F811
    wl = S.small(8, 12, ny, ns, wid=160 + ny)
    coef = S.coefficients(wl)
    ref, _ = run_gpu(N, wl, coef, precision=N.GKE_PREC_F64)
    got, _ = run_gpu(N, wl, coef, precision=N.GKE_PREC_F32)
    errs = [rel_err(got[t], ref[t]) for t in range(N.GKE_NTERM)]
    assert max(errs) <= TOL_SPLIT, dict(zip(N.TERMS, errs))


@pytest.mark.parametrize("ny,nz,ns", [(5, 5, 1), (5, 6, 3), (8, 8, 16), (5, 13, 17), (7, 9, 33), (6, 8, 4)])
def test_duct_tiles(ny, nz, ns):
    wl = S.duct_small(16, ny, nz, ns, wid=35)
    coef = S.duct_coefficients(wl)
    want, _ = _run(wl, coef)
    got, _ = _run(wl, coef, f32=True)
    for t in range(want.shape[0]):
        err = np.abs(got[t] - want[t]).max() / np.abs(want[t]).max()
        assert err < TOL32, (t, err)
