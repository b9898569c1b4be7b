"""The products pass of one homogeneous direction by register transforms
(k1_products_r in csrc/gke1h.cu): snapshot counts around the 8 (nx = 256) and 16
(nx = 128) that a CTA takes at a time, against the CPU oracle; the bar is the
FP64 one of test_gpu_one_homog.py."""
import numpy as np
import pytest

import synthetic as S
from oracle import one_homog as O1
from test_gpu_one_homog import TOL, _run, _triangle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(256, 5, 5, 1), (256, 5, 6, 9), (128, 6, 5, 17), (128, 5, 5, 8)])
def test_snapshot_groups(dims):
    nx, ny, nz, ns = dims
    wl = S.duct_small(nx, ny, nz, ns, wid=36)
    ref = O1.full(S.duct_physical(wl), S.cgl_grid(ny), S.cgl_grid(nz), wl.Lx, wl.nu)
    got, prof = _run(wl, S.duct_coefficients(wl))
    want = _triangle(ref["terms"])
    for t, name in enumerate(O1.TERMS):
        err = np.abs(got[t] - want[t]).max() / np.abs(want[t]).max()
        assert err < TOL, (name, err)
    np.testing.assert_allclose(prof, ref["prof"], rtol=0, atol=TOL * np.abs(ref["prof"]).max())
