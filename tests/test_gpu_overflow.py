"""FP64 plans whose finite inputs overflow in the products: terms of interior
points are infinite or NaN, as FP64 arithmetic leaves them, on the paths that
work in integers (digit products, fixed-point transforms)."""
import numpy as np
import pytest

import synthetic as S
from test_gpu_one_homog import _run
from test_gpu_split import N, run_gpu  # noqa: F401

pytestmark = pytest.mark.gpu


def test_channel(N):  # noqa: F811
    wl = S.small(32, 16, 9, 2, wid=170)
    terms, _ = run_gpu(N, wl, S.coefficients(wl) * 1e170, precision=N.GKE_PREC_F64)
    i1, i2 = np.triu_indices(wl.ny)
    inner = (i1 > 0) & (i2 < wl.ny - 1)
    assert not np.isfinite(terms[:, inner]).any()


@pytest.mark.parametrize("nx", [16, 128])
def test_duct(nx):
    wl = S.duct_small(nx, 5, 6, 2, wid=37)
    terms, _ = _run(wl, S.duct_coefficients(wl) * 1e170)
    P = wl.ny * wl.nz
    i1, i2 = np.triu_indices(P)
    wall = np.array([(p // wl.nz) % (wl.ny - 1) == 0 or (p % wl.nz) % (wl.nz - 1) == 0 for p in range(P)])
    inner = ~wall[i1] & ~wall[i2]
    assert not np.isfinite(terms[:, inner]).any()
