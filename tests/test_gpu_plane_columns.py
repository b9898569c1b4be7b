"""Column pass of the plane spectra by register transforms (csrc/gke_terms.cu,
k_terms_colpass_planes_r): every length with one, pair counts and x half
spectra that leave its groups of four partly empty, full and strided
separations; against the FP64 path on the same inputs."""
import pytest

import synthetic as S
from test_gpu_split import N, TOL_SPLIT, rel_err, run_gpu  # noqa: F401
from test_gpu_undersample import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz,ny,stride", [(8, 32, 6, 1), (16, 64, 5, 1), (8, 128, 9, 1), (32, 256, 5, 1),
                                             (12, 64, 7, 1), (8, 32, 6, 2), (16, 128, 5, 4)])
def test_register_columns_match_f64(N, nx, nz, ny, stride):  # noqa: F811
    wl = S.small(nx, nz, ny, 3, wid=150 + ny)
    coef = S.coefficients(wl)
    if stride > 1:
        u = (0, 0, 0, stride)
        ref, _, _ = run(N, wl, coef, N.GKE_PREC_F64, ux=u, uz=u)
        got, _, _ = run(N, wl, coef, N.GKE_PREC_BF16X3, ux=u, uz=u)
    else:
        ref, _ = run_gpu(N, wl, coef, precision=N.GKE_PREC_F64)
        got, _ = run_gpu(N, wl, coef, precision=N.GKE_PREC_BF16X3)
    errs = [rel_err(got[t], ref[t]) for t in range(N.GKE_NTERM)]
    assert max(errs) <= TOL_SPLIT, dict(zip(N.TERMS, errs))
