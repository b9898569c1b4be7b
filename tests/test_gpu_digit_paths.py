"""The ways an FP64 plan can take through its contractions: chunks of one
wavenumber instead of one chunk, the FMA kernels that stand in where no digit
workspace can be allocated, and the duct's tiles at cross-sections around one
and two 128-row tiles, with one and two groups of 16 snapshots.

Bars: chunks change nothing, bit for bit; the duct against the oracle as in
test_gpu_one_homog.py (1e-11 of each term's largest value); the two channel
correlators against each other by the FP64 bar of test_gpu_digits.py."""
import ctypes

import numpy as np
import pytest

import synthetic as S
from oracle import one_homog as O1

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def native():
    from paper_1910_06409_gb300 import build as B
    B.build()
    import paper_1910_06409_gb300._native as N
    return N


def workspace(N, plan, nbytes, duct=False):
    f = N.lib().gke1h_test_digit_workspace if duct else N.lib().gke_test_digit_workspace
    f.argtypes = [ctypes.c_void_p, ctypes.c_longlong]
    f.restype = ctypes.c_int
    assert f(plan, nbytes) == N.GKE_OK


def channel(N, wl, coef, ws=None, nu=None, mask=0):
    plan = N.gke_plan(wl.nx, wl.nz, wl.ny, wl.Lx, wl.Lz, wl.nu if nu is None else nu, S.cgl_grid(wl.ny), coef.shape[0],
                      term_mask=mask)
    try:
        if ws is not None:
            workspace(N, plan, ws)
        terms = torch.zeros((N.GKE_NTERM, N.gke_npair(plan), wl.nz, wl.nx), dtype=torch.float64, device="cuda")
        N.gke_compute(plan, torch.from_numpy(np.ascontiguousarray(coef)).cuda(), coef.shape[0], terms)
        return terms.cpu().numpy()
    finally:
        N.gke_destroy(plan)


def duct(N, wl, coef, ws=None, nu=None):
    plan = N.gke1h_plan(wl.nx, wl.ny, wl.nz, wl.Lx, wl.nu if nu is None else nu, S.cgl_grid(wl.ny), S.cgl_grid(wl.nz),
                        coef.shape[0])
    try:
        if ws is not None:
            workspace(N, plan, ws, duct=True)
        terms = torch.zeros((N.GKE1H_NTERM, N.gke1h_npair(plan), wl.nx), dtype=torch.float64, device="cuda")
        N.gke1h_compute(plan, torch.from_numpy(np.ascontiguousarray(coef)).cuda(), coef.shape[0], terms)
        return terms.cpu().numpy()
    finally:
        N.gke1h_destroy(plan)


@pytest.mark.parametrize("dims", [(8, 8, 33, 9), (16, 8, 33, 1), (16, 8, 65, 17), (8, 8, 130, 2)])
def test_channel_chunks_and_fallback(dims):
    N = native()
    nx, nz, ny, ns = dims
    wl = S.small(nx, nz, ny, ns, wid=75)
    coef = S.to_coefficients(S.physical(wl))
    one = channel(N, wl, coef)
    assert np.array_equal(channel(N, wl, coef, ws=1), one)
    fma = channel(N, wl, coef, ws=0)
    g = max(1.0, (ny / 33.0) ** 2)
    tol = {"Phi_y": g, "phi": g, "residual": g * g}
    for t, name in enumerate(N.TERMS):
        assert np.abs(one[t] - fma[t]).max() <= 1e-12 * tol.get(name, 1.0) * np.abs(fma[t]).max(), name


# points: 121, 128, 132, 256, 260 (one row tile, just over, two, just over)
@pytest.mark.parametrize("dims", [(8, 11, 11, 16), (8, 8, 16, 2), (8, 11, 12, 17), (8, 16, 16, 1), (8, 13, 20, 16)])
def test_duct_tiles_chunks_and_fallback(dims):
    N = native()
    nx, ny, nz, ns = dims
    wl = S.duct_small(nx, ny, nz, ns, wid=38)
    coef = S.duct_coefficients(wl)
    ref = O1.full(S.duct_physical(wl), S.cgl_grid(ny), S.cgl_grid(nz), wl.Lx, wl.nu)["terms"]
    i1, i2 = np.triu_indices(wl.npoint)
    one = duct(N, wl, coef)
    assert np.array_equal(duct(N, wl, coef, ws=1), one)
    fma = duct(N, wl, coef, ws=0)
    for t, name in enumerate(O1.TERMS):
        want = ref[t][i1, i2]
        for got in (one, fma):
            assert np.abs(got[t] - want).max() < 1e-11 * np.abs(want).max(), name
