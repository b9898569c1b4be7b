"""Duct products by register transforms (k1_products_r in csrc/gke1h.cu) carry
two fields at a time: v and w 2^-30 of u and p, which share their transforms, still
have to give the terms made of their products to those terms' own size.

Against the CPU oracle at the FP64 bar of test_gpu_one_homog.py (1e-11 of each term's
largest value), with a viscosity so small that no viscous part is larger than the term:
the terms that are linear in v and w, at the two lengths of the kernel and one of the other."""
import numpy as np
import pytest

import synthetic as S
from oracle import one_homog as O1
from test_gpu_digit_paths import duct, native
from test_gpu_one_homog import TOL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(128, 5, 6, 3), (256, 6, 5, 9), (16, 5, 6, 3)])
def test_small_v_and_w(dims):
    N = native()
    nx, ny, nz, ns = dims
    wl = S.duct_small(nx, ny, nz, ns, wid=41, nu=1e-30)
    phys = S.duct_physical(wl)
    phys[:, 1:3] *= 2.0 ** -30
    ref = O1.full(phys, S.cgl_grid(ny), S.cgl_grid(nz), wl.Lx, wl.nu)["terms"]
    got = duct(N, wl, np.fft.rfft(phys, norm="forward"))
    i1, i2 = np.triu_indices(wl.npoint)
    for t in (2, 3, 4, 5, 6):
        want = ref[t][i1, i2]
        err = np.abs(got[t] - want).max() / np.abs(want).max()
        assert err < TOL, (N.TERMS_1H[t], err)
