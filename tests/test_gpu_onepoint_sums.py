"""One-point sums of FP32 and split plans are FP64 sums of FP64 products at every
transform length but 256 (csrc/gke_products.cu).

Fluctuations that are constant in x and z pass the transforms exactly, and their
products need more than FP32's 24 bits: the statistics of a checkpoint equal an FP64
plan's to rounding (1e-14), where FP32 products are 2^-24 off."""
import numpy as np
import pytest

import synthetic as S
from test_gpu_digit_paths import native

pytestmark = pytest.mark.gpu


def statistics(N, nx, precision, path):
    import torch
    nz, ny = 8, 5
    coef = np.zeros((1, 4, ny, nz, nx // 2 + 1), dtype=np.complex128)
    for f, c in enumerate((1 + 2.0 ** -20, 1 - 2.0 ** -21, 1 + 2.0 ** -19, 3 + 2.0 ** -18)):
        coef[0, f, :, 0, 0] = c
    plan = N.gke_plan(nx, nz, ny, 12.0, 6.0, 0.005, S.cgl_grid(ny), 1, precision)
    try:
        N.gke_set_mean(plan, np.zeros((4, ny)))
        N.gke_accumulate_snapshot(plan, torch.from_numpy(coef).cuda(), 1)
        N.gke_checkpoint(plan, path)
    finally:
        N.gke_destroy(plan)
    return np.fromfile(path, dtype=np.float64, offset=96, count=11 * ny).reshape(11, ny)[4:10]


@pytest.mark.parametrize("nx", [16, 32, 64, 128])
def test_products_wider_than_fp32(nx, tmp_path):
    N = native()
    want = statistics(N, nx, N.GKE_PREC_F64, str(tmp_path / "f64"))
    assert (np.abs(want) > 0).all()
    for precision in (N.GKE_PREC_F32, N.GKE_PREC_BF16X3):
        got = statistics(N, nx, precision, str(tmp_path / "f32"))
        assert (np.abs(got / want - 1) <= 1e-14).all(), np.abs(got / want - 1).max()


def test_transforms_keep_the_energy(tmp_path):
    """The mean energy of random fields from FP32 transforms of 128 x 128 points
    (twiddles within half a unit of 2^-24) is the FP64 plan's within one FP32
    rounding, 2^-24: sampling noise is 1e-10, what remains is the transforms' gain."""
    import torch
    N = native()
    wl = S.small(128, 128, 9, 4, wid=77)
    f = torch.from_numpy(S.coefficients(wl)).cuda()
    q = []
    for precision in (N.GKE_PREC_F64, N.GKE_PREC_F32):
        path = str(tmp_path / "stats")
        plan = N.gke_plan(wl.nx, wl.nz, wl.ny, wl.Lx, wl.Lz, wl.nu, S.cgl_grid(wl.ny), wl.nsnap, precision)
        try:
            N.gke_accumulate_mean(plan, f, wl.nsnap)
            N.gke_accumulate_snapshot(plan, f, wl.nsnap)
            N.gke_checkpoint(plan, path)
        finally:
            N.gke_destroy(plan)
        q.append(np.fromfile(path, dtype=np.float64, offset=96, count=5 * wl.ny).reshape(5, wl.ny)[4])
    inner = q[0] > 0
    gain = (q[1][inner] / q[0][inner]).mean() - 1
    assert abs(gain) <= 2.0 ** -24, gain


@pytest.mark.parametrize("n", [32, 64, 128, 256])
def test_fp64_transforms_keep_the_energy(n, tmp_path):
    """The mean energy of random fields from fixed-point transforms of n x n points
    against Parseval's sum in extended precision, averaged over 31 planes: their sums
    of positive numbers round at random (about 1e-16 a plane, 2e-17 of the average), and
    the average stays within half an FP64 rounding, 2^-54, if the transforms have no gain of
    their own (constants of 53 bits gave 1.4e-16 at 64 points: sqrt(1/2) is 6.8e-17 too large)."""
    import torch
    N = native()
    wl = S.small(n, n, 33, 2, wid=78)
    coef = S.coefficients(wl)
    path = str(tmp_path / "stats")
    plan = N.gke_plan(n, n, wl.ny, wl.Lx, wl.Lz, wl.nu, S.cgl_grid(wl.ny), wl.nsnap)
    try:
        f = torch.from_numpy(coef).cuda()
        N.gke_accumulate_mean(plan, f, wl.nsnap)
        N.gke_accumulate_snapshot(plan, f, wl.nsnap)
        N.gke_checkpoint(plan, path)
    finally:
        N.gke_destroy(plan)
    got = np.fromfile(path, dtype=np.float64, offset=96, count=5 * wl.ny).reshape(5, wl.ny)[4]
    want = np.zeros(wl.ny, dtype=np.longdouble)
    for c in coef:                                     # [4][ny][nz][nxh]
        u = np.array(c[:3])
        u[:, :, 0, 0] = 0.0                            # the snapshots' means are equal: no fluctuation
        e = u.real.astype(np.longdouble) ** 2 + u.imag.astype(np.longdouble) ** 2
        want += 2 * e.sum((0, 2, 3)) - e[..., 0].sum((0, 2)) - e[..., -1].sum((0, 2))
    gain = got[1:-1] / (n * n * want[1:-1]) - 1
    assert np.abs(gain).max() < 1e-14, gain
    assert abs(gain.mean()) <= 2.0 ** -54, float(gain.mean())
