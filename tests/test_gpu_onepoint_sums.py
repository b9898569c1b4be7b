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
