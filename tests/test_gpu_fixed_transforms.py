"""The FP64 register transforms in fixed point (csrc/gke_fixed.cuh): every
length with one, spectra of all ranges, and exponents near the ends of the FP64
range, where the conversions take another way.

One homogeneous direction with a single snapshot whose fluctuations are one
x-mode times a random profile has A = 2-point sums with a closed form; instead
of restating it, the tests compare passes of the library whose results must
agree: scaled inputs (exact powers of two), and lengths against the oracle.
"""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def N():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1910_06409_gb300 import build as B
    B.build()
    import paper_1910_06409_gb300._native as native
    return native


def duct(N, wl, coef):
    import torch
    plan = N.gke1h_plan(wl.nx, wl.ny, wl.nz, wl.Lx, wl.nu, S.cgl_grid(wl.ny), S.cgl_grid(wl.nz), wl.nsnap)
    try:
        terms = torch.zeros((N.GKE1H_NTERM, N.gke1h_npair(plan), wl.nx), dtype=torch.float64, device="cuda")
        N.gke1h_compute(plan, torch.from_numpy(np.ascontiguousarray(coef)).cuda(), wl.nsnap, terms)
        return terms.cpu().numpy()
    finally:
        N.gke1h_destroy(plan)


@pytest.mark.parametrize("k", [-300, -40, 40, 300])
def test_scaled_velocities(N, k):
    """Fluctuations and mean times 2^k: A times 2^2k exactly (its transform works
    on a 1-norm times 2^2k; 2^+-600 is past FP32's range and the fast
    conversions' own)."""
    wl = S.duct_small(256, 5, 5, 2, wid=73)
    coef = S.duct_coefficients(wl)
    coef[:, 3] = 0.0
    one, got = duct(N, wl, coef)[0], duct(N, wl, coef * 2.0 ** k)[0]
    if abs(2 * k) < 880:
        assert np.array_equal(got, one * 2.0 ** (2 * k))
    else:
        assert np.abs(got - one * 2.0 ** (2 * k)).max() <= 1e-15 * np.abs(one).max() * 2.0 ** (2 * k)


@pytest.mark.parametrize("nx,nz", [(256, 8), (8, 256), (64, 128), (128, 64)])
def test_lengths_against_the_oracle(N, nx, nz):
    """Bar: 1e-12 of each term's largest value (the repository's FP64 bar)."""
    import oracle
    import torch
    wl = S.small(nx, nz, 6, 2, wid=74)
    phys = S.physical(wl)
    ref = oracle.full(phys, S.cgl_grid(wl.ny), wl.Lx, wl.Lz, wl.nu)["terms"]
    plan = N.gke_plan(nx, nz, wl.ny, wl.Lx, wl.Lz, wl.nu, S.cgl_grid(wl.ny), 2)
    try:
        terms = torch.zeros((N.GKE_NTERM, N.gke_npair(plan), nz, nx), dtype=torch.float64, device="cuda")
        N.gke_compute(plan, torch.from_numpy(S.to_coefficients(phys)).cuda(), 2, terms)
        got = terms.cpu().numpy()
    finally:
        N.gke_destroy(plan)
    iu = np.triu_indices(wl.ny)
    for t, name in enumerate(N.TERMS):
        want = ref[t][iu]
        assert np.abs(got[t] - want).max() <= 1e-12 * np.abs(want).max(), name
