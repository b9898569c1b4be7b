"""The FP64 contractions by exact digit products (csrc/gke_digits.cu) at the
edges of their tiles: row tiles of 40, 72 and 128 rows, column tiles of 24 and
32, the thin remainder past 128 rows, one and two groups of 16 snapshots.

Bar against the oracle: 1e-12 of each term's largest value, the repository's
FP64 bar, for the terms without stencils; the Step-3 stencils multiply
rounding by sum |w| ~ 1 / dy_min ~ ny^2 once (Phi_y, phi) or twice (residual),
so their bars grow from the 33-point grid of the parity tests with (ny / 33)^2
and (ny / 33)^4.
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


def run(N, wl, coef, mask=0):
    import torch
    plan = N.gke_plan(wl.nx, wl.nz, wl.ny, wl.Lx, wl.Lz, wl.nu, S.cgl_grid(wl.ny), coef.shape[0], term_mask=mask)
    try:
        terms = torch.zeros((N.GKE_NTERM, N.gke_npair(plan), wl.nz, wl.nx), dtype=torch.float64, device="cuda")
        N.gke_compute(plan, torch.from_numpy(np.ascontiguousarray(coef)).cuda(), coef.shape[0], terms)
        return terms.cpu().numpy()
    finally:
        N.gke_destroy(plan)


@pytest.mark.parametrize("ny,ns", [(5, 9), (24, 17), (25, 16), (32, 16), (33, 1), (40, 3), (41, 16), (65, 33), (72, 2),
                                   (73, 5), (128, 2), (129, 2), (133, 1)])
def test_tile_edges(N, ny, ns):
    import oracle
    wl = S.small(8, 8, ny, ns, wid=70)
    phys = S.physical(wl)
    ref = oracle.full(phys, S.cgl_grid(ny), wl.Lx, wl.Lz, wl.nu)["terms"]
    got = run(N, wl, S.to_coefficients(phys))
    iu = np.triu_indices(ny)
    g = max(1.0, (ny / 33.0) ** 2)
    tol = {"Phi_y": g, "phi": g, "residual": g * g}
    for t, name in enumerate(N.TERMS):
        want = ref[t][iu]
        err = np.abs(got[t] - want).max() / max(np.abs(want).max(), 1e-300)
        assert err <= 1e-12 * tol.get(name, 1.0), f"{name}: {err:.3e}"


def test_rows_far_apart_and_coherent_snapshots(N):
    """Snapshots that are multiples of one field (every product of a sum has
    the same sign) by factors from 1 to 2^-40, and wall-normal rows scaled by
    powers of two down to 2^-60: A at every pair is exactly
    f^2 |a_1|^2 + |a_2|^2 - 2 a_1 a_2 of the unscaled rows up to rounding of the pair's
    own size."""
    wl = S.small(16, 8, 33, 1, wid=71)
    base = S.to_coefficients(S.physical(wl))
    base[:, :, :, 0, 0] = 0.0                                  # no mean: the fluctuations are the fields
    fac = np.array([1.0, -1.0, 0.75, -0.75, 2.0 ** -40, -2.0 ** -40])
    row = 2.0 ** -np.linspace(0, 60, 33).round()
    coef = fac[:, None, None, None, None] * base * row[None, None, :, None, None]
    got = run(N, S.small(16, 8, 33, 6, wid=71), coef, mask=1)[0]
    ph = np.fft.irfft2(coef[0, :3], s=(8, 16), norm="forward")
    w = (fac ** 2).mean()
    i1, i2 = np.triu_indices(33)
    k = np.fft.rfft2(ph, norm="forward")
    cross = np.fft.irfft2((k[:, i1].conj() * k[:, i2]).sum(0), s=(8, 16), norm="forward")
    q = (ph * ph).sum(0).mean((1, 2))
    want = w * (q[i1] + q[i2])[:, None, None] - 2 * w * cross
    size = w * (q[i1] + q[i2])[:, None, None]
    keep = size[:, 0, 0] > 0
    assert (np.abs(got - want)[keep] / size[keep]).max() <= 1e-14


def test_power_of_two_scaling_is_exact(N):
    """Velocities times 2^k: A times 2^2k, bit for bit (exponents far from the
    products' own ranges)."""
    wl = S.small(8, 12, 26, 9, wid=72)
    coef = S.to_coefficients(S.physical(wl))
    one = run(N, wl, coef, mask=1)[0]
    for k in (-240, 240):
        assert np.array_equal(run(N, wl, coef * 2.0 ** k, mask=1)[0], one * 2.0 ** (2 * k))
