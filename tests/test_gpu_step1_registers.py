"""Step 1 with the lengths whose transforms run in registers, and at the edges
of its row blocks and stencil windows, against the CPU oracle; a NaN of the
input reaches what it reached in FP64 transforms.  Tolerances as in
test_gpu_step1.py (5-point sums 1e-13, the banded solve 1e-10)."""
import numpy as np
import pytest

import synthetic as S
from oracle import step1 as O
from test_gpu_step1 import TOL, _errors, _native, _plan

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(wl, v_eta, mean_uw, shape):
    N = _native()
    plan = _plan(wl)
    try:
        out = torch.empty(shape, dtype=torch.complex128, device="cuda")
        N.gke_velocity_vorticity(plan, torch.from_numpy(v_eta).cuda(), torch.from_numpy(mean_uw).cuda(), wl.nsnap, out)
        return out.cpu().numpy()
    finally:
        N.gke_destroy(plan)


@pytest.mark.parametrize("shape", [(64, 32, 33, 1), (32, 64, 16, 2), (128, 256, 6, 1), (256, 128, 5, 1), (24, 64, 17, 1),
                                   (64, 12, 18, 1), (32, 32, 5, 1)])
def test_lengths_and_rows_match_oracle(shape):
    nx, nz, ny, ns = shape
    wl = S.small(nx, nz, ny, ns, wid=43)
    v_eta, mean_uw = S.vorticity_inputs(wl)
    want = O.step1(v_eta, mean_uw, S.cgl_grid(ny), wl.Lx, wl.Lz, wl.nu, nx)
    for f, e in enumerate(_errors(_run(wl, v_eta, mean_uw, want.shape), want)):
        assert e < TOL[f], (f, e)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_input_is_not_hidden(bad):
    """One non-finite coefficient of v: u and w at its wavenumber and the rows
    its stencils reach, p at every wavenumber."""
    wl = S.small(64, 64, 9, 1, wid=44)
    v_eta, mean_uw = S.vorticity_inputs(wl)
    v_eta[0, 0, 4, 3, 2] = bad
    got = _run(wl, v_eta, mean_uw, (1, 4, 9, 64, 33))
    assert not np.isfinite(got[0, 0, 4, 3, 2]) and np.isfinite(got[0, 0, 4, 3, 3])
    assert not np.isfinite(got[0, 3]).any()
