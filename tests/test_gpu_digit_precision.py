"""The digit products against the FMA kernels on the same operands where one
velocity component is small beside the others, everywhere or on some of the
points: a term that is made of products of the small component has to come out
to that product's size, not to that of the larger components.

The bar of a value is derived from the fields.  Both sides' error of a sum
over snapshots and terms is below g = (2 x 16 x 4 + 2) 2^-53 times the sum of |a| |b|, which
over all wavenumbers is at most the product of the two fields' rms at the
pair's points (Parseval, Cauchy-Schwarz): 2 g = 3e-14 of that.  The one-point
parts, the same on both sides, add the rounding of the last addition: 1e-15 of theirs.
The viscosity is tiny, so that no viscous part is larger than what it is added to; the
difference of its parts, NU sum |w| 2 g of A, is below NU times A (sum |w| < 1e3).
The channel is asked for one term at a time and the duct's bar is taken over the two
pairs of a packed transform (2 i, 2 i + 1), since a transform rounds at the size of all it
carries; the residual, which mixes all, is left out."""
import numpy as np
import pytest

import synthetic as S
from test_gpu_digit_paths import channel, duct, native

pytestmark = pytest.mark.gpu

NU = 1e-30
BAR, ONE = 3e-14, 1e-15
CASES = [(0, 20, 16), (1, 20, 17), (1, 20, 1), (1, 40, 16), (2, 20, 17), (2, 40, 2), (1, 6, 16), ("mixed", 20, 16),
         ("mixed", 8, 1)]


def scaled(phys, field, bits):
    """component `field` times 2^-bits, or with "mixed" another component on each
    of the first axis' points"""
    c = phys.copy()
    if field == "mixed":
        for f in range(3):
            c[:, f, f::3] *= 2.0 ** -bits
    else:
        c[:, field] *= 2.0 ** -bits
    return c


class Sizes:
    """rms products of a set of points; phys[s][4][P][...], G[i][b] the gradients of the
    mean of u_i along the inhomogeneous directions b"""

    def __init__(self, phys, G, dirs):
        a = phys.reshape(phys.shape[0], 4, phys.shape[2], -1)
        self.U = a.mean((0, 3))
        f = a - self.U[None, :, :, None]
        rms = lambda x: np.sqrt((x * x).mean((0, 2)))  # noqa: E731
        u = [f[:, i] for i in range(3)]
        q = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        self.i1, self.i2 = np.triu_indices(a.shape[2])
        self.u, self.p, self.q = [rms(x) for x in u], rms(f[:, 3]), rms(q)
        self.uu = [[rms(u[i] * u[k]) for k in range(3)] for i in range(3)]
        self.G, self.dirs = G, dirs

    def cross(self, a, b):
        return a[self.i1] * b[self.i2] + b[self.i1] * a[self.i2]

    def both(self, a):
        return a[self.i1] + a[self.i2]

    def triple(self, k):
        return self.cross(self.q, self.u[k]) + 2 * sum(self.cross(self.uu[i][k], self.u[i]) for i in range(3))

    def energy(self):
        return 2 * sum(self.cross(x, x) for x in self.u)

    def jump(self, k):
        return np.abs(self.U[k][self.i2]) + np.abs(self.U[k][self.i1])

    def A(self):
        return BAR * self.energy() + ONE * self.both(sum(x * x for x in self.u))

    def phi(self, k):                                  # Phi_k
        return (BAR * (self.triple(k) + self.jump(k) * self.energy())
                + ONE * (self.both(self.q * self.u[k]) + self.jump(k) * self.both(sum(x * x for x in self.u))))

    def psi(self, k):
        return (BAR * 2 * self.cross(self.p, self.u[k]) + ONE * 4 * self.both(self.p * self.u[k])) + self.phi(k)

    def xi(self):
        s, o = 0, 0
        for a in range(3):
            for b in self.dirs:
                g = np.abs(self.G[a, b])
                s = s + 2 * (g[self.i2] * self.cross(self.u[a], self.u[b]) + g[self.i1] * self.cross(self.u[a], self.u[b]))
                o = o + 4 * (g[self.i1] + g[self.i2]) * self.both(self.u[a] * self.u[b])
        return BAR * s + ONE * o


def check(got, want, bar, name, s):
    bar = bar + NU * s.energy().max()
    err = np.abs(got - want).reshape(got.shape[0], -1).max(1)
    bad = err > bar
    assert not bad.any(), (name, int(bad.sum()), float((err[bad] / bar[bad]).max()))


@pytest.mark.parametrize("field,bits,ns", CASES)
def test_channel(field, bits, ns):
    N = native()
    wl = S.small(16, 8, 33, ns, wid=76)                # 72 wavenumbers: digits at any snapshot count
    phys = scaled(S.physical(wl), field, bits)
    coef = S.to_coefficients(phys)
    y = S.cgl_grid(wl.ny)
    D = np.zeros((wl.ny, wl.ny))
    for j in range(wl.ny):
        l0, w = N.gke_fd_weights(y, j)
        D[j, l0:l0 + 5] = w
    s = Sizes(phys, None, (1,))
    s.G = {(i, 1): (D @ s.U[0] if i == 0 else 0 * s.U[0]) for i in range(3)}
    s.U[1:] = 0.0                                      # the mean flow is U(y)
    bars = (s.A(), s.phi(0), s.phi(1), s.phi(2), s.psi(1), s.xi())
    for t, bar in enumerate(bars):
        one = channel(N, wl, coef, nu=NU, mask=1 << t)[t]
        check(one, channel(N, wl, coef, ws=0, nu=NU, mask=1 << t)[t], bar, N.TERMS[t], s)


@pytest.mark.parametrize("field,bits,ns", CASES)
def test_duct(field, bits, ns):
    N = native()
    wl = S.duct_small(8, 7, 6, ns, wid=39)
    phys = scaled(S.duct_physical(wl), field, bits)
    coef = np.fft.rfft(phys, norm="forward")
    D = []
    for n in (wl.ny, wl.nz):
        D.append(np.zeros((n, n)))
        for j in range(n):
            l0, w = N.gke_fd_weights(S.cgl_grid(n), j)
            D[-1][j, l0:l0 + 5] = w
    flat = phys.reshape(ns, 4, wl.npoint, wl.nx)
    s = Sizes(flat, None, (1, 2))
    U = s.U.reshape(4, wl.ny, wl.nz)
    s.G = {(i, 1): (D[0] @ U[i]).ravel() for i in range(3)}
    s.G.update({(i, 2): (U[i] @ D[1].T).ravel() for i in range(3)})
    bars = (s.A(), s.phi(0), s.phi(1), s.phi(2), s.psi(1), s.psi(2), s.xi())
    one, fma = duct(N, wl, coef, nu=NU), duct(N, wl, coef, ws=0, nu=NU)
    for t, bar in enumerate(bars):
        two = np.maximum.reduceat(bar, np.arange(0, len(bar), 2))
        check(one[t], fma[t], np.repeat(two, 2)[:len(bar)], N.TERMS_1H[t], s)
