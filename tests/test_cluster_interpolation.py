"""Interpolation error of the FP32 cross-patch sum's clusters (CPU, FP64).

A cluster's density acts through 8 x 8 charges on the Chebyshev points of its
square, on targets at least 4 half widths from its centre (maximum norm); a block of
targets takes the field of far clusters and cells on its own 8 x 8 points, from
four half widths on, and interpolates it. Restated here from the published form
(Lagrange interpolation on Chebyshev points, barycentric Lagrange treecode of Wang,
Krasny & Tlupova 2020): one charge at any place y of the square, one target X.

Bound, from theory alone: interpolating f on 8 Chebyshev points errs by at most
4 M rho^-7 / (rho - 1), M the largest |f| on the Bernstein ellipse of any rho that
leaves the kernel's singularities outside (Trefethen, Approximation Theory and
Approximation Practice, theorem 8.2); the second axis adds the same times the
Lebesgue constant of the points, (2 / pi) (ln 8 + gamma + ln(8 / pi)) = 2.29. The
target side has the same weights, so the same bound."""
import numpy as np
import pytest

NP = 8
C = np.cos((2 * np.arange(NP) + 1) * np.pi / (2 * NP))


def _lagrange(x):
    """Weights [n, point] of the Chebyshev points at x in [-1, 1]."""
    out = np.ones((NP,) + x.shape)
    for n in range(NP):
        for r in range(NP):
            if r != n:
                out[n] *= (x - C[r]) / (C[n] - C[r])
    return out


def _field(kind, dx, dy, z):
    r2 = dx * dx + dy * dy + z * z
    if kind == "potential":
        return np.stack([r2 ** -0.5])
    k = np.stack([dx, dy, np.full_like(dx, -z)]) * r2 ** -1.5
    return k if kind == "offplane" else k[:2]


def _bound(kind, ring, z):
    """Largest over the places of one axis of the theorem's bound, per target, as a
    multiple of the charge's own field (both axes; a field's norm by its components')."""
    th = np.linspace(0, np.pi, 61)  # the kernel's modulus is the same on both halves
    s = np.linspace(-1, 1, 17)
    rho = np.linspace(1.5, 14.0, 26)
    x = 0.5 * (rho[:, None] * np.exp(1j * th) + np.exp(-1j * th) / rho[:, None])  # [rho, angle]
    out = np.zeros(ring.shape[1])
    for k, (X, Y) in enumerate(ring.T):
        for a, b in ((X, Y), (Y, X)):  # interpolation along either axis
            for v in s:
                h = np.hypot(b - v, z)
                # the singularity a + i h and rho of its ellipse
                w = a + 1j * h
                lim = max(abs(w + np.sqrt(w * w - 1)), abs(w - np.sqrt(w * w - 1)))
                ok = rho < 0.999 * lim
                f = _field(kind, a - x[ok], (b - v) + 0 * x[ok], z)
                M = np.sqrt((np.abs(f).max(-1) ** 2).sum(0))
                e = (4 * M * rho[ok] ** -7 / (rho[ok] - 1)).min()
                own = _field(kind, a - s, (b - v) + 0 * s, z)  # the weakest own field along the line
                out[k] = max(out[k], e / np.sqrt((own ** 2).sum(0)).min())
    return (1 + 2.29) * out


@pytest.mark.parametrize("kind, z", [("force", 0.0), ("potential", 0.0), ("offplane", 0.01), ("offplane", 0.5),
                                     ("offplane", 3.0)])
@pytest.mark.parametrize("dist", [4.0, 8.0])
def test_interpolation_error_is_within_the_bound(kind, z, dist):
    t = np.linspace(-dist, dist, 17)
    ring = np.concatenate([np.stack([np.full_like(t, dist), t]), np.stack([t, np.full_like(t, -dist)])], axis=1)
    nodes = np.stack(np.meshgrid(C, C, indexing="ij")).reshape(2, -1)
    s = np.concatenate([np.linspace(-1, 1, 33), 0.5 * (C[1:] + C[:-1])])
    y = np.stack(np.meshgrid(s, s, indexing="ij")).reshape(2, -1)
    w = (_lagrange(y[0])[:, None, :] * _lagrange(y[1])[None, :, :]).reshape(NP * NP, -1)  # [node, place]
    kern = lambda a: _field(kind, a[0][:, None] - ring[0][None, :], a[1][:, None] - ring[1][None, :], z)
    exact = kern(y)
    e = np.sqrt(((exact - np.einsum("np,cnt->cpt", w, kern(nodes))) ** 2).sum(0) / (exact ** 2).sum(0))
    print("%s z %g at %g: worst %.2e rms %.2e" % (kind, z, dist, e.max(), np.sqrt(np.mean(e ** 2))))
    assert np.all(e.max(0) <= _bound(kind, ring, z))
