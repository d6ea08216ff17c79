"""The skip test of the z pass clears the two minor axes through the identity
g_i(F) - g_0(F) = (lam_0 - lam_i)(F^2 + (3/14) lam_k F + (5/84) lam_k mu1)
between the axis cubics (collapse_x2.cuh): the identity itself, and that the
cleared minor axes have no root at or above t, against numpy's roots."""
import numpy as np
import pytest


def _cubic(lam, i):
    j, k = (i + 1) % 3, (i + 2) % 3
    e = [0.5 * lam[a] * (lam[(a + 1) % 3] + lam[(a + 2) % 3]) for a in range(3)]
    c3 = 10 / 84 * (lam[i] * (e[j] + e[k]) + e[i] * (lam[j] + lam[k])) - lam[0] * lam[1] * lam[2] / 9
    return np.array([1.0, -lam[i], -3 / 7 * e[i], -c3])


@pytest.mark.parametrize("scale", [1.0, 1e-3, 30.0])
def test_identity_and_cleared_axes(scale):
    rng = np.random.default_rng(4)
    cleared = 0
    for n in range(4000):
        lam = np.sort(rng.normal(size=3) * scale + rng.normal() * scale * (n % 3))[::-1]
        mu1 = lam.sum()
        g = [_cubic(lam, i) for i in range(3)]
        for i, k in ((1, 2), (2, 1)):
            q = (lam[0] - lam[i]) * np.array([0.0, 1.0, 3 / 14 * lam[k], 5 / 84 * lam[k] * mu1])
            assert np.allclose(g[i] - g[0], q, rtol=0, atol=1e-12 * max(1, scale) ** 3)
        roots0 = np.roots(g[0])
        real0 = roots0[np.abs(roots0.imag) < 1e-6 * scale].real
        t = max(0.0, real0.max() if real0.size else 0.0) + scale * rng.exponential(0.3)
        ok = True
        for lk in lam[1:]:
            ok &= lk * (3 / 14 * t + 5 / 84 * mu1) + t * t * (1 - 1e-4) > 0
            ok &= t + 3 / 28 * lk > 0 or 9 / 196 * lk - 5 / 21 * mu1 > 0
        if ok:
            cleared += 1
            for i in (1, 2):
                r = np.roots(g[i])
                real = r[np.abs(r.imag) < 1e-9 * scale].real
                assert not (real >= t).any(), (lam, t, i)
    assert cleared > 2000
