"""The envelope solver's features against extended precision on the same
discrete equation: what is left is the stopping rule and the rounding of a
residual whose second difference is taken from differences."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _extended(E, n):
    """w_phi and p_phi by Newton with a tridiagonal elimination in np.longdouble."""
    T = np.longdouble
    E = E.astype(T)
    L = np.sqrt(E) + 8
    h = 2 * L / (n + 1)
    t2 = (-L + h * np.arange(1, n + 1, dtype=T)[:, None]) ** 2
    phi = np.maximum(np.sqrt(np.maximum(E - t2, 0)), T(2) ** T(0.25) * np.sqrt(E - 1) * np.exp(-t2 / 2))
    off = -1 / (h * h)
    zero = np.zeros((1, E.size), T)
    for _ in range(12):
        d = np.diff(np.concatenate([zero, phi, zero]), axis=0)
        f = off * (d[1:] - d[:-1]) + (t2 + phi * phi - E) * phi
        b = -2 * off + t2 + 3 * phi * phi - E
        for i in range(1, n):
            w = off / b[i - 1]
            b[i] -= w * off
            f[i] -= w * f[i - 1]
        f[n - 1] /= b[n - 1]
        for i in range(n - 2, -1, -1):
            f[i] = (f[i] - off * f[i + 1]) / b[i]
        phi = phi - f
    d = np.diff(np.concatenate([zero, phi, zero]), axis=0)
    pi = T("3.14159265358979323846264338327950288")
    return np.sqrt((d * d).sum(0) / (h * h) / (phi * phi).sum(0)) / (2 * pi), (h * phi.sum(0)) ** 2 / (4 * pi * pi)


@pytest.mark.parametrize("n", [255, 2047, 8191])
def test_features_against_extended_precision(n):
    from paper_0809_1547_gb300.binding import mb_gp_features
    E = np.array([1.3, 1.7, 2.5, 4.0, 7.1, 12.0, 23.0, 60.0])
    w, p = mb_gp_features(E, n)
    rw, rp = _extended(E, n)
    # a residual of 1e-13 E over the Jacobian's smallest eigenvalue, about
    # 2 (E - 1), relative to a peak of about sqrt(E - 1), twice for the square;
    # 2e-13 for the sums of n terms
    bound = 1e-13 * E / ((E - 1) * np.sqrt(E - 1)) + 2e-13
    assert np.all(np.abs(p / rp - 1) <= bound), np.abs(p / rp - 1)
    assert np.all(np.abs(w / rw - 1) <= bound), np.abs(w / rw - 1)
