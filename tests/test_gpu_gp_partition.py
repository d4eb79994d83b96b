"""The envelope solver's partitioned Newton step at the sizes where the
partition changes shape: fewer points than threads, a last thread with one
point, exact multiples of the thread count, arrays past shared memory."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _dense_solution(E, n):
    """phi by Newton with numpy's dense solver on the same grid (FP64)."""
    L = np.sqrt(E) + 8.0
    h = 2.0 * L / (n + 1)
    t = -L + h * np.arange(1, n + 1)
    phi = np.maximum(np.sqrt(np.maximum(E - t * t, 0.0)), 2 ** 0.25 * np.sqrt(E - 1) * np.exp(-0.5 * t * t))
    A = (np.diag(np.full(n, 2.0)) - np.diag(np.ones(n - 1), 1) - np.diag(np.ones(n - 1), -1)) / h ** 2
    for _ in range(40):
        f = A @ phi + (t * t + phi * phi - E) * phi
        d = np.linalg.solve(A + np.diag(t * t + 3 * phi * phi - E), f)
        phi = phi - d
        if np.abs(d).max() < 1e-13:
            break
    dphi = np.diff(np.concatenate([[0.0], phi, [0.0]]))
    return (np.sqrt((dphi ** 2).sum() / h ** 2 / (phi ** 2).sum()) / (2 * np.pi),
            (h * phi.sum()) ** 2 / (4 * np.pi ** 2), phi)


# 17..255: threads without points and threads with a lone separator;
# 256, 257: the first size of two points for every thread and one past it
@pytest.mark.parametrize("n", [17, 127, 128, 129, 255, 256, 257, 641])
def test_partition_edges(n):
    from paper_0809_1547_gb300.binding import mb_gp_features
    E = np.array([1.3, 4.0, 17.0])
    w, p, phi = mb_gp_features(E, n, want_phi=True)
    for q, e in enumerate(E):
        rw, rp, rphi = _dense_solution(e, n)
        # Newton converged on both sides to residuals of 1e-12 max(1, E); the
        # Jacobian's smallest eigenvalue is about 2 (E - 1) or more, so phi
        # agrees to 1e-11 and the features to 1e-10
        assert np.abs(phi[q] - rphi).max() <= 1e-10
        assert abs(w[q] / rw - 1) <= 1e-10 and abs(p[q] / rp - 1) <= 1e-10


def test_arrays_past_shared_memory():
    from paper_0809_1547_gb300.binding import mb_gp_features
    E = np.array([2.0, 9.0])
    # 6400 points fill shared memory exactly, 6401 go to global scratch: the
    # features differ by the grids' second-order error, h^2 (1 / n^2 relative)
    a, b = mb_gp_features(E, 6400), mb_gp_features(E, 6401)
    for x, y in zip(a, b):
        assert np.all(np.abs(x / y - 1) <= 1e-7)
