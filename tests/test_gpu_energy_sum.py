"""The energy sums keep what an FP64 sum of the cells' FP32 terms keeps."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N = 8192   # one block's cells; a thread takes every 256th


def _sum(e, h, w):
    """mb_energy_sum_noalloc of Ex = e, Hx = h (the other components zero)."""
    import torch
    from paper_0809_1547_gb300.binding import mb_energy_sum_noalloc
    out = torch.zeros(2, dtype=torch.float64, device="cuda")
    a = [torch.from_numpy(np.asarray(v, np.float32)).cuda() for v in (e, h, w)]
    z = torch.zeros(len(e), device="cuda")
    torch.cuda.synchronize()
    mb_energy_sum_noalloc(*(t.data_ptr() for t in (a[0], z, z, a[1], z, z, a[2])), len(e), out.data_ptr())
    torch.cuda.synchronize()
    v = out.cpu().numpy()
    assert v[1] == 0.0
    return v[0]


def _exact(e, h, w):
    e, h, w = (np.asarray(v, np.float32) for v in (e, h, w))
    with np.errstate(under="ignore"):
        e2, h2 = (e * e).astype(np.float64), (h * h).astype(np.float64)
    return math.fsum((w.astype(np.float64) * e2).tolist() + h2.tolist())


def test_terms_fifty_bits_apart_in_one_thread():
    e = np.zeros(N, np.float32)
    e[0], e[256] = 1.0, 1.5 * 2.0 ** -13
    e[512::256] = 2.0 ** -25
    # 1 + 2.25 * 2^-26 + 30 * 2^-50: every partial sum is an FP64 number
    assert _sum(e, np.zeros(N), np.ones(N)) == _exact(e, np.zeros(N), np.ones(N))


# weights around and outside the eps_r of a map, terms outside FP32's range of exact products
@pytest.mark.parametrize("scale", [1.0, 1e-12, 1e-14, 1e-18, 1e13, 1e15, 1e18])
@pytest.mark.parametrize("w", [(1.0, 12.0), (1e-30, 1e-2), (1e3, 1e6), (0.0, 0.0)])
def test_sum_of_random_terms(scale, w):
    rng = np.random.default_rng(7)
    e = rng.standard_normal(3 * N + 77) * scale * 10.0 ** rng.uniform(-3, 0, 3 * N + 77)
    h = rng.standard_normal(e.size) * scale
    eps = rng.uniform(*w, e.size)
    ref = _exact(e, h, eps)
    # 49152 additions at most, of one sign, in trees and runs of at most 64
    # terms: 64 + 16 roundings of 2^-53 each
    assert _sum(e, h, eps) == pytest.approx(ref, rel=80 * 2.0 ** -53, abs=0)
