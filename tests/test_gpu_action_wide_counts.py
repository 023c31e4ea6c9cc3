"""Smeared sums of histograms whose counts do not fit a double, and sums that cancel to a
small part of their terms, against the sum in exact rationals."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _f(dim, k, eps):
    """f_d(k, eps), exactly."""
    e = Fraction(eps)
    x, y, z = k * e / (1 - e), k * (k - 1) * (e / (1 - e)) ** 2, k * (k - 1) * (k - 2) * (e / (1 - e)) ** 3
    p = (1 - e) ** k
    return p * (1 - 2 * x + y / 2 if dim == 2 else 1 - 27 * x / 8 + 9 * y / 8 if dim == 3
                else 1 - 9 * x + 8 * y - 4 * z / 3)


@pytest.mark.parametrize("dim", [2, 3, 4])
@pytest.mark.parametrize("top", [2 ** 53 - 1, 2 ** 53 + 1, 2 ** 56 + 3, 2 ** 60 + 1])
def test_counts_past_a_double(dim, top):
    """N_0 odd and large, cancelled by one abundance of negative weight to about that weight: a count rounded to
    53 bits moves the sum by one and more.  The bound: each of the four
    terms and sums 2^-99 of its size, and three roundings of the result."""
    import torch
    from paper_1805_04463_gb300 import build
    build.build()
    import paper_1805_04463_gb300 as cs
    n, eps = 4096, 0.125
    low = min(range(2, 40), key=lambda k: _f(dim, k, eps))
    h = np.zeros(n - 1, dtype=np.int64)
    h[0], h[low] = top, int(-top / _f(dim, low, eps))
    h[1], h[30] = 3, 5
    total = sum(int(h[k]) * _f(dim, k, eps) for k in (0, 1, 30, low))
    size = sum(abs(int(h[k]) * _f(dim, k, eps)) for k in (0, 1, 30, low))
    hist = torch.from_numpy(h).cuda()
    out = torch.zeros(16, dtype=torch.float64, device="cuda")
    ws = torch.empty(cs.action_workspace_bytes(), dtype=torch.uint8, device="cuda")
    cs.action_device(dim, n, hist, [eps], out, torch.zeros(1, dtype=torch.int64, device="cuda"), ws)
    host, _ = cs.action(dim, n, h, eps)
    e = Fraction(eps)
    c3 = Fraction(0.9066587296704361)
    inner = n - (2 * e if dim == 2 else e) * total
    want = float(2 * e * inner) if dim == 2 else float(c3 * inner) * eps ** (2 / 3) if dim == 3 else \
        4 * (eps / 6) ** 0.5 * float(inner)
    bound = 8e-16 * abs(want) + float(size) * 2.0 ** -99 * 4
    assert abs(float(out[0]) - want) <= bound
    assert abs(host - want) <= bound
