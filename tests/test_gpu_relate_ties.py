"""Relate on a circle where the wrapped tests need the exact word: elements of
equal time in several words, exactly opposite angles, the full angular range.
And 2+1 / 3+1 with every pair near the light cone or out of the filter's range.
All bits against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _bits(kind, c):
    import torch
    from paper_1805_04463_gb300 import build
    build.build()
    import paper_1805_04463_gb300 as cs
    n = c.shape[1]
    coords = torch.from_numpy(np.ascontiguousarray(c)).cuda()
    bits = torch.full((n, cs.row_words(n)), -1, dtype=torch.int64, device="cuda")
    cs.causal_matrix(kind, n, coords, bits)
    return bits.cpu().numpy().view(np.uint64)


@pytest.mark.parametrize("kind", [4, 6])
@pytest.mark.parametrize("n,times", [(65, 1), (200, 2), (777, 3), (2300, 40), (4500, 2000)])
def test_equal_times_and_opposite_angles(oracle, kind, n, times):
    rng = np.random.default_rng(n)
    top = 2 ** 29 - 1 if kind == 4 else 683565275
    eta = rng.integers(-top, top, times)[rng.integers(0, times, n)]
    theta = rng.integers(0, 2 ** 32, n)
    theta[::3] = rng.choice(np.array([0, 2 ** 31, 2 ** 31 - 1, 2 ** 31 + 1, 2 ** 32 - 1, 2 ** 30]), len(theta[::3]))
    o = np.argsort(eta, kind="stable")
    c = np.stack([eta[o].astype(np.int32), theta[o].astype(np.uint32).view(np.int32)])
    assert (_bits(kind, c) == oracle.causal_matrix(kind, c)).all()


@pytest.mark.parametrize("kind", [2, 3])
@pytest.mark.parametrize("n", [64, 130, 1000, 2500])
@pytest.mark.parametrize("span", [40, 3000, 2 ** 20, 2 ** 20 + 1, 2 ** 28])
def test_near_cone_and_beyond_the_filter(oracle, kind, n, span):
    rng = np.random.default_rng(span + n)
    d = 3 if kind == 3 else 4
    x = rng.integers(-span, span + 1, (d, n))
    # half the elements on light rays from the origin along one axis, give or take one grid step
    x[1:, ::2] = 0
    x[1, ::2] = np.clip(x[0, ::2] + rng.integers(-1, 2, len(x[0, ::2])), -span, span)
    c = x[:, np.argsort(x[0], kind="stable")].astype(np.int32)
    assert (_bits(kind, c) == oracle.causal_matrix(kind, c)).all()
