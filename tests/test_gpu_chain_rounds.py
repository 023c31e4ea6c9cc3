"""Chains and antichains where the one-launch rounds change shape: one CTA,
several, every SM; more removed candidates in a round than are listed at once;
more elements than one slot per lane.  Lengths and members are exact."""
import bisect

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cs():
    from paper_1805_04463_gb300 import build
    build.build()
    import paper_1805_04463_gb300 as m
    return m


def _bits(cs, kind, n, coords=None, seed=5):
    import torch
    b = cs.allocate(kind, n, path=1)
    if coords is None:
        cs.sprinkle(kind, n, seed, b.coords, b.workspace)
    else:
        b.coords.copy_(torch.from_numpy(np.ascontiguousarray(coords, dtype=np.int32)))
    cs.causal_matrix(kind, n, b.coords, b.bits)
    return b


@pytest.mark.parametrize("kind,n", [(0, 127), (0, 128), (0, 129), (4, 1025), (2, 4097), (0, 5000), (2, 9001), (0, 12000)])
def test_against_oracle(cs, oracle, kind, n):
    b = _bits(cs, kind, n)
    bits = b.bits.cpu().numpy().view(np.uint64)
    assert cs.longest_chain(n, b.bits) == oracle.longest_chain(bits)
    for i, j in ((0, n - 1), (n // 9, n - n // 7), (3, 5), (n // 2, n // 2 + 1)):
        assert cs.longest_chain(n, b.bits, i, j) == oracle.longest_chain(bits, i, j), (i, j)
    for s in (0, n // 2):
        size, members = cs.greedy_antichain(n, b.bits, s)
        w_size, w_members = oracle.greedy_antichain(bits, s)
        assert size == w_size and (members.cpu().numpy().view(np.uint64) == w_members).all()


@pytest.mark.parametrize("n", [1, 64, 1000, 3000])
def test_total_order_and_antichain(cs, n):
    """n rounds of one element, and one round of n."""
    for v, height in ((np.arange(n), n), (np.arange(n)[::-1], 1)):
        b = _bits(cs, 0, n, np.stack([np.arange(n), v]))
        assert cs.longest_chain(n, b.bits) == height
        size, _ = cs.greedy_antichain(n, b.bits, n // 2)
        assert size == (1 if height == n else n)


def test_more_elements_than_one_slot(cs):
    n = 170_003
    b = _bits(cs, 0, n)
    tails = []
    for x in b.coords[1].cpu().numpy().tolist():
        k = bisect.bisect_left(tails, x)
        tails[k:k + 1] = [x]
    assert cs.longest_chain(n, b.bits) == len(tails)
