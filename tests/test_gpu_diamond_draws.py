"""Rejection draws shared by the lanes of a warp: warps with few elements, and
batch warps that hold elements of several sets and kinds.  Integers, exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _cs():
    from paper_1805_04463_gb300 import build
    build.build()
    import paper_1805_04463_gb300 as cs
    return cs


@pytest.mark.parametrize("kind", [2, 3])
@pytest.mark.parametrize("n", [1, 2, 3, 15, 16, 17, 31, 32, 33, 1025, 2049])
def test_coordinates(oracle, kind, n):
    import torch
    cs = _cs()
    coords = torch.full((cs.dim(kind), n), -7, dtype=torch.int32, device="cuda")
    ws = torch.full((cs.sprinkle_workspace_bytes(kind, n),), 255, dtype=torch.uint8, device="cuda")
    for seed in (1, 2, 3):
        cs.sprinkle(kind, n, seed, coords, ws)
        assert cs.workspace_status(ws) == 0
        assert (coords.cpu().numpy() == np.asarray(oracle.sprinkle(kind, n, seed))).all()


@pytest.mark.parametrize("sets", [33, 40, 70, 1100])
def test_batches_of_sets_smaller_than_a_warp(oracle, sets):
    """Sets of 1 to 40 elements of every kind side by side, 33 sets and more (the search for a
    warp's set takes more than one step)."""
    import torch
    cs = _cs()
    plan = [((2, 3, 0, 2, 4, 3, 1, 6, 5)[s % 9], 1 + (7 * s) % 40, 500 + s) for s in range(sets)]
    b = cs.Batch(plan, n_eps=1)
    b.launch((0.0,))
    torch.cuda.synchronize()
    assert b.status() == 0
    for s, (kind, n, seed) in enumerate(plan):
        want = oracle.interval_abundance(oracle.causal_matrix(kind, oracle.sprinkle(kind, n, seed)))
        assert (b.set_hist(s).cpu().numpy() == want).all(), (s, kind, n)
