"""Sprinkle at the sizes where its route changes: one CTA up to 2048 elements,
bucket tables of 2^12 .. 2^16 entries above, more than one element per bucket
past 65536.  Coordinates are integers and must match the oracle exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", [0, 1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("n", [1023, 1025, 2047, 2048, 2049, 4096, 65537, 200003])
def test_coordinates_at_route_edges(oracle, kind, n):
    import torch
    from paper_1805_04463_gb300 import build
    build.build()
    import paper_1805_04463_gb300 as cs
    coords = torch.full((cs.dim(kind), n), -7, dtype=torch.int32, device="cuda")
    # a workspace full of ones: nothing may rest on its old contents
    ws = torch.full((cs.sprinkle_workspace_bytes(kind, n),), 255, dtype=torch.uint8, device="cuda")
    want = oracle.sprinkle(kind, n, 0x51000 + n)
    for _ in range(2):  # and a second time on the same workspace
        cs.sprinkle(kind, n, 0x51000 + n, coords, ws)
        assert cs.workspace_status(ws) == 0
        assert (coords.cpu().numpy() == np.asarray(want)).all()


@pytest.mark.parametrize("n", [2, 255, 256, 257, 511, 512, 513])
@pytest.mark.parametrize("path", [1, 2, 3])
def test_count_runs_in_exactly_the_workspace_it_asks_for(oracle, path, n):
    """The planned workspace is enough for the count, at sizes of one to three panels too."""
    import torch
    from paper_1805_04463_gb300 import build
    build.build()
    import paper_1805_04463_gb300 as cs
    buf = cs.allocate(0, n)
    cs.sprinkle(0, n, 77 + n, buf.coords, buf.workspace)
    cs.causal_matrix(0, n, buf.coords, buf.bits)
    ws = torch.empty(cs.interval_abundance_workspace(n, path), dtype=torch.uint8, device="cuda")
    cs.interval_abundance(n, buf.bits, buf.hist, path, ws)
    assert cs.workspace_status(ws) == 0
    want = oracle.interval_abundance(oracle.causal_matrix(0, oracle.sprinkle(0, n, 77 + n)))
    assert (buf.hist.cpu().numpy() == want).all()
