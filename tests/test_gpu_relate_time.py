"""Causal matrices of the 1+1 kinds take no longer than a 3+1 diamond's of the same size, whose
test is five packed operations per two pairs: the slab at a size where the mirror's blocks could crowd onto the
SMs that the upper part leaves first, the 2D order where the chunks are few."""
import pytest

pytestmark = pytest.mark.gpu


def _best(cs, kind, n):
    import torch
    coords = torch.empty((cs.dim(kind), n), dtype=torch.int32, device="cuda")
    ws = torch.empty(cs.sprinkle_workspace_bytes(kind, n), dtype=torch.uint8, device="cuda")
    cs.sprinkle(kind, n, 3, coords, ws)
    bits = torch.empty((n, cs.row_words(n)), dtype=torch.int64, device="cuda")
    times = []
    for _ in range(10):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(30):
            cs.causal_matrix(kind, n, coords, bits)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    return min(times)


@pytest.mark.parametrize("kind,n", [(4, 4099), (0, 5000)])
def test_against_3d_space(kind, n):
    from paper_1805_04463_gb300 import build
    build.build()
    import paper_1805_04463_gb300 as cs
    assert _best(cs, kind, n) < 1.12 * _best(cs, 2, n)
