"""The causal matrix on both sides of the line between chunks of 8 and of 32
words, and at their edges.  Every word of every row against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", [0, 1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("n", [1, 64, 511, 512, 513, 2047, 2049, 6144, 6145])
def test_every_word(oracle, kind, n):
    import torch
    from paper_1805_04463_gb300 import build
    build.build()
    import paper_1805_04463_gb300 as cs
    c = np.ascontiguousarray(oracle.sprinkle(kind, n, 0xC0 + n), dtype=np.int32)
    want = np.asarray(oracle.causal_matrix(kind, c)).view(np.int64)
    bits = torch.full((n, cs.row_words(n)), -1, dtype=torch.int64, device="cuda")
    cs.causal_matrix(kind, n, torch.from_numpy(c).cuda(), bits)
    got = bits.cpu().numpy()
    w = want.shape[1]
    assert (got[:, :w] == want).all() and not got[:, w:].any()
