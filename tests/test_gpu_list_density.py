"""Sparse lists where a step's columns are placed word after word or lane by
lane: empty, few, just under and over the limit, full words.  Exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [33, 64, 2047, 2050, 4500])
@pytest.mark.parametrize("share", [0.0, 0.05, 0.15, 0.16, 0.5, 1.0])
def test_rows_of_any_density(n, share):
    """Any symmetric bit matrix has lists: rows of random density around `share`."""
    import torch
    from paper_1805_04463_gb300 import build
    build.build()
    import paper_1805_04463_gb300 as cs
    rng = np.random.default_rng(n)
    up = np.triu(rng.random((n, n)) < share * np.where(rng.random(n) < 0.3, rng.random(n), 1.0)[:, None], 1)
    m = up | up.T
    padded = np.zeros((n, cs.row_words(n) * 64), dtype=bool)
    padded[:, :n] = m
    bits = torch.from_numpy(np.packbits(padded, axis=1, bitorder="little").view(np.int64).copy()).cuda()
    for direction, part in ((0, np.tril(m, -1)), (1, np.triu(m, 1))):
        offsets, cols = cs.sparse_relations(n, bits, direction)
        assert (offsets.cpu().numpy() == np.concatenate([[0], np.cumsum(part.sum(1))])).all()
        assert (cols.cpu().numpy() == np.nonzero(part)[1]).all()
