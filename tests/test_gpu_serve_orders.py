"""Product orders on the server hold and are charged the table they are counted from, not a causal matrix."""
import pytest

pytestmark = pytest.mark.gpu


def test_no_matrix_for_a_product_order():
    import torch
    from paper_1805_04463_gb300 import build
    build.build()
    import paper_1805_04463_gb300 as cs
    from paper_1805_04463_gb300 import serve
    n = 1 << 16
    srv = serve.Server(bitset_budget=20e6)  # a table of 2^16 fits it, a bitset of 512 MB does not
    base = torch.cuda.memory_allocated()
    torch.cuda.reset_peak_memory_stats()
    wide = serve.Server()
    stats, first = wide.run([(0.0, 0, n, 5), (0.0, 1, 2000, 6)], realtime=False)
    assert stats["requests"] == 2
    assert torch.cuda.max_memory_allocated() - base < cs.bitset_bytes(n) / 4
    # one at a time under the small budget, the same results
    stats, res = srv.run([(0.0, 0, n, 5), (0.0, 1, 2000, 6)], realtime=False)
    assert stats["requests"] == 2
    for r in (0, 1):
        assert (res[r][0] == first[r][0]).all() and (res[r][1] == first[r][1]).all()
