"""What Buffers plans on PATH_AUTO (no GPU: buffers on the meta device)."""
import pytest


@pytest.fixture
def cs():
    from paper_1805_04463_gb300 import build
    build.build()
    import paper_1805_04463_gb300 as m
    yield m
    m.set_auto_memory_limit(0)


@pytest.mark.parametrize("kind", [0, 1, 5])
def test_a_product_order_keeps_to_the_memory_limit(cs, kind):
    """The count from coordinates takes n^2/256 bytes: only where they fit beside the bitset."""
    n = 1 << 16
    table = cs.coords_abundance_workspace(kind, n)
    small = max(cs.sprinkle_workspace_bytes(kind, n), cs.action_workspace_bytes())
    assert small < table
    for limit, by_coords in ((cs.bitset_bytes(n) + table, True), (cs.bitset_bytes(n) + table - 1, False),
                             (cs.bitset_bytes(n) + small, False)):
        cs.set_auto_memory_limit(limit)
        buf = cs.Buffers(kind, n, device="meta")
        assert buf.by_coords == by_coords
        assert buf.bits.numel() * 8 + buf.workspace.numel() <= limit


@pytest.mark.parametrize("path", [0, 1, 2, 3])
def test_run_counts_on_the_path_the_buffers_name(cs, monkeypatch, path):
    """A path set on the buffers after they were planned is the one that counts."""
    cs.set_auto_memory_limit(1 << 34)
    buf = cs.Buffers(0, 2000, device="meta")
    assert buf.by_coords
    calls = []
    for name in ("sprinkle", "causal_matrix", "coords_abundance", "interval_abundance", "action_device"):
        monkeypatch.setattr(cs, name, lambda *a, _n=name, **k: calls.append((_n, a)))
    buf.path = path
    cs.run(buf, 1)
    assert [c for c, _ in calls] == ["sprinkle", "causal_matrix",
                                     "interval_abundance" if path else "coords_abundance", "action_device"]
    if path:
        assert calls[2][1][3] == path


def test_buffers_without_a_matrix_are_for_product_orders(cs):
    cs.set_auto_memory_limit(1)  # no bitset, nothing to fit beside it
    buf = cs.Buffers(1, 3000, device="meta", matrix=False)
    assert buf.by_coords and buf.bits is None and buf.workspace.numel() < cs.bitset_bytes(3000)
    for kind, path in ((2, 0), (4, 0), (1, 3)):
        with pytest.raises(ValueError):
            cs.Buffers(kind, 3000, device="meta", path=path, matrix=False)
